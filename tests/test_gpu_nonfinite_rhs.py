"""A right-hand side with one NaN ends a solve with GL_ERR_NAN in every form: a zero norm
and one that compares as nothing are told apart.  A zero right-hand side still has the
solution zero, from any guess."""
import numpy as np
import pytest

import gl_inputs as gi

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1204_5125_gb300 as gl  # noqa: E402

DEV = torch.device("cuda:0")
GL_ERR_NAN = 6
FORMS = {"fp64": gl.GL_FP64, "mixed": gl.GL_MIXED, "fp32vc": gl.GL_MIXED_PRECOND}


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


@pytest.mark.parametrize("device_loop", [1, 0], ids=["device", "host"])
@pytest.mark.parametrize("form,cycles", [("fp64", 0), ("fp64", 1), ("mixed", 1), ("fp32vc", 1)])
def test_nan_in_the_right_hand_side(form, cycles, device_loop):
    n = 40 * 40
    m = gl.gl_mesh_create(2, 40, 1.0)
    psi, b = gi.disk(n, 31), gi.complex_normal(n, 32)
    opts = gl.options(precision=FORMS[form], cycles=cycles, max_coarse=64, device_loop=device_loop)
    try:
        for at, value in [(0, np.nan), (n - 1, 1j * np.nan)]:
            bad = b.copy()
            bad[at] = value
            x = torch.zeros(n, dtype=torch.complex128, device=DEV)
            st, info = gl.gl_jacobian_solve(m, dev(psi), None, dev(bad), x, opts, raise_on_fail=False)
            assert st == GL_ERR_NAN and not info.converged and info.iters == 0
            assert np.isnan(info.true_relres)
        x = torch.full((n,), complex("nan"), dtype=torch.complex128, device=DEV)
        st, info = gl.gl_jacobian_solve(m, dev(psi), None, dev(0 * b), x, opts)
        assert st == 0 and info.converged and bool((x == 0).all())
    finally:
        gl.gl_mesh_destroy(m)


def test_newton_step_from_a_nan_state():
    m = gl.gl_mesh_create(2, 24, 1.0)
    psi = gi.psi_noisy_one(24 * 24, 33)
    psi[100] = np.nan
    t = dev(psi)
    try:
        with pytest.raises(gl.GLError) as e:
            gl.gl_newton_step(m, t, gl.options(cycles=0))
        assert e.value.status == GL_ERR_NAN
        assert np.array_equal(t.cpu().numpy(), psi, equal_nan=True)  # no step was taken
    finally:
        gl.gl_mesh_destroy(m)


@pytest.mark.parametrize("form", ["fp64", "fp32vc"])
def test_nan_in_one_system_of_a_batch(form):
    sides = (24, 33, 40)
    ms = [gl.gl_mesh_create(2, N, 1.0) for N in sides]
    psi = [dev(gi.disk(N * N, 34 + N)) for N in sides]
    b = [gi.complex_normal(N * N, 35 + N) for N in sides]
    opts = gl.options(precision=FORMS[form], max_coarse=64)
    B = gl.gl_batch_create(ms, psi, opts)
    try:
        good = [torch.zeros(N * N, dtype=torch.complex128, device=DEV) for N in sides]
        st, infos = gl.gl_batch_run(B, [dev(v) for v in b], good)
        assert st == 0 and all(i.converged for i in infos)
        b[1][7] = np.nan
        x = [torch.zeros_like(v) for v in good]
        with pytest.raises(gl.GLError) as e:
            gl.gl_batch_run(B, [dev(v) for v in b], x)
        assert e.value.status == GL_ERR_NAN
        assert torch.equal(x[0], good[0]) and torch.equal(x[2], good[2])
    finally:
        gl.gl_batch_destroy(B)
        for m in ms:
            gl.gl_mesh_destroy(m)
