"""The forms of the coarse sweeps that only the setup's timing chooses: every number of
lanes per row with one and two shifts of warps (and the entries loaded ahead that go with
the lanes and the rows' length), dataflow against the grid barrier on one shift, bit for
bit: equal lanes sum a row in the same order.  Levels with fewer rows than a warp's step,
with short and long rows, and with more rows than the warps take at once; a solve after a
change of form must not run a captured graph of the form before."""
import pytest

import gl_inputs as gi

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1204_5125_gb300 as gl  # noqa: E402

DEV = torch.device("cuda:0")
FORMS = [(G, K) for G in (2, 4, 8, 16, 32) for K in (1, 2)]


def form(P, G, K):
    gl.gl_precond_debug(P, gl.GL_DEBUG_SWEEP_FORM + 64 * K + G)


@pytest.mark.parametrize("dim,N,max_coarse", [(2, 20, 16), (2, 45, 24), (2, 300, 512), (3, 18, 24), (3, 37, 64),
                                              (3, 112, 4096), ("circ", 0.35, 64)], ids=lambda p: str(p))
def test_lanes_and_shifts(dim, N, max_coarse):
    if dim == "circ":
        pytest.importorskip("scipy")
        m = gl.gl_mesh_create_simplicial(*gi.delaunay_domain("circ", N), 1.0)
    else:
        m = gl.gl_mesh_create(dim, N, 1.0, gi.WORKLOADS["cube128"][3] if dim == 3 else (0.0, 0.0, 1.0))
    n, _ = gl.gl_mesh_info(m)
    psi, v = (torch.from_numpy(a).to(DEV) for a in (gi.disk(n, 41), gi.complex_normal(n, 42)))
    P = {}
    try:
        for sync in (1, 2):
            P[sync] = gl.gl_precond_setup(m, psi, gl.options(max_coarse=max_coarse, sweep_sync=sync, autotune=0,
                                                             precision=gl.GL_MIXED_PRECOND))
        z = {s: torch.empty_like(v) for s in P}
        for G, K in FORMS:
            form(P[1], G, 1)
            form(P[2], G, K)
            for precision in (gl.GL_FP64, gl.GL_MIXED_PRECOND):
                lv = gl.gl_precond_level_sweep(P[2], 1, precision)
                assert lv["lanes"] == G and lv["sync"] == 1
                for _ in range(3):  # the slots' two sets in turn
                    for s in P:
                        gl.gl_precond_apply_precision(P[s], v, z[s], precision)
                    assert torch.equal(z[1], z[2]), (G, K, precision)
    finally:
        for p in P.values():
            gl.gl_precond_destroy(p)
        gl.gl_mesh_destroy(m)


def test_solve_after_a_change_of_form():
    n = 48 ** 3
    m = gl.gl_mesh_create(3, 48, 1.0, gi.WORKLOADS["cube128"][3])
    psi, b = (torch.from_numpy(a).to(DEV) for a in (gi.disk(n, 43), gi.complex_normal(n, 44)))
    opts = gl.options(max_coarse=64, autotune=0)
    P = gl.gl_precond_setup(m, psi, opts)
    try:
        x = {}
        for G, K in [(8, 1), (2, 2), (8, 1), (8, 2)]:
            form(P, G, K)
            x[G, K] = torch.zeros_like(b)
            st, info = gl.gl_jacobian_solve(m, psi, P, b, x[G, K], opts)
            assert st == 0 and info.converged
        assert torch.equal(x[8, 1], x[8, 2])
        for bad in (0, 64 + 3, 64 + 64 + 64 + 4, 64, 4):
            with pytest.raises(gl.GLError):
                gl.gl_precond_debug(P, gl.GL_DEBUG_SWEEP_FORM + bad)
    finally:
        gl.gl_precond_destroy(P)
        gl.gl_mesh_destroy(m)
