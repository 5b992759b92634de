"""The finest level of a triangulation on either side of the size where its Gauss-Seidel
steps go from one launch to a launch per colour: R_1 in FP32 against R_1 in FP64, whose
line lies at twice the size, so that the two V-cycles relax that level in different forms.

Bound: 2^8 eps, as for the FP32 V-cycle elsewhere (a row's sum of 7 products, the residual
and the transfers, over the levels)."""
import numpy as np
import pytest

import gl_inputs as gi

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1204_5125_gb300 as gl  # noqa: E402

DEV = torch.device("cuda:0")


def triangular_lattice(N):
    j, i = np.divmod(np.arange(N * N), N)
    x = np.stack([i + 0.5 * (j % 2), j * np.sqrt(0.75), 0.0 * i], axis=1) * (7.0 / N)
    a = (np.arange(N - 1)[:, None] * N + np.arange(N - 1)).ravel()
    odd = ((a // N) % 2 == 1)[:, None]
    lower = np.where(odd, np.stack([a, a + 1, a + N + 1], 1), np.stack([a, a + 1, a + N], 1))
    upper = np.where(odd, np.stack([a, a + N + 1, a + N], 1), np.stack([a + 1, a + N + 1, a + N], 1))
    return x, np.concatenate([lower, upper]).astype(np.int32)


@pytest.mark.parametrize("N,sync,form", [(1024, 2, 1), (1025, 2, -1), (886, 1, 0), (887, 1, -1)])
def test_forms_of_the_finest_level(N, sync, form):
    n = N * N
    x, simplices = triangular_lattice(N)
    m = gl.gl_mesh_create_simplicial(2, x, simplices, 1.0)
    psi, v = (torch.from_numpy(a).to(DEV) for a in (gi.psi_noisy_one(n, 61), gi.complex_normal(n, 62)))
    P = gl.gl_precond_setup(m, psi, gl.options(precision=gl.GL_MIXED_PRECOND, autotune=0, sweep_sync=sync))
    try:
        z = {}
        for precision, want in ((gl.GL_FP64, sync - 1), (gl.GL_MIXED_PRECOND, form)):
            assert gl.gl_precond_level_sweep(P, 0, precision)["sync"] == want
            assert gl.gl_precond_level_sweep(P, 1, precision)["sync"] == sync - 1
            z[precision] = torch.empty_like(v)
            gl.gl_precond_apply_precision(P, v, z[precision], precision)
        d = z[gl.GL_MIXED_PRECOND] - z[gl.GL_FP64]
        assert float(torch.linalg.vector_norm(d) / torch.linalg.vector_norm(z[gl.GL_FP64])) <= 2 ** 8 * 2.0 ** -24
    finally:
        gl.gl_precond_destroy(P)
        gl.gl_mesh_destroy(m)
