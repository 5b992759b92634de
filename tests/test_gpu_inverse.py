"""The dense coarsest inverse at the edges of its 16-row pivot blocks and 32 x 32 tiles:
on a one-level hierarchy R_1 v = P-hat^-1 D v with the inverse of the whole operator.

Bound: z = X (D v) with X the computed inverse.  Every entry of X is the result of at
most n updates with one product each, so the residual D v - P-hat z is at most a small
multiple of n eps ||P-hat|| ||z||; 8 covers the complex products and the sum of X's row."""
import numpy as np
import pytest

import gl_inputs as gi

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1204_5125_gb300 as gl  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("dim,N", [(2, 2), (3, 2), (2, 4), (2, 5), (3, 3), (2, 6), (2, 7), (2, 8), (2, 9), (3, 5), (2, 23),
                                   (3, 12)], ids=lambda p: str(p))
def test_inverse_residual(dim, N):
    n = N ** dim
    m = gl.gl_mesh_create(dim, N, 1.0)
    psi = torch.from_numpy(gi.psi_noisy_one(n, 71)).to(DEV)
    P = gl.gl_precond_setup(m, psi, gl.options(max_coarse=4096))
    try:
        assert gl.gl_precond_levels(P) == 1
        rp, ci, v = gl.gl_precond_level_matrix(P, 0)
        A = np.zeros((n, n), complex)
        A[np.repeat(np.arange(n), np.diff(rp)), ci] = v
        vol = torch.empty(n, dtype=torch.float64, device=DEV)
        gl.gl_mesh_info(m, vol)
        b = torch.from_numpy(gi.complex_normal(n, 72)).to(DEV)
        z = torch.empty_like(b)
        gl.gl_precond_apply(P, b, z)
        z, d = z.cpu().numpy(), (vol * b).cpu().numpy()
        res = np.linalg.norm(A @ z - d) / (np.linalg.norm(A, 2) * np.linalg.norm(z))
        print(f"n={n}: residual {res:.2e}")
        assert res <= 8 * n * 2.0 ** -52
    finally:
        gl.gl_precond_destroy(P)
        gl.gl_mesh_destroy(m)
