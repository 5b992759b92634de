"""Solves without a preconditioner on meshes made and destroyed in turn: a square and a
cube of equally many nodes, so that the next mesh finds the last one's address and
buffers free.  A captured solve kept from the destroyed mesh would read its operator.

Bound: the true residual that the solve reports is at most tol; the same residual from the
oracle's Jacobian differs by rounding only (1e-3 of tol is far more)."""
import numpy as np
import pytest

import gl_inputs as gi

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1204_5125_gb300 as gl  # noqa: E402

DEV = torch.device("cuda:0")
TOL = 1e-8


@pytest.mark.parametrize("device_loop", [1, 0], ids=["device", "host"])
def test_solves_over_meshes_made_in_turn(oracle_mod, device_loop):
    n = 4096
    psi, b = gi.psi_noisy_one(n, 51), gi.complex_normal(n, 52)
    tp, tb = torch.from_numpy(psi).to(DEV), torch.from_numpy(b).to(DEV)
    opts = gl.options(cycles=0, tol=TOL, maxit=4000, device_loop=device_loop)
    for dim, N in [(2, 64), (3, 16), (2, 64), (3, 16)]:
        field = (0.0, 0.0, 1.0) if dim == 2 else gi.WORKLOADS["cube128"][3]
        m = gl.gl_mesh_create(dim, N, 1.0, field, edge=7.0)
        om = oracle_mod.Mesh(dim, N, 1.0, field, edge=7.0)
        try:
            x = torch.zeros_like(tb)
            st, info = gl.gl_jacobian_solve(m, tp, None, tb, x, opts)
            assert st == 0 and info.converged, info.as_dict()
        finally:
            gl.gl_mesh_destroy(m)
        vol = om.volumes()
        r = b - om.jacobian(psi, x.cpu().numpy())
        assert np.sqrt(np.sum(vol * np.abs(r) ** 2) / np.sum(vol * np.abs(b) ** 2)) <= 1.001 * TOL
