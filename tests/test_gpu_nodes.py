"""The FP64 Jacobian and residual of the public calls run on node-order vectors; meshes
whose node count is not a multiple of a 32-row slice (down to 4 nodes), odd and even
sides, and a general triangulation, against the oracle.

Bound: a row sums at most w + 4 products (w its stored neighbours, at most 16 here), so
|y - y_ref| is within 64 eps of the row's magnitude sum."""
import numpy as np
import pytest

import gl_inputs as gi

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1204_5125_gb300 as gl  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("kind,N", [("2d", 2), ("2d", 5), ("2d", 6), ("2d", 33), ("3d", 2), ("3d", 3), ("3d", 10),
                                    ("circ", 0.9)], ids=lambda p: str(p))
def test_node_order_operators(oracle_mod, kind, N):
    if kind == "circ":
        pytest.importorskip("scipy")
        dim, x, sp = gi.delaunay_domain("circ", N)
        m, om = gl.gl_mesh_create_simplicial(dim, x, sp, 1.0), oracle_mod.Mesh.from_simplices(dim, x, sp, 1.0)
    else:
        m, om = gl.gl_mesh_create(int(kind[0]), N, 1.0), oracle_mod.Mesh(int(kind[0]), N, 1.0)
    n = om.n
    try:
        psi, phi = gi.disk(n, 81), gi.complex_normal(n, 82)
        tp, tf = torch.from_numpy(psi).to(DEV), torch.from_numpy(phi).to(DEV)
        y, r = torch.empty_like(tp), torch.empty_like(tp)
        gl.gl_jacobian_apply(m, tp, tf, y)
        gl.gl_residual(m, tp, r)
        rp, ci, v = om.khat_csr()
        vol = om.volumes()
        mag = lambda u: np.add.reduceat(np.abs(v) * np.abs(u)[ci], rp[:-1]) / vol + 4 * np.abs(u)  # noqa: E731
        eps = 2.0 ** -52
        assert (np.abs(y.cpu().numpy() - om.jacobian(psi, phi)) <= 64 * eps * mag(phi)).all()
        assert (np.abs(r.cpu().numpy() - om.residual(psi)) <= 64 * eps * mag(psi)).all()
    finally:
        gl.gl_mesh_destroy(m)
