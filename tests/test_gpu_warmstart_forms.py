"""The learned warm start where its tiling ends: one ragged tile, more tiles than SMs (a
block builds several, from buffers it reuses), rows wider than the staged K entries and
meshes whose slices differ in width, with and without the hint's channels.

Bar as for the other forward tests: activations and aggregated features rounded to BF16
(2^-9) over four layers, 2e-2 in norm.
"""
import numpy as np
import pytest

import gl_inputs as gi
from oracle import warmstart as ows

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1204_5125_gb300 as gl  # noqa: E402

DEV = torch.device("cuda:0")
INV_SQRT3 = 1.0 / np.sqrt(3.0)


def meshes(oracle_mod, case):
    if isinstance(case[0], str):
        pytest.importorskip("scipy")
        dim, x, sp = gi.delaunay_domain(*case)
        return gl.gl_mesh_create_simplicial(dim, x, sp, 1.0), oracle_mod.Mesh.from_simplices(dim, x, sp, 1.0)
    dim, N = case
    field = (INV_SQRT3,) * 3 if dim == 3 else (0.0, 0.0, 1.0)
    return gl.gl_mesh_create(dim, N, 1.0, field), oracle_mod.Mesh(dim, N, 1.0, field)


@pytest.mark.parametrize("hint", [False, True], ids=["plain", "hint"])
@pytest.mark.parametrize("case", [(2, 3), (2, 150), (3, 45), ("circ", 0.35), ("ball", 1.1)], ids=str)
def test_forward_forms(oracle_mod, case, hint):
    m, om = meshes(oracle_mod, case)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)  # noqa: E731
    psi, b = gi.disk(om.n, 61), gi.complex_normal(om.n, 62)
    a = gi.complex_normal(om.n, 63) + 0.5 * b if hint else None
    theta = gi.warmstart_init(9)
    ws = gl.gl_warmstart_create(theta)
    try:
        x0 = torch.zeros(om.n, dtype=torch.complex128, device=DEV)
        kw = {"hint": dev(a)} if hint else {}
        gl.gl_warmstart_predict(ws, m, dev(psi), dev(b), x0, **kw)
        g = ows.Graph(om)
        args = (g, psi, b, a) if hint else (g, psi, b)
        base = ows.predict(np.zeros(ows.NPARAM), *args)
        expect = ows.predict(theta.astype(np.float64), *args)
        err = np.linalg.norm(x0.cpu().numpy() - expect) / np.linalg.norm(expect - base)
        assert err <= 2e-2, err
    finally:
        gl.gl_warmstart_destroy(ws)
        gl.gl_mesh_destroy(m)
