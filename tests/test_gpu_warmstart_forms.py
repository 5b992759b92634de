"""The learned warm start where its tiling ends: one ragged tile, more tiles than SMs (a
block builds several, from buffers it reuses), rows wider than the staged K entries and
meshes whose slices differ in width, with and without the hint's channels.

Bars: activations and aggregated features rounded to BF16 (2^-9) over four layers, 2e-2 in
norm for the guess, as in the other forward tests.  A gradient sums terms of either sign
over the nodes, which magnifies those roundings (to 0.13 in norm on a cube of 63^3 nodes),
so it is compared with a reference that rounds at the same places: what is left are values
next to a rounding boundary that FP32 sums (relative error up to 1e-6 in dy) take to the
other side, 5e-4 of them, 0.04 of the whole roundings' effect in the mean square: 5e-3,
and the bar is four times that.
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


def bf16(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.float32)).to(torch.bfloat16).double().numpy()


def rounded_loss_and_grad(theta, g, psi, b):
    """ows.loss_and_grad with the kernels' roundings to BF16: activations, aggregated
    features, weights and dz; everything else in FP64."""
    Ws, U = ows.split(theta.astype(np.float64))
    bhat = b / g.dnorm(b)
    h = bf16(ows.features(g, psi, bhat))
    hs, As = [h], []
    for W in Ws:
        As.append(np.concatenate([h, bf16(g.aggregate(h))], axis=1))
        h = np.maximum(As[-1] @ bf16(W).T, 0.0)
        h[:, ows.C - 1] = 1.0
        h = bf16(h)
        hs.append(h)
    y = h @ U.T
    xhat = (y[:, 0] + 1j * y[:, 1]) / g.kdiag
    r = bhat - g.mesh.jacobian(psi, xhat)
    gy = -2.0 * g.vol * g.mesh.jacobian(psi, r) / g.kdiag
    dy = np.stack([gy.real, gy.imag], axis=1)
    dh, dWs = dy @ U, [None] * ows.LAYERS
    for l in range(ows.LAYERS - 1, -1, -1):
        dz = dh * (hs[l + 1] > 0.0)
        dz[:, ows.C - 1] = 0.0
        dz = bf16(dz)
        dWs[l] = dz.T @ As[l]
        da = dz @ bf16(Ws[l])
        dh = da[:, :ows.C] + g.aggregate_adjoint(da[:, ows.C:])
    return float(np.sum(g.vol * np.abs(r) ** 2)), np.concatenate([w.ravel() for w in dWs] + [(dy.T @ h).ravel()])


@pytest.mark.parametrize("case", [(2, 150), (3, 45), ("circ", 0.35), ("ball", 1.1)], ids=str)
def test_gradient_forms(oracle_mod, case):
    m, om = meshes(oracle_mod, case)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)  # noqa: E731
    psi, b = gi.disk(om.n, 71), gi.complex_normal(om.n, 72)
    theta = gi.warmstart_init(10)
    ws = gl.gl_warmstart_create(theta)
    try:
        L, grad = gl.gl_warmstart_grad(ws, m, dev(psi), dev(b))
        Lo, go = rounded_loss_and_grad(theta, ows.Graph(om), psi, b)
        assert abs(L - Lo) <= 1e-3 * Lo, (L, Lo)
        Ws, U = ows.split(np.arange(ows.NPARAM))
        for name, idx in [("W0", Ws[0]), ("W1", Ws[1]), ("W2", Ws[2]), ("W3", Ws[3]), ("U", U)]:
            x, e = grad[idx.ravel()].astype(np.float64), go[idx.ravel()]
            err = np.linalg.norm(x - e) / np.linalg.norm(e)
            assert err <= 2e-2, (name, err)
    finally:
        gl.gl_warmstart_destroy(ws)
        gl.gl_mesh_destroy(m)
