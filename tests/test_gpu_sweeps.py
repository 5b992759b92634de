"""The coarse levels' symmetric Gauss-Seidel steps: the dataflow form (rows poll the
neighbour values they need) against the grid-barrier form, bit for bit.

Both relax every row from the same neighbour values and sum its entries in the same
order (same lanes per row: the setup timing is off), so R_1 of any vector is the same
bits.  The sizes reach levels with fewer rows than one warp's step, ragged last steps,
short and long rows, and a level with more rows of a colour than the resident warps
take at once; several applications in a row alternate the dataflow form's two sets of
slots.  A vector of NaN must come back as NaN, not as a wait that runs out.
"""
import pytest

import gl_inputs as gi

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1204_5125_gb300 as gl  # noqa: E402

DEV = torch.device("cuda:0")
SIZES = [(2, 20, 16), (2, 45, 24), (2, 300, 512), (3, 18, 24), (3, 37, 64), (3, 112, 4096)]


@pytest.mark.parametrize("precision", [gl.GL_FP64, gl.GL_MIXED_PRECOND], ids=["fp64", "fp32vc"])
@pytest.mark.parametrize("dim,N,max_coarse", SIZES, ids=lambda p: str(p))
def test_dataflow_matches_grid_barrier(dim, N, max_coarse, precision):
    n = N ** dim
    m = gl.gl_mesh_create(dim, N, 1.0, gi.WORKLOADS["cube128"][3] if dim == 3 else (0.0, 0.0, 1.0))
    psi = torch.from_numpy(gi.disk(n, 41)).to(DEV)
    P = {}
    try:
        for sync in (1, 2):
            P[sync] = gl.gl_precond_setup(m, psi, gl.options(max_coarse=max_coarse, sweep_sync=sync, autotune=0,
                                                             precision=precision))
        assert gl.gl_precond_levels(P[1]) >= 3
        assert [gl.gl_precond_level_sweep(P[s], 1, precision)["sync"] for s in (1, 2)] == [0, 1]
        for seed in range(42, 45):
            v = torch.from_numpy(gi.complex_normal(n, seed)).to(DEV)
            z = {s: torch.empty_like(v) for s in P}
            for s in P:
                gl.gl_precond_apply_precision(P[s], v, z[s], precision)
            assert torch.equal(z[1], z[2])
        bad = torch.full_like(v, float("nan"))
        gl.gl_precond_apply_precision(P[2], bad, z[2], precision)
        assert bool(torch.isnan(z[2].real).all())
        gl.gl_precond_apply_precision(P[2], v, z[2], precision)
        assert torch.equal(z[1], z[2])
    finally:
        for p in P.values():
            gl.gl_precond_destroy(p)
        gl.gl_mesh_destroy(m)


@pytest.mark.parametrize("precision", [gl.GL_FP64, gl.GL_MIXED_PRECOND], ids=["fp64", "fp32vc"])
@pytest.mark.parametrize("domain,h", [("circ", 0.35), ("ball", 1.1)])
def test_finest_level_of_a_triangulation(domain, h, precision):
    """On a general mesh the finest level has many colours and takes the same sweeps,
    with the residual scaled by the control volumes."""
    pytest.importorskip("scipy")
    dim, x, simplices = gi.delaunay_domain(domain, h)
    m = gl.gl_mesh_create_simplicial(dim, x, simplices, 1.0)
    n, _ = gl.gl_mesh_info(m)
    psi, v = (torch.from_numpy(a).to(DEV) for a in (gi.disk(n, 46), gi.complex_normal(n, 47)))
    z = []
    try:
        for sync in (1, 2):
            P = gl.gl_precond_setup(m, psi, gl.options(max_coarse=64, sweep_sync=sync, autotune=0,
                                                       precision=precision))
            try:
                assert gl.gl_precond_levels(P) >= 2
                assert gl.gl_precond_level_sweep(P, 0, precision)["sync"] == sync - 1
                z.append(torch.empty_like(v))
                gl.gl_precond_apply_precision(P, v, z[-1], precision)
            finally:
                gl.gl_precond_destroy(P)
        assert torch.equal(z[0], z[1])
    finally:
        gl.gl_mesh_destroy(m)
