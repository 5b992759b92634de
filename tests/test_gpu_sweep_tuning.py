"""The timing of the sweeps' forms at setup when their waits run out: the FP32 forms are
timed by the first call that needs them, here with every wait target out of reach.  That
call ends with GL_ERR_TIMEOUT, and the forms kept are those of a setup without timing, not
the launch that returned fastest."""
import pytest

import gl_inputs as gi

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1204_5125_gb300 as gl  # noqa: E402

DEV = torch.device("cuda:0")
GL_ERR_TIMEOUT = 7


@pytest.mark.parametrize("sync", [1, 2], ids=["grid", "dataflow"])
def test_tuning_with_waits_that_run_out(sync):
    n = 48 ** 3
    m = gl.gl_mesh_create(3, 48, 1.0, gi.WORKLOADS["cube128"][3])
    psi, b = (torch.from_numpy(a).to(DEV) for a in (gi.disk(n, 21), gi.complex_normal(n, 22)))
    P = {a: gl.gl_precond_setup(m, psi, gl.options(max_coarse=64, autotune=a, sweep_sync=sync)) for a in (0, 1)}
    z = {a: torch.empty_like(b) for a in P}
    try:
        assert gl.gl_precond_levels(P[1]) >= 3
        gl.gl_precond_apply_precision(P[0], b, z[0], gl.GL_MIXED_PRECOND)
        gl.gl_precond_debug(P[1], gl.GL_DEBUG_STALL_SWEEPS)
        with pytest.raises(gl.GLError) as e:
            gl.gl_precond_apply_precision(P[1], b, z[1], gl.GL_MIXED_PRECOND)
        assert e.value.status == GL_ERR_TIMEOUT
        for l in range(1, gl.gl_precond_levels(P[1]) - 1):
            form = [gl.gl_precond_level_sweep(P[a], l, gl.GL_MIXED_PRECOND) for a in (0, 1)]
            assert form[0] == form[1], l
        gl.gl_precond_apply_precision(P[1], b, z[1], gl.GL_MIXED_PRECOND)
        # the same sweeps; the restriction's lanes may differ, which is its rounding in FP32
        assert float(torch.linalg.vector_norm(z[1] - z[0]) / torch.linalg.vector_norm(z[0])) <= 2 ** 8 * 2.0 ** -24
    finally:
        for p in P.values():
            gl.gl_precond_destroy(p)
        gl.gl_mesh_destroy(m)


@pytest.mark.parametrize("precision", [gl.GL_FP64, gl.GL_MIXED_PRECOND], ids=["fp64", "fp32vc"])
def test_long_rows_are_timed_on_more_lanes(precision):
    # 97^3: level 1 has 33 entries a row, level 2 (1252 nodes) 55
    n = 97 ** 3
    m = gl.gl_mesh_create(3, 97, 1.0, gi.WORKLOADS["cube128"][3])
    psi, b = (torch.from_numpy(a).to(DEV) for a in (gi.disk(n, 23), gi.complex_normal(n, 24)))
    P = {a: gl.gl_precond_setup(m, psi, gl.options(autotune=a, precision=precision)) for a in (0, 1)}
    z = {a: torch.empty_like(b) for a in P}
    try:
        assert gl.gl_precond_levels(P[1]) == 4
        rows = [gl.gl_precond_level_info(P[1], l) for l in (1, 2)]
        assert rows[0]["nnz"] < 48 * rows[0]["n"] and rows[1]["nnz"] >= 49 * rows[1]["n"]
        assert gl.gl_precond_level_sweep(P[1], 1, precision)["lanes"] in (2, 4, 8)
        assert gl.gl_precond_level_sweep(P[1], 2, precision)["lanes"] in (4, 8, 16)
        if precision == gl.GL_FP64:  # 185 us on sixteen, 226 on eight
            assert gl.gl_precond_level_sweep(P[1], 2, precision)["lanes"] == 16
        for a in P:
            gl.gl_precond_apply_precision(P[a], b, z[a], precision)
        eps = 2.0 ** -24 if precision != gl.GL_FP64 else 2.0 ** -53
        assert float(torch.linalg.vector_norm(z[1] - z[0]) / torch.linalg.vector_norm(z[0])) <= 2 ** 8 * eps
    finally:
        for p in P.values():
            gl.gl_precond_destroy(p)
        gl.gl_mesh_destroy(m)
