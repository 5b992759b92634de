"""The measured FP64 peak bounds what the library's own kernels reach: the FP64 Jacobian
on 128^3 nodes issues 35 FP64 instructions a row (24 for six complex products, eleven for
the local terms), boundary rows included (their slices are padded to six entries but for
whole slices of them, fewer than one in a hundred), in the time of a whole call."""
import pytest

import gl_inputs as gi

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1204_5125_gb300 as gl  # noqa: E402

DEV = torch.device("cuda:0")


def test_fp64_peak_is_not_exceeded():
    n = 128 ** 3
    m = gl.gl_mesh_create(3, 128, 1.0, gi.WORKLOADS["cube128"][3])
    psi, phi = (torch.from_numpy(a).to(DEV) for a in (gi.disk(n, 1), gi.complex_normal(n, 2)))
    y = torch.empty_like(phi)
    try:
        peak = gl.gl_measure_fma_peak(gl.GL_FP64)
        best = float("inf")
        for _ in range(5):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(50):
                gl.gl_jacobian_apply(m, psi, phi, y)
            e1.record()
            e1.synchronize()
            best = min(best, e0.elapsed_time(e1) / 50)
    finally:
        gl.gl_mesh_destroy(m)
    rate = 2 * 35 * 0.99 * n / (best * 1e-3) / 1e9
    print(f"{1e3 * best:.1f} us a call: {rate:.0f} of {peak:.0f} GFLOP/s")
    assert 0.6 * peak < rate < peak
