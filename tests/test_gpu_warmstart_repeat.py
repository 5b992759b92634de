"""The gradient of the learned warm start, call after call.  Its reductions have a fixed
order, so equal inputs give equal bits; a warp of a backward layer that misses a tile's
completion would run its wait out (GL_ERR_TIMEOUT) and leave its quarter of dW at zero.
One tile a block, two, three (where a buffer of the accumulators comes round again) and
many, the last one ragged.
"""
import numpy as np
import pytest

import gl_inputs as gi

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1204_5125_gb300 as gl  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("dim,N", [(2, 11), (2, 190), (2, 237), (3, 63)], ids=str)
def test_gradient_repeats_bit_for_bit(dim, N):
    n = N ** dim
    m = gl.gl_mesh_create(dim, N, 1.0, gi.WORKLOADS["cube128"][3] if dim == 3 else (0.0, 0.0, 1.0))
    psi, b = (torch.from_numpy(a).to(DEV) for a in (gi.disk(n, 91), gi.complex_normal(n, 92)))
    ws = gl.gl_warmstart_create(gi.warmstart_init(11))
    try:
        loss, grad = gl.gl_warmstart_grad(ws, m, psi, b)
        # every warp of the first layer wrote its 32 inputs (each has the constant or a feature)
        assert grad[: 64 * 128].reshape(64, 4, 32).any(axis=(0, 2)).all()
        for _ in range(40):
            again = gl.gl_warmstart_grad(ws, m, psi, b)
            assert again[0] == loss and np.array_equal(again[1], grad)
    finally:
        gl.gl_warmstart_destroy(ws)
        gl.gl_mesh_destroy(m)
