"""The default colouring on the device against the oracle's sequential one on the same level
graph, colour for colour: levels of fewer vertices than a block, with rows shorter and
longer than the eight neighbours read at a time, and chains of dependent vertices."""
import numpy as np
import pytest

import gl_inputs as gi

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1204_5125_gb300 as gl  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("dim,N,max_coarse", [(2, 24, 8), (2, 301, 64), (3, 12, 8), (3, 48, 128)])
def test_colours_match_the_sequential_order(oracle_mod, dim, N, max_coarse):
    m = gl.gl_mesh_create(dim, N, 1.0, gi.WORKLOADS["cube128"][3] if dim == 3 else (0.0, 0.0, 1.0))
    psi = torch.from_numpy(gi.disk(N ** dim, 81)).to(DEV)
    G = gl.gl_precond_setup(m, psi, gl.options(max_coarse=max_coarse, autotune=0))
    try:
        levels = gl.gl_precond_levels(G)
        assert levels >= 3
        for lv in range(1, levels - 1):
            rp, ci, _ = gl.gl_precond_level_matrix(G, lv)
            np.testing.assert_array_equal(gl.gl_precond_level_colors(G, lv), oracle_mod.color_psl(rp, ci)[1])
    finally:
        gl.gl_precond_destroy(G)
        gl.gl_mesh_destroy(m)
