"""The node-order operators where the result's memory begins inside an argument's or ends
in it: the same bits as with vectors of their own.  Equal pointers stay refused."""
import ctypes

import pytest

import gl_inputs as gi

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1204_5125_gb300 as gl  # noqa: E402

DEV = torch.device("cuda:0")


def noalloc(m, psi, phi, y):
    p = [ctypes.c_void_p(t.data_ptr()) for t in (psi, phi, y)]
    st = gl.library().gl_jacobian_apply_noalloc(m, *p, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    if st:
        raise gl.GLError(st, gl.gl_last_error())


@pytest.mark.parametrize("dim,N", [(2, 33), (2, 300), (3, 40)], ids=str)
def test_result_partly_over_an_argument(dim, N):
    n = N ** dim
    m = gl.gl_mesh_create(dim, N, 1.0)
    psi, phi = (torch.from_numpy(a).to(DEV) for a in (gi.disk(n, 11), gi.complex_normal(n, 12)))
    calls = {"residual": (lambda a, b, y: gl.gl_residual(m, a, y), (0,)),
             "jacobian": (lambda a, b, y: gl.gl_jacobian_apply(m, a, b, y), (0, 1)),
             "noalloc": (lambda a, b, y: noalloc(m, a, b, y), (0, 1))}
    try:
        for f, over in calls.values():
            ref = torch.empty_like(psi)
            f(psi, phi, ref)
            for arg in over:
                for off in (1, n // 3, n - 1):
                    for first in (True, False):  # the argument or the result at the lower address
                        buf = torch.empty(n + off, dtype=torch.complex128, device=DEV)
                        a, y = (buf[:n], buf[off:]) if first else (buf[off:], buf[:n])
                        a.copy_((psi, phi)[arg])
                        args = [psi, phi]
                        args[arg] = a
                        f(*args, y)
                        assert torch.equal(y, ref)
            for arg in over:
                same = [psi.clone(), phi.clone()]
                with pytest.raises(gl.GLError) as e:
                    f(*same, same[arg])
                assert e.value.status == 1
    finally:
        gl.gl_mesh_destroy(m)
