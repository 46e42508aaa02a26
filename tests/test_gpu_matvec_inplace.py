"""msp_matvec_f64 with y over x (the caller's own buffer): the FP32 product splits x into
two floats ahead of the pass, or beside it where the result goes elsewhere."""

import ctypes as C

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [128, 512, 1000, 1024, 1028, 1400, 1536, 1540])
def test_y_over_x(n):
    from paper_2405_05865_gb300 import Context, _lib
    ctx = Context(0)
    g = torch.Generator(device="cuda").manual_seed(n)
    A = torch.randn((n, n), generator=g, device="cuda", dtype=torch.float32)
    x = torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
    want = ctx.matvec_f64(A, x, 0.25)
    ref = A.double() @ x + 0.25 * x
    assert float((want - ref).abs().max()) <= 1e-12 * float((A.double().abs() @ x.abs()).max())
    for _ in range(20):
        y = x.clone()
        p = C.c_void_p(y.data_ptr())
        _lib.check(ctx.ptr, ctx.lib.msp_matvec_f64(ctx.ptr, C.c_void_p(A.data_ptr()), _lib.MSP_F32, n, n, 0.25, p, p))
        torch.cuda.synchronize()
        # apart or in place: the same sums over the same pairs
        assert torch.equal(y, want)
    ctx.close()
