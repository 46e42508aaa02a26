"""msp_sketch_get_C into what the copy kernel takes (device memory of the context's GPU,
managed memory) and into what is left to the copies (rows off 16-byte boundaries, pinned
host memory): the same C. (Memory of another GPU, also left to the copies, needs a second
device.)"""

import ctypes as C

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sketch():
    from paper_2405_05865_gb300 import Context
    ctx = Context(0)
    g = torch.Generator(device="cuda").manual_seed(2)
    A = ctx.rbf_kernel(torch.rand((901, 3), generator=g, device="cuda", dtype=torch.float64), 0.1)
    sk = ctx.sketch(A, 132, 8)
    yield ctx, sk, sk.C().clone()
    sk.close()
    ctx.close()


def _get(ctx, sk, ptr, ldc):
    from paper_2405_05865_gb300 import _lib
    _lib.check(ctx.ptr, ctx.lib.msp_sketch_get_C(ctx.ptr, sk.handle, C.c_void_p(ptr), ldc))
    torch.cuda.synchronize()


@pytest.mark.parametrize("ldc,offset", [(132, 0), (136, 4), (133, 0), (136, 1)])
def test_device(sketch, ldc, offset):
    ctx, sk, want = sketch
    buf = torch.full((901 * ldc + offset,), 7.0, device="cuda", dtype=torch.float32)
    _get(ctx, sk, buf.data_ptr() + 4 * offset, ldc)
    out = buf[offset:].view(901, ldc)
    assert torch.equal(out[:, :132], want)
    assert bool((out[:, 132:] == 7.0).all()) and bool((buf[:offset] == 7.0).all())


def test_pinned_host(sketch):
    ctx, sk, want = sketch
    out = torch.zeros((901, 132), dtype=torch.float32, pin_memory=True)
    _get(ctx, sk, out.data_ptr(), 132)
    assert torch.equal(out, want.cpu())


def test_managed(sketch):
    ctx, sk, want = sketch
    cu = C.CDLL("libcuda.so.1")
    p = C.c_uint64()
    assert cu.cuMemAllocManaged(C.byref(p), C.c_size_t(901 * 132 * 4), 1) == 0
    try:
        _get(ctx, sk, p.value, 132)
        got = torch.frombuffer((C.c_float * (901 * 132)).from_address(p.value), dtype=torch.float32).clone()
        assert torch.equal(got.view(901, 132), want.cpu())
    finally:
        assert cu.cuMemFree_v2(p) == 0
