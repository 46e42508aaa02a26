"""Breakdowns of the mixed-precision solve (packed A pass) report MSP_ENOTPD at once,
whichever launch finds them, and leave the context usable.

A = -5 I is negative definite, and M2 = 25 P - 5 lam~ P with P = Pi^T Pi is positive
definite for lam~ < 5. lam~ = 0.01: z = M^{-1} r lies mostly outside the sketch's range,
where M^{-1} = I / lam~, so r^T z > 0 and p^T (A + lam I) p < 0 (found by the level-2
launch that forms the step). lam~ = 4.91: M^{-1} = -I / (5 - lam~) on the range
outweighs I / lam~ outside it, so r^T z < 0 (found by the A pass)."""

import time

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SEED = 0x4D5350
LAM = 1e-2


@pytest.fixture(scope="module")
def ctx():
    from paper_2405_05865_gb300 import Context
    c = Context(0)
    yield c
    c.close()


def _negative(ctx, n, lam0):
    A = -5.0 * torch.eye(n, device="cuda", dtype=torch.float32)
    b = torch.randn(n, generator=torch.Generator(device="cuda").manual_seed(n), device="cuda", dtype=torch.float64)
    sk = ctx.sketch(A, 32 if n < 2000 else n // 8, 4, SEED)
    return A, b, ctx.nystrom(sk, LAM, lam0, phi=0)


def _expect_not_pd(ctx, A, b, f):
    from paper_2405_05865_gb300 import MspError
    t0 = time.monotonic()
    with pytest.raises(MspError) as e:
        ctx.solve(f, A, b, LAM, precision="mixed", max_inner=0)
    assert e.value.status == 4
    assert time.monotonic() - t0 < 1.0


@pytest.mark.parametrize("n", [40, 100, 151, 256, 1000, 4096])   # the first three: fewer rows than SMs
@pytest.mark.parametrize("lam0", [0.0, 4.9])
def test_negative_definite_mixed(ctx, n, lam0):
    A, b, f = _negative(ctx, n, lam0)
    for _ in range(10):
        _expect_not_pd(ctx, A, b, f)
    f.close()
    B = torch.eye(n, device="cuda", dtype=torch.float32)
    f = ctx.nystrom(ctx.sketch(B, 32, 4, SEED), LAM, 0.0, phi=0)
    x, info = ctx.solve(f, B, b, LAM, precision="mixed", max_inner=0)
    assert info["status"] == 0 and torch.allclose(x, b / (1.0 + LAM), rtol=1e-9, atol=1e-9)
    f.close()
