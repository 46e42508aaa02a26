"""The unit width of the batched A passes selects how the work is cut, not how far the
FP32 sums run: the solution's true residual (FP64) is the same with units of 16 tiles and
with whole rows (64 tiles and more)."""

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

LAM = 1e-2


def test_residual_does_not_follow_the_unit_width():
    from paper_2405_05865_gb300 import Context
    ctx = Context(0)
    g = torch.Generator(device="cuda").manual_seed(9)
    insts = []
    for n in (4096, 3001):
        A = ctx.rbf_kernel(torch.rand((n, 3), generator=g, device="cuda", dtype=torch.float64), 0.07)
        insts.append(dict(A=A, B=torch.randn((n, 16), generator=g, device="cuda", dtype=torch.float64), lam=LAM,
                          s=n // 4 // 64 * 64))
    rel = {}
    for ut in (16, 64, 256):
        bt = ctx.batch(insts)
        assert bt.autotune(ut) == ut
        bt.solve(tol=1e-10, refine_tol=1e-4)
        rel[ut] = []
        for k, I in enumerate(insts):
            R = I["B"] - I["A"].double() @ bt.X(k) - LAM * bt.X(k)
            rel[ut].append(float((R.norm(dim=0) / I["B"].norm(dim=0)).square().mean().sqrt()))
        bt.close()
    for ut in (64, 256):
        for k in range(len(insts)):
            # 16 right-hand sides' mean: sums of the same length, in another order
            assert rel[ut][k] <= 1.5 * rel[16][k], rel
    ctx.close()
