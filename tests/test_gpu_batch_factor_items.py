"""The batched factor steps on either side of the line where their items have 64 rows
instead of 32 (two 32-row chunks for each of 152 SMs), with long and short factors: every
column's FP64 residual against the stopping rule."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from workloads import rbf_kernel, rbf_points

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count,s", [(18, 500), (19, 500), (37, 200), (38, 200), (76, 100)])
def test_factor_items(count, s):
    from paper_2405_05865_gb300 import Context
    ctx = Context(0)
    lam, n = 1e-2, 540
    A = torch.from_numpy(rbf_kernel(rbf_points(n, seed=9), 0.08, out_dtype=np.float32)).cuda()
    gen = torch.Generator(device="cuda").manual_seed(count)
    Bs = [torch.randn((n, 3), generator=gen, device="cuda", dtype=torch.float64) for _ in range(count)]
    bt = ctx.batch([dict(A=A, B=B, lam=lam, s=s) for B in Bs])
    bt.solve(tol=1e-9, refine_tol=1e-4)
    Ad = A.double()
    for k, B in enumerate(Bs):
        X = bt.X(k)
        r = (B - Ad @ X - lam * X).norm(dim=0)
        assert bool((r <= 1.01e-9 * B.norm(dim=0)).all())
    bt.close()
    ctx.close()
