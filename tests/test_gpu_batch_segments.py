"""The batched solve at the edges of its work items: one row block and one factor
chunk (n = 100), exactly one and just over one G segment of 10 row blocks (n = 1280,
1290), and a ragged sketch size; every column against the dense solution of the FP64
system through |x - x*| <= |r| / lam."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import reference
from workloads import rbf_kernel, rbf_points

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[(100, 64)], [(1280, 320), (1290, 200), (100, 64)], [(2600, 640), (300, 96)]])
def test_batch_item_edges(sizes):
    from paper_2405_05865_gb300 import Context
    ctx = Context(0)
    lam, insts, host = 1e-2, [], []
    for k, (n, s) in enumerate(sizes):
        K = rbf_kernel(rbf_points(n, seed=k), 0.08, out_dtype=np.float32)
        B = np.random.default_rng(k).standard_normal((n, 5))
        host.append((K, B))
        insts.append(dict(A=torch.from_numpy(K).cuda(), B=torch.from_numpy(B).cuda(), lam=lam, s=s))
    bt = ctx.batch(insts)
    infos = bt.solve(tol=1e-9, refine_tol=1e-4)
    for k, (K, B) in enumerate(host):
        X = bt.X(k).cpu().numpy()
        A = K.astype(np.float64)
        for j in range(B.shape[1]):
            r = np.linalg.norm(B[:, j] - A @ X[:, j] - lam * X[:, j])
            assert r <= 1.01e-9 * np.linalg.norm(B[:, j])
        xs = reference.solve_dense(A, B[:, 0], lam)
        assert np.linalg.norm(X[:, 0] - xs) <= 1.01e-9 * np.linalg.norm(B[:, 0]) / lam
        assert infos[k]["status"] == 0
    bt.close()
    ctx.close()


@pytest.mark.parametrize("count,s", [(56, 500), (57, 500), (115, 200)])
def test_many_factor_chunks(count, s):
    """Just below and at the number of factor chunks where their items have 64 rows (912
    chunks of 32 on 152 SMs), and short factors (s_pad = 256); every column's FP64
    residual against the stopping rule."""
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
