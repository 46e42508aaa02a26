"""SolveM1 with a sketched level 2 (phi > 0): the sizes whose level-2 iteration runs
on the formed operator in one cluster (padded sketch sizes 128, 256 and, in FP32, 384)
and the next size up, which iterates by passes over C, against the FP64 oracle's exact
level-2 solve of the same matrix."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import msp as omsp

pytestmark = pytest.mark.gpu

SEED = 0x4D5350
LAM = 1e-2


@pytest.fixture(scope="module")
def ctx():
    from paper_2405_05865_gb300 import Context
    c = Context(0)
    yield c
    c.close()


@pytest.fixture(scope="module")
def matrix():
    n = 901
    Q, _ = np.linalg.qr(np.random.default_rng(12).standard_normal((n, n)))
    A = (Q * np.logspace(2, -3, n) ** 0.4) @ Q.T
    return 0.5 * (A + A.T), np.random.default_rng(1).standard_normal(n)


@pytest.mark.parametrize("s", [16, 128, 130, 256, 300, 384, 400])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_solve_m1_sketched_level2(ctx, matrix, s, dtype):
    A, r = matrix
    if dtype == torch.float32:
        A = A.astype(np.float32).astype(np.float64)
        r = r.astype(np.float32).astype(np.float64)
    sk = ctx.sketch(torch.from_numpy(A).to("cuda", dtype), s, 8, SEED)
    f = ctx.nystrom(sk, LAM, 0.0, phi=4 * s, gamma_phi=8, seed=SEED)
    w, its = ctx.solve_m1(f, torch.from_numpy(r).to("cuda", dtype), max_inner=300,
                          inner_tol=1e-14 if dtype == torch.float64 else 1e-7)
    p = omsp.MspParams(s=s, phi=4 * s, lam0=0.0, inner="exact")
    ref = omsp.solve_m1(omsp.setup(A, LAM, p), r, p)
    err = np.linalg.norm(w.double().cpu().numpy() - ref)
    assert 0 < its <= 300
    if dtype == torch.float64:
        # as the FP64 test of the same matrix family at s = 64
        assert err <= 1e-9 * np.linalg.norm(ref)
    else:
        # w = (r - C y) / lam: the difference carries a few units of |r|, times the
        # condition |A| / lam of the level-2 system
        assert err <= 64 * 2.0 ** -24 * (np.linalg.norm(A, 2) / LAM) * np.linalg.norm(r) / LAM
    # a few steps only: the cap holds
    _, its = ctx.solve_m1(f, torch.from_numpy(r).to("cuda", dtype), max_inner=3, inner_tol=1e-14)
    assert its == 3
    f.close()
    sk.close()
