"""SolveM1 and the solve at the two widest padded sketch sizes (1536 and 2048
columns), on so many rows that part of each block's rows of C stays in global memory,
against the Woodbury form in FP64 from the factor's own pieces."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SEED = 0x4D5350
N, LAM = 6100, 1e-2


@pytest.fixture(scope="module")
def ctx():
    from paper_2405_05865_gb300 import Context
    c = Context(0)
    yield c
    c.close()


@pytest.fixture(scope="module")
def system(ctx):
    g = torch.Generator(device="cuda").manual_seed(5)
    P = torch.rand((N, 3), generator=g, device="cuda", dtype=torch.float64)
    return ctx.rbf_kernel(P, 0.1), torch.randn(N, generator=g, device="cuda", dtype=torch.float64)


@pytest.mark.parametrize("s", [1500, 2048])
@pytest.mark.parametrize("data", ["fp32", "bf16"])
def test_wide_sketches(ctx, system, s, data):
    A, b = system
    sk = ctx.sketch(A, s, 8, SEED)
    lam0 = 1e-3 * N
    f = ctx.nystrom(sk, LAM, lam0, phi=0, data=data)
    p = f.parts()
    C = sk.C().double()
    if data == "bf16":
        C = C.to(torch.bfloat16).double()
    r = b.float()
    w, _ = ctx.solve_m1(f, r, max_inner=0)
    X, r64, lt = torch.tril(p["Linv"].double()), r.double(), LAM + lam0
    ref = (r64 - C @ (X.T @ (X @ (C.T @ r64)))) / lt
    # w = (r - C y) / lam~: C y carries a few FP32 units of |C| |y|, y at most
    # |M2^-1 C^T r|
    y = X.T @ (X @ (C.T @ r64))
    bound = 64 * 2.0 ** -24 * (float(r64.norm()) + float(torch.linalg.matrix_norm(C, 2)) * float(y.norm())) / lt
    assert float((w.double() - ref).norm()) <= bound
    x, info = ctx.solve(f, A, b, LAM, tol=1e-10, max_inner=0, max_outer=2000)
    assert info["status"] == 0
    res = b - (A.double() @ x + LAM * x)
    assert float(res.norm()) <= 1.2e-10 * float(b.norm())
    f.close()
    sk.close()


@pytest.mark.parametrize("n,s", [(16001, 500), (16001, 640), (16001, 1000), (7993, 1500), (7993, 2048)])
@pytest.mark.parametrize("data", ["fp32", "bf16"])
def test_level2_iteration_on_rows_from_global_memory(ctx, n, s, data):
    """The level-2 PCG where each block's rows of C exceed its shared memory (in BF16 they all
    fit up to s = 640): SolveM1 against the exact level 2 in FP64."""
    g = torch.Generator(device="cuda").manual_seed(s)
    G = torch.randn((n, 64), generator=g, device="cuda", dtype=torch.float32) / n ** 0.5
    A = G @ G.T
    A.diagonal().add_(0.5)
    sk = ctx.sketch(A, s, 8, SEED)
    f = ctx.nystrom(sk, LAM, 1.0, phi=4 * s, data=data)
    W, C, lt = f.parts()["W"].double(), sk.C().double(), LAM + 1.0
    if data == "bf16":
        W, C = W.to(torch.bfloat16).double(), C.to(torch.bfloat16).double()
    M = C.T @ C + lt * W
    r = torch.randn(n, generator=g, device="cuda", dtype=torch.float32)
    w, its = ctx.solve_m1(f, r, max_inner=300, inner_tol=1e-7)
    assert 0 < its < 300
    r64 = r.double()
    h = C.T @ r64
    y = torch.linalg.solve(M, h)
    ref = (r64 - C @ y) / lt
    # FP32 units of |r| and |C| |y|, and what the tolerance leaves of y
    ev = torch.linalg.eigvalsh(M)
    c2 = float(torch.linalg.matrix_norm(C, 2))
    bound = (64 * 2.0 ** -24 * (float(r64.norm()) + c2 * float(y.norm())) + c2 * 2e-7 * float(h.norm()) / float(ev[0])) / lt
    assert float((w.double() - ref).norm()) <= bound
    f.close()
    sk.close()
