"""The three-level method at every padded sketch size that has a level-3 kernel of its own
(128, 256, 384, and beyond), on clusters of 16 and of 8 CTAs, against the same PCG steps
in FP64 from the handle's own pieces; and solves with more than 4096 columns, where a
thread of the level-1 vector kernels takes two entries of four.

Tolerance of SolveM2 (u = 2^-24): z = (u_3 - v_3) / lam~ is formed from FP32 copies of
the two level-3 solutions, amplified by the cancellation of 1 + |W| / lam~: 4 u (1 + |W| / lam~)."""

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

U32 = 2.0 ** -24
LAM = 1e-3


@pytest.fixture(scope="module")
def ctx():
    from paper_2405_05865_gb300 import Context
    c = Context(0)
    yield c
    c.set_level3_ctas(16)
    c.close()


def _tall(m, n, seed):
    """G diag(d) / sqrt(m): 16 outliers 1e2 -> 1e1 over a tail in [0.5, 1], and lambda0 of the 32 largest."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    d = torch.cat([torch.logspace(2, 1, 16, device="cuda", dtype=torch.float64),
                   0.5 + 0.5 * torch.rand(n - 16, generator=g, device="cuda", dtype=torch.float64)])
    A = torch.randn((m, n), generator=g, device="cuda", dtype=torch.float64) * (d / m ** 0.5)
    return A.float(), 2.0 / 32 * float((d[32:] ** 2).sum()), g


def _pcg(W, shift, M, r, steps):
    L = torch.linalg.cholesky(M)
    solve = lambda v: torch.cholesky_solve(v[:, None], L)[:, 0]
    x = torch.zeros_like(r)
    z = solve(r)
    p, rz = z, r @ z
    for k in range(steps):
        q = W @ p + shift * p
        alpha = rz / (p @ q)
        x, r = x + alpha * p, r - alpha * q
        z = solve(r)
        p, rz = z + (r @ z) / rz * p, r @ z
    return x


@pytest.mark.parametrize("s", [100, 128, 256, 330, 384, 500, 640, 1000])
def test_solve_m2_sizes(ctx, s):
    A, lam0, gen = _tall(6000, 1400, s)
    g = ctx.general(A, LAM, s, lam0=lam0)
    p = g.setup(s)
    At = p["At"].double()
    W = At.T @ At
    lt = LAM + lam0
    bound = 4 * U32 * (1.0 + float(torch.linalg.matrix_norm(W, 2)) / lt)
    r = torch.randn(s, generator=gen, device="cuda", dtype=torch.float32)
    for t3 in (1, 5):
        ref = (_pcg(W, 0.0, p["M3a"], r.double(), t3) - _pcg(W, lt, p["M3b"], r.double(), t3)) / lt
        for ctas in (16, 8):
            ctx.set_level3_ctas(ctas)
            z = g.solve_m2(r, t3).double()
            assert float((z - ref).norm()) <= bound * float(ref.norm()), (ctas, t3)
    g.close()


def test_level3_cluster_sizes_refused(ctx):
    from paper_2405_05865_gb300 import MspError
    for bad in (0, 4, 12, 32):
        with pytest.raises(MspError) as e:
            ctx.set_level3_ctas(bad)
        assert e.value.status == 1


@pytest.mark.parametrize("n", [4096, 4099, 4608, 8192])
@pytest.mark.parametrize("levels", [0, 8])
def test_solve_wide(ctx, n, levels):
    ctx.set_level3_ctas(16)
    A, lam0, gen = _tall(n + n // 2, n, 7)
    g = ctx.general(A, LAM, 128, lam0=lam0)
    c = torch.randn(n, generator=gen, device="cuda", dtype=torch.float64)
    x, info = g.solve(c, tol=1e-10, refine_tol=1e-4, level2_iters=levels, level3_iters=levels, max_outer=400)
    assert info["status"] == 0
    A64 = A.double()
    assert float((c - A64.T @ (A64 @ x) - LAM * x).norm()) <= 1.2e-10 * float(c.norm())
    g.close()
