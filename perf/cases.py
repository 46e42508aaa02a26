"""Timed cases of the library, each through its public Python entry points.

A case is a dict of plain values. ``prepare`` makes its inputs on the GPU from a
seed, ``run`` makes one pass, ``work`` counts the bytes and operations that a pass
cannot do without, and ``exact`` gives the outputs in 64 bits from torch and numpy
alone. The sizes are those of the benchmark and of the tests: RBF kernel matrices on
uniform points in the unit cube (length scale 0.1, lam = 1e-2, sketch size n / 16,
8 nonzeros per row), the 32-outlier spectrum at n = 1024 (lam = 1e-3, s = 64), and
tall matrices G diag(d) / sqrt(m) with 32 outlying singular values.

Solves stop at a relative residual of 1e-10, the library's default rule.
"""

import math

import numpy as np
import torch

from paper_2405_05865_gb300 import Context
from paper_2405_05865_gb300.autograd import rbf_solve

SEED = 0x4D5350          # the library's default seed of its sketches and probes
LAM = 1e-2               # the kernel systems' regularisation

_CTX = None


def _context():
    """One context for the process, as a program that solves many systems keeps."""
    global _CTX
    if _CTX is None:
        _CTX = Context()
    return _CTX


def listed():
    return [
        # the residual product y = (A + lam I) x of a small system: the smallest
        # call, bound by its launches
        dict(name="matvec_1000", kind="matvec", n=1000, dtype="float32"),
        # forming the kernel matrix of the benchmark's GP-regression system
        dict(name="kernel_16384", kind="kernel", n=16384, dim=3, ell=0.1),
        # the sketch C = A Pi of that system (with the packed copy its solves read)
        dict(name="sketch_16384", kind="sketch", n=16384, s=1024, gamma=8, dtype="float32"),
        # the Nystrom core and its factor (lambda0 of the order of (2 / l) times the tail of
        # the spectrum, as Algorithm 1 takes it), and one application of the preconditioner
        dict(name="factor_16384", kind="factor", n=16384, s=1024, lam0=16.4, ell=0.1),
        # a right-hand side solved with a kept factor, mixed precision
        dict(name="solve_16384", kind="solve", n=16384, s=1024, ell=0.1),
        # the whole call on a small ill-conditioned FP64 system, with the sketched
        # level 2 (phi = 4 s) and its inner iteration
        dict(name="full_fp64_1024", kind="full64", n=1024, s=64),
        # the whole call, mixed precision, on a size that no tile divides, with the
        # sketched level 2
        dict(name="full_4999", kind="full", n=4999, s=312, phi=1248, ell=0.1),
        # a training step of the kernel's hyperparameters: kernel, factor, solve,
        # and the gradients of b^T x from the adjoint solve
        dict(name="gradient_8192", kind="gradient", n=8192, s=512, ell=0.1),
        # a batch of kernel systems of uneven size, 16 right-hand sides each, set-up
        # and solve
        dict(name="batch_24", kind="batch", count=24, n_lo=512, n_hi=4096, m=16, sizes=0),
        # Hutchinson's estimate of the Schatten-1 norm, per probe
        dict(name="trace_16384", kind="trace", n=16384, probes=256, ell=0.1),
        # (A^T A + lam I) x = c of the benchmark's tall matrix, the inner levels exact
        dict(name="general_65536", kind="general", m=65536, n=4096, s=256, levels=0),
        # the same method with its three sketched levels
        dict(name="levels_16384", kind="general", m=16384, n=2048, s=128, levels=8),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["matvec", "kernel", "sketch", "factor", "solve", "full64", "full", "gradient", "batch",
                       "trace", "general", "levels"])
    if kind == "matvec":
        return dict(kind=kind, n=_log_int(rng, 300, 16384), dtype=rng.choice(["float32", "float64", "bfloat16"]))
    if kind == "kernel":
        return dict(kind=kind, n=_log_int(rng, 700, 16384), dim=rng.randint(1, 4), ell=round(rng.uniform(0.05, 0.2), 4))
    if kind == "sketch":
        n = _log_int(rng, 700, 16384)
        return dict(kind=kind, n=n, s=rng.randint(max(64, n // 24), min(1024, n // 8 + 64)), gamma=rng.choice([4, 8]),
                    dtype=rng.choice(["float32", "float32", "float64", "bfloat16"]))
    if kind in ("factor", "solve"):
        n = _log_int(rng, 700, 16384)
        c = dict(kind=kind, n=n, s=max(32, n // 16 + rng.randint(-8, 0)), ell=round(rng.uniform(0.08, 0.12), 4))
        return dict(c, lam0=round(1e-3 * n, 2)) if kind == "factor" else c
    if kind == "full64":
        n = _log_int(rng, 500, 1500)
        return dict(kind=kind, n=n, s=n // 16)
    if kind == "full":
        n = _log_int(rng, 700, 6000)
        s = max(48, n // 16)
        return dict(kind=kind, n=n, s=s, phi=rng.choice([0, 4 * s]), ell=round(rng.uniform(0.08, 0.12), 4))
    if kind == "gradient":
        n = _log_int(rng, 700, 8192)
        return dict(kind=kind, n=n, s=max(48, n // 16), ell=round(rng.uniform(0.08, 0.12), 4))
    if kind == "batch":
        hi = rng.randint(1024, 4096)
        return dict(kind=kind, count=rng.randint(3, 24), n_lo=rng.randint(300, 800), n_hi=hi,
                    m=rng.choice([1, 4, 7, 16]), sizes=rng.randint(1, 10 ** 6))
    if kind == "trace":
        return dict(kind=kind, n=_log_int(rng, 700, 16384), probes=64 * rng.randint(1, 4),
                    ell=round(rng.uniform(0.05, 0.2), 4))
    if kind == "general":
        n = _log_int(rng, 500, 4096)
        return dict(kind="general", m=_log_int(rng, 8 * n, 65536), n=n, s=rng.choice([128, 192, 256]), levels=0)
    n = rng.randint(1536, 2048)
    return dict(kind="general", m=8 * n, n=n, s=128, levels=8)


# ------------------------------------------------------------------ inputs


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _randn(n, seed):
    return torch.randn(n, generator=_gen(seed), device="cuda", dtype=torch.float64)


def _points(n, dim, seed):
    return torch.rand((n, dim), generator=_gen(seed), device="cuda", dtype=torch.float64)


def _rbf(points, ell):
    """exp(-|p_i - p_j|^2 / (2 ell^2)) in FP64, exactly symmetric."""
    n, dim = points.shape
    K = torch.empty((n, n), device="cuda", dtype=torch.float64)
    for i in range(0, n, 4096):
        P = points[i:i + 4096]
        d2 = torch.zeros((P.shape[0], n), device="cuda", dtype=torch.float64)
        for d in range(dim):
            d2 += (P[:, d, None] - points[None, :, d]) ** 2
        K[i:i + 4096] = torch.exp_(d2 * (-0.5 / (ell * ell)))
    return K


def _rbf_stored(case, seed, dtype=torch.float32):
    """The kernel matrix of a case, rounded once to its storage type: the problem's A."""
    return _rbf(_points(case["n"], 3, seed), case.get("ell", 0.1)).to(dtype)


def _outliers(n, k, hi, lo):
    return torch.logspace(math.log10(hi), math.log10(lo), k, device="cuda", dtype=torch.float64)


def _outlier_system(n, seed):
    """A = Q diag(sigma) Q^T (FP64): outliers 1e4 -> 1e2, then i^-1.5, and lambda0 of the n / 32 largest."""
    k = n // 32
    i = torch.arange(k + 1, n + 1, device="cuda", dtype=torch.float64)
    sigma = torch.cat([_outliers(n, k, 1e4, 1e2), i ** -1.5])
    Q, _ = torch.linalg.qr(torch.randn((n, n), generator=_gen(seed), device="cuda", dtype=torch.float64))
    A = (Q * sigma) @ Q.T
    return 0.5 * (A + A.T), 2.0 / k * float(sigma[k:].sum())


def _tall(case, seed):
    """A = G diag(d) / sqrt(m) (FP32), d 32 outliers 1e2 -> 1e1 then U(0.5, 1), and lambda0 of the 64 largest."""
    m, n = case["m"], case["n"]
    g = _gen(seed)
    tail = 0.5 + 0.5 * torch.rand(n - 32, generator=g, device="cuda", dtype=torch.float64)
    d = torch.cat([_outliers(n, 32, 1e2, 1e1), tail])
    A = torch.randn((m, n), generator=g, device="cuda", dtype=torch.float32)
    A *= (d / math.sqrt(m)).float()
    return A, 2.0 / 64 * float((d[64:] ** 2).sum())


def _batch_sizes(case):
    """(n, ell, s) of every instance: n ~ U{n_lo..n_hi}, ell ~ U(0.05, 0.1), s = n / 4 in whole 64s up to 1024."""
    g = np.random.default_rng([case["sizes"], 3])
    out = []
    for _ in range(case["count"]):
        n = int(g.integers(case["n_lo"], case["n_hi"] + 1))
        out.append((n, float(g.uniform(0.05, 0.1)), min(1024, max(64, n // 4 // 64 * 64))))
    return out


def prepare(case, seed):
    kind, ctx = case["kind"], _context()
    st = dict(case=case, ctx=ctx)
    if kind == "kernel":
        st.update(points=_points(case["n"], case["dim"], seed))
    elif kind == "matvec":
        st.update(A=_rbf_stored(case, seed, getattr(torch, case["dtype"])), x=_randn(case["n"], seed + 1))
    elif kind == "sketch":
        st.update(A=_rbf_stored(case, seed, getattr(torch, case["dtype"])))
    elif kind in ("factor", "solve"):
        A = _rbf_stored(case, seed)
        st.update(A=A, b=_randn(case["n"], seed + 1), sketch=ctx.sketch(A, case["s"], 8))
        if kind == "factor":
            st.update(r=st["b"].float())
        else:
            st.update(factor=ctx.nystrom(st["sketch"], LAM, phi=0))
    elif kind == "full64":
        A, lam0 = _outlier_system(case["n"], seed)
        st.update(A=A, lam0=lam0, b=_randn(case["n"], seed + 1))
    elif kind == "full":
        st.update(A=_rbf_stored(case, seed), b=_randn(case["n"], seed + 1))
    elif kind == "gradient":
        st.update(points=_points(case["n"], 3, seed), b=_randn(case["n"], seed + 1).requires_grad_(True),
                  ell=torch.tensor(case["ell"], dtype=torch.float64, requires_grad=True),
                  lam=torch.tensor(LAM, dtype=torch.float64, requires_grad=True))
    elif kind == "batch":
        insts = []
        for k, (n, ell, s) in enumerate(_batch_sizes(case)):
            A = _rbf_stored(dict(n=n, ell=ell), 64 * seed + k)
            B = torch.randn((n, case["m"]), generator=_gen(64 * seed + k + 7), device="cuda", dtype=torch.float64)
            insts.append(dict(A=A, B=B, lam=LAM, s=s))
        st.update(instances=insts)
    elif kind == "trace":
        st.update(A=_rbf_stored(case, seed))
    elif kind == "general":
        A, lam0 = _tall(case, seed)
        st.update(A=A, lam0=lam0, c=_randn(case["n"], seed + 1),
                  general=ctx.general(A, 1e-3, case["s"], lam0=lam0, phi=4 * case["s"]))
    return st


# -------------------------------------------------------------------- runs


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    if kind == "matvec":
        return ctx.matvec_f64(state["A"], state["x"], LAM)
    if kind == "kernel":
        return ctx.rbf_kernel(state["points"], case["ell"])
    if kind == "sketch":
        sk = ctx.sketch(state["A"], case["s"], case["gamma"])
        C = sk.C()
        sk.close()
        return C
    if kind == "factor":
        f = ctx.nystrom(state["sketch"], LAM, case["lam0"], phi=0)
        w, _ = ctx.solve_m1(f, state["r"], max_inner=0)
        f.close()
        return w
    if kind == "solve":
        x, _ = ctx.solve(state["factor"], state["A"], state["b"], LAM, tol=1e-10, refine_tol=3e-3, max_inner=0)
        return x
    if kind == "full64":
        x, _ = ctx.solve_full(state["A"], state["b"], 1e-3, case["s"], 8, state["lam0"], precision="fp64", tol=1e-10,
                              inner_tol=1e-10)
        return x
    if kind == "full":
        x, _ = ctx.solve_full(state["A"], state["b"], LAM, case["s"], 8, phi=case["phi"], tol=1e-10, refine_tol=3e-3,
                              max_inner=50 if case["phi"] else 0)
        return x
    if kind == "gradient":
        x = rbf_solve(state["points"], state["ell"], state["lam"], state["b"], ctx, case["s"], tol=1e-10,
                      refine_tol=3e-3)
        grads = torch.autograd.grad(state["b"] @ x, (state["ell"], state["lam"], state["b"]))
        return dict(x=x.detach(), ell=grads[0], lam=grads[1], b=grads[2])
    if kind == "batch":
        bt = ctx.batch(state["instances"])
        bt.solve(tol=1e-10, refine_tol=1e-4)
        xs = [bt.X(k) for k in range(bt.count)]
        bt.close()
        return xs
    if kind == "trace":
        return ctx.hutchinson(state["A"], case["probes"])
    if kind == "general":
        levels = case["levels"]
        x, _ = state["general"].solve(state["c"], tol=1e-10, refine_tol=1e-3 if levels else 1e-4, level2_iters=levels,
                                      level3_iters=levels, max_outer=400)
        return x
    raise ValueError(kind)


def work(case):
    """Bytes: inputs read once, outputs written once. Operations: one product with the
    matrix for an iterative solve, whose number of them depends on the spectrum."""
    kind, n = case["kind"], case.get("n", 0)
    if kind == "matvec":
        size = {"float32": 4, "float64": 8, "bfloat16": 2}[case["dtype"]]
        return dict(bytes=n * n * size + 16 * n, flops=2 * n * n)
    if kind == "kernel":
        return dict(bytes=4 * n * n + 8 * n * case["dim"], flops=n * n * (3 * case["dim"] + 2) / 2)
    if kind == "sketch":
        size = {"float32": 4, "float64": 8, "bfloat16": 2}[case["dtype"]]
        return dict(bytes=n * n * size + n * case["s"] * (8 if size == 8 else 4), flops=n * n * case["gamma"])
    if kind == "factor":
        s = case["s"]
        return dict(bytes=4 * n * s + 8 * n, flops=n * s * s + s * s * s + 4 * n * s)
    if kind in ("solve", "full", "full64"):
        size = 8 if kind == "full64" else 4
        return dict(bytes=size * n * (n + 1) // 2 + 16 * n, flops=2 * n * n)
    if kind == "gradient":
        return dict(bytes=2 * n * (n + 1) + 64 * n, flops=4 * n * n)
    if kind == "batch":
        mean = (case["n_lo"] + case["n_hi"]) / 2
        square = mean * mean + (case["n_hi"] - case["n_lo"]) ** 2 / 12
        return dict(bytes=case["count"] * (2 * square + 16 * mean * case["m"]),
                    flops=2 * case["count"] * square * case["m"])
    if kind == "trace":
        return dict(bytes=2 * n * (n + 1) + 8 * case["probes"], flops=n * n * case["probes"])
    if kind == "general":
        return dict(bytes=4 * case["m"] * n + 16 * n, flops=4 * case["m"] * n)
    raise ValueError(kind)


# -------------------------------------------------- the same in 64 bits


def _draws(stream, rows, q):
    """Output k = (stream << 56) | (row << 8) | q of SplitMix64 seeded with SEED (Steele, Lea and Flood 2014)."""
    with np.errstate(over="ignore"):
        k = (np.uint64(stream) << np.uint64(56)) | (np.asarray(rows, np.uint64) << np.uint64(8)) | np.uint64(q)
        z = np.uint64(SEED) + (k + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def _sketch_matrix(n, s, gamma):
    """Pi = S^T (n x s): gamma entries +-1 / sqrt(gamma) per row by Floyd's sampling (Bentley and Floyd 1987)."""
    rows = np.arange(n)
    picked = np.zeros((n, gamma), np.int64)
    for q, t in enumerate(range(s - gamma, s)):
        u = _draws(0, rows, q)
        m, low = np.uint64(t + 1), np.uint64(0xFFFFFFFF)
        r = ((u >> np.uint64(32)) * m + (((u & low) * m) >> np.uint64(32))) >> np.uint64(32)
        r = r.astype(np.int64)
        seen = (picked[:, :q] == r[:, None]).any(axis=1)
        picked[:, q] = np.where(seen, t, r)
    picked.sort(axis=1)
    Pi = torch.zeros((n, s), device="cuda", dtype=torch.float64)
    at = torch.arange(n, device="cuda")
    for q in range(gamma):
        sign = np.where(_draws(1, rows, q) >> np.uint64(63), -1.0, 1.0) / math.sqrt(gamma)
        Pi[at, torch.from_numpy(picked[:, q]).cuda()] = torch.from_numpy(sign).cuda()
    return Pi


def _dense_solve(A, lam, B):
    """(A + lam I)^{-1} B by Cholesky, A overwritten."""
    A.diagonal().add_(lam)
    return torch.cholesky_solve(B, torch.linalg.cholesky(A))


def exact(case, seed):
    kind, n = case["kind"], case.get("n", 0)
    if kind == "matvec":
        A = _rbf_stored(case, seed, getattr(torch, case["dtype"])).double()
        x = _randn(n, seed + 1)
        return A @ x + LAM * x
    if kind == "kernel":
        return _rbf(_points(n, case["dim"], seed), case["ell"])
    if kind == "sketch":
        A = _rbf_stored(case, seed, getattr(torch, case["dtype"])).double()
        return A @ _sketch_matrix(n, case["s"], case["gamma"])
    if kind == "factor":
        # w = (r - C (C^T C + t W + nu I)^{-1} C^T r) / t, t = lam + lambda0, nu = 2^-24 |C^T C + t W|_F
        t = LAM + case["lam0"]
        Pi = _sketch_matrix(n, case["s"], 8)
        C = _rbf_stored(case, seed).double() @ Pi
        W = Pi.T @ C
        M = C.T @ C + 0.5 * t * (W + W.T)
        r = _randn(n, seed + 1).float().double()
        y = _dense_solve(M, 2.0 ** -24 * float(M.norm()), (C.T @ r)[:, None])
        return (r - (C @ y)[:, 0]) / t
    if kind in ("solve", "full"):
        return _dense_solve(_rbf_stored(case, seed).double(), LAM, _randn(n, seed + 1)[:, None])[:, 0]
    if kind == "full64":
        # two steps of refinement with residuals in numpy's long double
        A, _ = _outlier_system(n, seed)
        b = _randn(n, seed + 1)
        L = torch.linalg.cholesky(A + 1e-3 * torch.eye(n, device="cuda", dtype=torch.float64))
        wide, bw = A.cpu().numpy().astype(np.longdouble), b.cpu().numpy().astype(np.longdouble)
        x = np.zeros(n, np.longdouble)
        for _ in range(3):
            r = bw - (wide * x).sum(axis=1) - np.longdouble(1e-3) * x
            r = torch.from_numpy(r.astype(np.float64)).cuda()
            x = x + torch.cholesky_solve(r[:, None], L)[:, 0].cpu().numpy()
        return torch.from_numpy(x.astype(np.float64))
    if kind == "gradient":
        P, b, ell = _points(n, 3, seed), _randn(n, seed + 1), case["ell"]
        x = _dense_solve(_rbf(P, ell), LAM, b[:, None])[:, 0]
        # dK_ij / d ell = K_ij d_ij^2 / ell^3, and d_ij^2 = -2 ell^2 log K_ij
        grad_ell = 0.0
        for i in range(0, n, 2048):
            d2 = sum((P[i:i + 2048, d, None] - P[None, :, d]) ** 2 for d in range(P.shape[1]))
            grad_ell -= float(x[i:i + 2048] @ ((torch.exp(d2 * (-0.5 / ell ** 2)) * d2) @ x)) / ell ** 3
        return dict(x=x, ell=torch.tensor(grad_ell, dtype=torch.float64), lam=-(x @ x), b=2.0 * x)
    if kind == "batch":
        out = []
        for k, (n, ell, s) in enumerate(_batch_sizes(case)):
            A = _rbf_stored(dict(n=n, ell=ell), 64 * seed + k).double()
            B = torch.randn((n, case["m"]), generator=_gen(64 * seed + k + 7), device="cuda", dtype=torch.float64)
            out.append(_dense_solve(A, LAM, B))
        return out
    if kind == "trace":
        A = _rbf_stored(case, seed).double()
        G = np.empty((n, case["probes"]))
        for j in range(case["probes"]):
            G[:, j] = np.where(_draws(7 + 2 * (j // 256), np.arange(n), j % 256) >> np.uint64(63), -1.0, 1.0)
        G = torch.from_numpy(G).cuda()
        return (G * (A @ G)).sum(0)
    if kind == "general":
        A, _ = _tall(case, seed)
        M = torch.zeros((n, n), device="cuda", dtype=torch.float64)
        for i in range(0, case["m"], 16384):
            a = A[i:i + 16384].double()
            M += a.T @ a
        return _dense_solve(M, 1e-3, _randn(n, seed + 1)[:, None])[:, 0]
    raise ValueError(kind)
