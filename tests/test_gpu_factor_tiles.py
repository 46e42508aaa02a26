"""The float-float Cholesky inverse as block elimination on 32 x 32 tiles: one
tile row (s_pad = 128 is four), a step's tiles fewer and more than the launch's
blocks, padding. X = L^{-1} of M = M2 + nu I satisfies |X M X^T - I|_2 <=
s 2^-40 kappa(M) (unit roundoff about 2^-46 and a margin of 2^6), and X is zero
above its diagonal.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from workloads import make_workload

pytestmark = pytest.mark.gpu

SEED = 0x4D5350


@pytest.fixture(scope="module")
def system():
    from paper_2405_05865_gb300 import Context
    ctx = Context(0)
    w = make_workload("rbf", seed=7, n=4096)
    yield ctx, w, torch.as_tensor(np.ascontiguousarray(w.A)).float().cuda()
    ctx.close()


@pytest.mark.parametrize("s", [33, 128, 384, 1024, 1500])
def test_tiled_inverse(system, s):
    ctx, w, A = system
    sk = ctx.sketch(A, s, 8, SEED)
    f = ctx.nystrom(sk, w.lam, 4.0, phi=0, seed=SEED)
    p = f.parts()
    M2, X, shift = p["M2"].cpu().numpy(), p["Linv"].cpu().numpy(), p["shift"]
    f.close()
    sk.close()
    M = M2 + shift * np.eye(M2.shape[0])
    M[s:], M[:, s:] = 0.0, 0.0
    M[range(s, len(M)), range(s, len(M))] = 1.0
    assert not np.triu(X, 1).any()
    ev = np.linalg.eigvalsh(M[:s, :s])
    E = X[:s, :s] @ M[:s, :s] @ X[:s, :s].T - np.eye(s)
    assert np.linalg.norm(E, 2) <= s * 2.0 ** -40 * ev.max() / ev.min()
