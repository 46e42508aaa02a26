"""The RBF kernel matrix at the edges of its 64 x 64 tiles: sizes below, at and past
a tile, rows that start on 16-byte boundaries (n a multiple of 4) and rows that do
not, every number of coordinates. Each entry against the oracle's FP64 value within
the FP32 bound of tests/test_gpu_adjoint.py (d^2 to 1e-7 relative, expf), and the
matrix equal to its transpose bit for bit."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import adjoint
from workloads import rbf_points

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2405_05865_gb300 import Context
    c = Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("dim", [1, 2, 3, 4])
@pytest.mark.parametrize("n", [1, 3, 63, 64, 65, 66, 127, 128, 132, 191, 260])
def test_rbf_kernel_tile_edges(ctx, n, dim):
    ell = 0.3
    P = rbf_points(n, seed=n + dim, dim=dim)
    K = ctx.rbf_kernel(torch.from_numpy(P).cuda(), ell).cpu().numpy()
    D2 = adjoint.rbf_sqdist(P)
    Kh = adjoint.rbf(P, ell)
    assert np.all(np.abs(K.astype(np.float64) - Kh) <= 4e-7 * (1.0 + D2 / (2 * ell * ell)) * Kh + 1e-30)
    assert np.array_equal(K, K.T)
    assert np.all(np.diag(K) == 1.0)
