"""Centre means at column tails and uneven centre sizes, against 64-bit numpy."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,D,K", [(17, 16, 17), (700, 528, 3), (2000, 1040, 40)])
def test_kmeans_means_of_uneven_centres(gpu_lib, n, D, K):
    """Column tails and centres of 1 to several hundred rows; one iteration from known centres."""
    import torch
    g = np.random.default_rng(n)
    X = g.standard_normal((n, D)).astype(np.float32)
    X[: n // 2] *= 0.05  # half of the rows sit near the origin, so centres are uneven
    init = np.sort(g.choice(n, K, replace=False)).astype(np.int32)
    C = gpu_lib.kmeans(torch.from_numpy(X).cuda(), init, 1).cpu().numpy()
    d = ((X[:, None].astype(np.float64) - X[init][None]) ** 2).sum(2) if n * K * D < 4e7 else \
        np.stack([((X.astype(np.float64) - X[c]) ** 2).sum(1) for c in init], 1)
    near = d.argmin(1)
    ref = np.stack([X[near == c].astype(np.float64).mean(0) for c in range(K)])
    assert np.abs(C - ref.astype(np.float32)).max() <= np.abs(ref).max() * 2.0 ** -23
