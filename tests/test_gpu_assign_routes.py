"""The quantiser where its tiles change with the rows and the vocabulary (items of 32, 64 or 256 codewords, pairs of SMs),
against float64."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,K,D,ma", [
    (1, 4096, 64, 2), (1, 4097, 64, 1), (20, 9001, 48, 4), (130, 5003, 256, 2),   # large vocabularies, few rows
    (400, 4096, 64, 1), (300, 4096, 64, 2), (3000, 1100, 64, 3), (3000, 1024, 80, 1),  # a third of the SMs' items
    (10000, 192, 64, 1), (10000, 193, 64, 2), (6700, 256, 512, 1),
    (513, 1000, 272, 2), (512, 1000, 272, 2), (700, 512, 64, 1)])                  # rounds of items of 32
def test_codes_where_tiles_change(gpu_lib, n, K, D, ma):
    import torch
    g = np.random.default_rng(K * 31 + n)
    cb = g.standard_normal((K, D)).astype(np.float32)
    x = (cb[g.integers(0, K, n)] + 0.7 * g.standard_normal((n, D))).astype(np.float32)
    ix = gpu_lib.Index(torch.from_numpy(x[:1].copy()).cuda(), torch.from_numpy(cb).cuda(), 1, 1, K, keep_exact=False)
    got = ix.assign(torch.from_numpy(x).cuda(), ma).cpu().numpy()
    cb64, x64 = cb.astype(np.float64), x.astype(np.float64)
    dist = (cb64 ** 2).sum(1)[None] - 2 * x64 @ cb64.T
    assert np.array_equal(got, np.argsort(dist, axis=1, kind="stable")[:, :ma])
