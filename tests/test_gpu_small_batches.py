"""Small batches: the quantiser's narrow tiles and block-per-row refine, and the FP32 scan at its tile edges, against
float64 numpy."""
import numpy as np
import pytest

from oracle import gift_oracle as O
from tests.parity import close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [1, 31, 33, 257, 1100])
@pytest.mark.parametrize("n,ma", [(1, 1), (127, 2), (129, 3), (1215, 1), (1217, 2)])
def test_codes_at_tile_edges(gpu_lib, K, n, ma):
    import torch
    g = np.random.default_rng(K * 131 + n)
    D, ma = 48, min(ma, K)
    cb = g.standard_normal((K, D)).astype(np.float32)
    x = (cb[g.integers(0, K, n)] + 0.7 * g.standard_normal((n, D))).astype(np.float32)
    ix = gpu_lib.Index(torch.from_numpy(x[:1].copy()).cuda(), torch.from_numpy(cb).cuda(), 1, 1, K, keep_exact=False)
    got = ix.assign(torch.from_numpy(x).cuda(), ma).cpu().numpy()
    dist = ((x[:, None].astype(np.float64) - cb[None]) ** 2).sum(2)
    assert np.array_equal(got, np.argsort(dist, axis=1, kind="stable")[:, :ma])


# few rows: the reduction in one to eight parts (D = 256 is one, 512 two, 4096 eight; 1025 codewords keep one)
@pytest.mark.parametrize("K", [1, 31, 32, 33, 512, 1000, 1024, 1025])
@pytest.mark.parametrize("n,ma,D", [(1, 1, 256), (3, 2, 512), (54, 2, 4096), (127, 3, 1024), (128, 1, 1104),
                                    (129, 2, 2048), (1215, 2, 528)])
def test_codes_from_parts_of_the_reduction(gpu_lib, K, n, ma, D):
    import torch
    g = np.random.default_rng(K * 17 + n)
    ma = min(ma, K)
    cb = g.standard_normal((K, D)).astype(np.float32)
    x = (cb[g.integers(0, K, n)] + 0.7 * g.standard_normal((n, D))).astype(np.float32)
    ix = gpu_lib.Index(torch.from_numpy(x[:1].copy()).cuda(), torch.from_numpy(cb).cuda(), 1, 1, K, keep_exact=False)
    got = ix.assign(torch.from_numpy(x).cuda(), ma).cpu().numpy()
    cb64, x64 = cb.astype(np.float64), x.astype(np.float64)
    dist = (cb64 ** 2).sum(1)[None] - 2 * x64 @ cb64.T  # less |x|^2; gaps are of order D, the rounding 1e-12
    assert np.array_equal(got, np.argsort(dist, axis=1, kind="stable")[:, :ma])


# one list (K = 1) makes every (slot, entry) tile of the FP32 scan: entries and slots at and around 64
@pytest.mark.parametrize("D", [16, 32, 48, 80])
@pytest.mark.parametrize("N,nv,vq", [(1, 1, 1), (9, 7, 64), (13, 5, 65), (16, 8, 3)])
def test_f32_scan_tiles(gpu_lib, D, N, nv, vq):
    import torch
    g = np.random.default_rng(D + N)
    db = g.random((N, nv, D)).astype(np.float32)
    q = g.random((vq, D)).astype(np.float32)
    cb = db[0, :1].copy()
    ix = gpu_lib.Index(torch.from_numpy(db).cuda(), torch.from_numpy(cb).cuda(), N, nv, 1, keep_exact=False)
    ids, sc = ix.query(torch.from_numpy(q).cuda(), np.array([0, vq], np.int32), topk=N)
    S = np.array([O.cosine(q, db[p]).max(1).mean() for p in range(N)])  # one codeword: Eq. 4 is Eq. 3
    ids, sc = ids.cpu().numpy()[0], sc.cpu().numpy()[0]
    assert sorted(ids) == list(range(N))
    assert close(sc, S[ids]).all() and (np.diff(sc) <= 0).all()
