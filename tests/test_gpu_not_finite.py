"""Views that are not finite get some codeword of the vocabulary, so that nothing is indexed past it, and leave the
other queries' results as they are."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("n,K,ma", [(40, 33, 3), (200, 300, 1), (1500, 1100, 2), (20000, 300, 2)])
def test_codes_stay_in_the_vocabulary(gpu_lib, value, n, K, ma):
    import torch
    g = torch.Generator(device="cuda").manual_seed(n)
    cb = torch.randn((K, 64), generator=g, device="cuda")
    x = torch.randn((n, 64), generator=g, device="cuda")
    ix = gpu_lib.Index(x[:1].contiguous(), cb, 1, 1, K, keep_exact=False)
    clean = ix.assign(x, ma)
    bad = torch.arange(0, n, 17, device="cuda")
    y = x.clone()
    y[bad, 5] = value
    got = ix.assign(y, ma)
    assert int(got.min()) >= 0 and int(got.max()) < K
    same = torch.ones(n, dtype=torch.bool, device="cuda")
    same[bad] = False
    assert torch.equal(got[same], clean[same])


@pytest.mark.parametrize("storage,rescore", [("f32", 0), ("bf16", 30), ("fp8", 30)])
def test_other_queries_are_not_affected(gpu_lib, storage, rescore):
    import torch
    g = torch.Generator(device="cuda").manual_seed(3)
    N, nv, D, K = 150, 16, 128, 12
    db = torch.rand((N * nv, D), generator=g, device="cuda")
    ix = gpu_lib.Index(db, db[:K].contiguous(), N, nv, K, storage=storage, rescore_r=rescore, query_ma=2, keep_exact=False)
    q = torch.rand((3 * nv, D), generator=g, device="cuda")
    off = np.arange(4) * nv
    ids, sc = ix.query(q, off, topk=20)
    y = q.clone()
    y[nv:nv + 3, 7] = float("nan")
    y[nv + 5, 2] = float("inf")
    i2, s2 = ix.query(y, off, topk=20)
    for b in (0, 2):
        assert torch.equal(ids[b], i2[b]) and torch.equal(sc[b], s2[b])
    x = db.clone()
    x[5 * nv, 3] = float("nan")
    gpu_lib.Index(x, db[:K].contiguous(), N, nv, K, storage=storage, rescore_r=rescore, keep_exact=False).close()
