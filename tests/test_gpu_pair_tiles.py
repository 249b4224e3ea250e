"""Contractions on pairs of SMs (256 x 256 tiles, large calls) against one-SM tiles (the same rows in small calls):
the same products in the same order, so the same bits, at ragged tile edges."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["float32", "bfloat16"])
@pytest.mark.parametrize("nv,Np,din,dout", [(64, 701, 96, 64), (20, 2003, 160, 144), (33, 1201, 64, 48),
                                            (64, 640, 1040, 1040)])
def test_forward_rows_do_not_depend_on_the_call(gpu_lib, dtype, nv, Np, din, dout):
    import torch
    g = torch.Generator(device="cuda").manual_seed(nv * Np)
    counts = np.resize([20, 33, 64], 30)
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    dt = getattr(torch, dtype)
    q = torch.randn((int(off[-1]), din), generator=g, device="cuda").to(dt)
    p = torch.randn((Np, nv, din), generator=g, device="cuda").to(dt)
    w = (torch.randn((dout, din), generator=g, device="cuda") / din ** 0.5).to(dt)
    S, am = gpu_lib.match_forward(q, off, p, w)
    for b in (0, 7, 28):  # two queries at a time: one row tile
        lo, hi = int(off[b]), int(off[b + 2])
        s1, a1 = gpu_lib.match_forward(q[lo:hi].contiguous(), off[b:b + 3] - off[b], p, w)
        assert torch.equal(S[b:b + 2], s1) and torch.equal(am[lo:hi], a1)


@pytest.mark.parametrize("storage,keep", [("bf16", True), ("fp8", False)])
def test_exact_scores_do_not_depend_on_the_batch(gpu_lib, storage, keep):
    import torch
    g = torch.Generator(device="cuda").manual_seed(5)
    N, nv, D = 1500, 21, 272
    db = torch.rand((N * nv, D), generator=g, device="cuda")
    ix = gpu_lib.Index(db, db[:40].contiguous(), N, nv, 40, storage=storage, rescore_r=50, keep_exact=keep)
    counts = np.resize([1, 64, 20], 24)
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    q = torch.rand((int(off[-1]), D), generator=g, device="cuda")
    ids, sc = ix.query(q, off, mode="exact", topk=40)
    for b in (0, 11, 23):
        lo, hi = int(off[b]), int(off[b + 1])
        i1, s1 = ix.query(q[lo:hi].contiguous(), off[b:b + 2] - off[b], mode="exact", topk=40)
        assert torch.equal(ids[b], i1[0]) and torch.equal(sc[b], s1[0])


@pytest.mark.parametrize("K,ma", [(300, 1), (640, 2), (1000, 3), (1100, 2), (2100, 1)])
def test_codes_do_not_depend_on_the_batch(gpu_lib, K, ma):
    import torch
    g = torch.Generator(device="cuda").manual_seed(K)
    n, D = 20011, 64
    cb = torch.randn((K, D), generator=g, device="cuda")
    x = (cb[torch.randint(0, K, (n,), generator=g, device="cuda")]
         + torch.randn((n, D), generator=g, device="cuda")).contiguous()
    ix = gpu_lib.Index(x[:1].contiguous(), cb, 1, 1, K, keep_exact=False)
    codes = ix.assign(x, ma)
    for lo in (0, 9999, n - 300):
        assert torch.equal(codes[lo:lo + 300], ix.assign(x[lo:lo + 300].contiguous(), ma))
