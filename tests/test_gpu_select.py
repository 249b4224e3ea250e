"""Block-wide selection and the one-block re-rank at the sizes where their paths change, against numpy."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _best(ids, scores, k):
    """The k best pairs of one row by (score desc, id asc); empty entries have id < 0."""
    keep = ids >= 0
    i, s = ids[keep], scores[keep]
    order = np.lexsort((i, -s))[:k]
    oi, os_ = np.full(k, -1, np.int32), np.full(k, -np.inf, np.float32)
    oi[:len(order)], os_[:len(order)] = i[order], s[order]
    return oi, os_


@pytest.mark.parametrize("k", [1, 100, 1024])
@pytest.mark.parametrize("n", [1, 33, 2047, 2049, 9000, 70001])
@pytest.mark.parametrize("values", ["distinct", "ties", "equal", "two", "signed"])
def test_merge_selects_like_a_sort(gpu_lib, n, k, values):
    import torch
    g = np.random.default_rng(n * 7 + k)
    B = 3
    ids = np.stack([g.permutation(2 * n)[:n] for _ in range(B)]).astype(np.int32)
    sc = {"distinct": lambda: g.random((B, n)), "ties": lambda: g.integers(0, 40, (B, n)) / 40.0,
          "equal": lambda: np.full((B, n), 0.25), "two": lambda: (g.random((B, n)) < 0.01) * 0.5,
          "signed": lambda: g.standard_normal((B, n)) * 10.0 ** g.integers(-20, 20, (B, n))}[values]().astype(np.float32)
    ids[1, g.random(n) < 0.3] = -1
    if values == "signed":
        sc[2, 0], sc[2, n // 2], sc[2, n - 1] = -np.inf, np.inf, 0.0
    oi, os_ = gpu_lib.merge_topk(torch.from_numpy(ids).cuda(), torch.from_numpy(sc).cuda(), k)
    for b in range(B):
        ri, rs = _best(ids[b], sc[b], k)
        assert np.array_equal(oi[b].cpu().numpy(), ri) and np.array_equal(os_[b].cpu().numpy(), rs)


def _members(s):
    return np.rint(np.clip(s, 0, 1).astype(np.float64) * 2.0 ** 31).astype(np.uint64)


# shapes, shapes per group that neighbours are drawn from, k1: whole table (256, 512 threads), its last size and
# the first of the hash table, hash, hash that overflows into two ranges of shapes
@pytest.mark.parametrize("N,group,k1", [(40, 40, 5), (1025, 200, 10), (5952, 300, 20), (5953, 300, 20), (40000, 400, 50),
                                        (30000, 30000, 125)])
@pytest.mark.parametrize("topk", [10, 1024])
def test_rerank_equals_integer_reference(gpu_lib, N, group, k1, topk):
    import torch
    g = np.random.default_rng(N + k1)
    x = torch.rand((8, 16), device="cuda")
    ix = gpu_lib.Index(x, x[:2].contiguous(), 8, 1, 2, keep_exact=False)
    base = np.arange(N) // group * group
    width = np.minimum(group, N - base)
    nbr = (base[:, None] + (np.arange(N)[:, None] + np.cumsum(g.integers(1, max(2, group // k1), (N, k1)), 1)) %
           width[:, None]).astype(np.int32) if group < N else g.integers(0, N, (N, k1)).astype(np.int32)
    nsc = np.sort(g.integers(-2, 9, (N, k1)) / 8.0, 1)[:, ::-1].astype(np.float32).copy()
    ix.set_sif(torch.from_numpy(nbr).cuda(), torch.from_numpy(nsc).cuda(), N, k1)
    B, n_cand = 5, k1 + 7
    cand = np.stack([g.permutation(min(N, group))[:min(n_cand, group)] for _ in range(B)]).astype(np.int32)
    n_cand = cand.shape[1]
    csc = np.sort(g.integers(1, 200, (B, n_cand)) / 200.0, 1)[:, ::-1].astype(np.float32).copy()
    cand[3, -2:] = -1
    csc[3, -2:] = -np.inf
    oi, os_ = ix.rerank(torch.from_numpy(cand).cuda(), torch.from_numpy(csc).cuda(), k1=k1, topk=topk)
    mem = _members(nsc)
    card = mem.sum(1)
    for b in range(B):
        num = np.zeros(N, np.uint64)
        norm = np.uint64(0)
        for r in range(k1):
            i = cand[b, r]
            if i < 0:
                continue
            f = _members(csc[b, r])
            norm += f
            p, c = np.nonzero(nbr == i)
            np.add.at(num, p, np.minimum(f, mem[p, c]))
        tie = np.full(N, -np.inf, np.float32)
        tie[cand[b][cand[b] >= 0]] = csc[b][cand[b] >= 0]
        den = norm + card - num
        sp = np.where(num > 0, num.astype(np.float32) / np.maximum(den, 1).astype(np.float32), np.float32(0))
        order = np.lexsort((np.arange(N), -tie, -sp))[:topk]
        got_i, got_s = oi[b].cpu().numpy(), os_[b].cpu().numpy()
        assert np.array_equal(got_i[:len(order)], order) and np.array_equal(got_s[:len(order)], sp[order])
        assert (got_i[len(order):] == -1).all() and np.isneginf(got_s[len(order):]).all()
