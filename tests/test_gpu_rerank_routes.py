"""The re-rank's routes (a table per query, a hash table, rows of every shape after an overflow, dense rows for long
walks of few queries) against an integer reference, for one measure and for two."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _members(s):
    return np.rint(np.clip(s, 0, 1).astype(np.float64) * 2.0 ** 31).astype(np.uint64)


def _index(gpu_lib, n):
    import torch
    x = torch.rand((n, 16), device="cuda")
    return gpu_lib.Index(x, x[:2].contiguous(), n, 1, 2, keep_exact=False)


def _neighbours(g, N, k1, kind):
    """Rows of k1 distinct neighbours: of the shape's group of 200, of all shapes, half of them of N / 100 hubs, or of
    the group but for ten hubs, which every row names but those by which a walk's cost is estimated."""
    out = np.empty((N, k1), np.int32)
    for p in range(N):
        if kind == "all":
            out[p] = g.choice(N, k1, replace=False)
        elif kind == "hubs":
            h = g.choice(N // 100, k1 // 2, replace=False)
            out[p] = np.concatenate([h, N // 100 + g.choice(N - N // 100, k1 - len(h), replace=False)])
        else:
            base = p // 200 * 200
            out[p] = base + g.choice(min(200, N - base), k1, replace=False)
    if kind == "unseen":
        rows = np.setdiff1d(np.arange(N), np.arange(64) * N // 64)
        hub = np.arange(10) * 200 + 7
        out[rows, :10] = hub
        for p in rows:  # (a hub that the group's own draw named too)
            own = np.isin(out[p, 10:], hub)
            out[p, 10:][own] = np.setdiff1d(p // 200 * 200 + np.arange(200), out[p])[:own.sum()]
    sc = np.sort(g.integers(1, 9, (N, k1)) / 8.0, 1)[:, ::-1].astype(np.float32).copy()
    return out, sc


def _check(num, norm, card, cand, csc, topk, got_i, got_s):
    N = len(card)
    tie = np.full(N, -np.inf, np.float32)
    tie[cand] = csc
    den = norm + card - num
    sp = np.where(num > 0, num.astype(np.float32) / np.maximum(den, 1).astype(np.float32), np.float32(0))
    order = np.lexsort((np.arange(N), -tie, -sp))[:topk]
    assert np.array_equal(got_i, order) and np.array_equal(got_s, sp[order])


def _launches(gpu_lib, call):
    import torch
    call()
    n = gpu_lib.launch_count()
    out = call()
    n = gpu_lib.launch_count() - n
    torch.cuda.synchronize()
    return n, out


# long: the walks are spread over the SMs (several kernels), otherwise one kernel with a block per query
@pytest.mark.parametrize("N,k1,kind,B,long", [
    (20000, 50, "group", 3, False), (20000, 40, "hubs", 3, True), (20000, 40, "hubs", 160, False),
    (20000, 30, "unseen", 3, False), (3000, 400, "all", 1, True), (3000, 400, "all", 400, False),
    (13000, 400, "all", 2, True)])
def test_one_measure(gpu_lib, N, k1, kind, B, long):
    import torch
    g = np.random.default_rng(N + k1 + B)
    nbr, nsc = _neighbours(g, N, k1, kind)
    ix = _index(gpu_lib, 8)
    ix.set_sif(torch.from_numpy(nbr).cuda(), torch.from_numpy(nsc).cuda(), N, k1)
    rows = g.integers(0, N // 50, B) * 50 + 1
    cand = np.stack([np.concatenate([nbr[p], np.setdiff1d(np.arange(k1 + 5), nbr[p])[:5]]) for p in rows])
    csc = np.sort(g.integers(1, 200, cand.shape) / 200.0, 1)[:, ::-1].astype(np.float32).copy()
    ci, cs = torch.from_numpy(cand.astype(np.int32)).cuda(), torch.from_numpy(csc).cuda()
    n, (oi, os_) = _launches(gpu_lib, lambda: ix.rerank(ci, cs, k1=k1, topk=100))
    assert (n > 1) == long
    mem = _members(nsc)
    order = np.argsort(nbr.reshape(-1), kind="stable")
    off = np.searchsorted(nbr.reshape(-1)[order], np.arange(N + 1))
    for b in range(0, B, max(1, B // 4)):
        num, norm = np.zeros(N, np.uint64), np.uint64(0)
        for r in range(k1):
            f = _members(csc[b, r])
            norm += f
            e = order[off[cand[b, r]]:off[cand[b, r] + 1]]
            np.add.at(num, e // k1, np.minimum(f, mem.reshape(-1)[e]))
        _check(num, norm, mem.sum(1), cand[b], csc[b], 100, oi[b].cpu().numpy(), os_[b].cpu().numpy())
    ix.close()


@pytest.mark.parametrize("N,k1,k2,kind,B,long", [
    (16500, 20, 2, "group", 3, False), (16500, 20, 2, "all", 3, False), (16500, 20, 10, "all", 3, True),
    (16500, 20, 10, "all", 160, False), (2000, 20, 20, "all", 1, True)])
def test_two_measures(gpu_lib, N, k1, k2, kind, B, long):
    import torch
    g = np.random.default_rng(N + k1 + k2 + B)
    ixs, nb, cand = [], [], []
    for m in range(2):
        nbr, nsc = _neighbours(g, N, k1, kind)
        ix = _index(gpu_lib, N)
        ix.set_sif(torch.from_numpy(nbr).cuda(), torch.from_numpy(nsc).cuda(), N, k1)
        rows = g.integers(0, N, B)
        csc = np.sort(g.integers(1, 200, (B, k1)) / 200.0, 1)[:, ::-1].astype(np.float32).copy()
        ixs.append(ix)
        nb.append((nbr, nsc))
        cand.append((nbr[rows].copy(), csc))
    aca = gpu_lib.Aca(ixs[0], ixs[1], k2=k2, alpha=0.5, mode="co")
    dev = [tuple(torch.from_numpy(x).cuda() for x in c) for c in cand]
    n, (oi, os_) = _launches(gpu_lib, lambda: aca.rerank(dev[0], dev[1], topk=50))
    assert (n > 2) == long  # the activations' kernel, then the re-rank's
    off, ids, mem, card = aca.export()
    for b in range(0, B, max(1, B // 4)):
        f = []  # co-augmentation: the rows, under measure l, of the query's first k2 neighbours under the other
        for l in range(2):
            src = cand[1 - l][0][b, :k2]
            s = np.zeros(N, np.float32)
            np.add.at(s, nb[l][0][src].reshape(-1), nb[l][1][src].reshape(-1))
            f.append(s / np.float32(k2))
        r = np.float32(0.5) * (np.sqrt(f[0]) + np.sqrt(f[1]))
        fq = _members(r * r)
        num = np.zeros(N, np.uint64)
        for i in np.nonzero(fq)[0]:
            e = slice(off[i], off[i + 1])
            np.add.at(num, ids[e], np.minimum(fq[i], mem[e].astype(np.uint64)))
        _check(num, fq.sum(), card, cand[0][0][b], cand[0][1][b], 50, oi[b].cpu().numpy(), os_[b].cpu().numpy())
    aca.close()
    for ix in ixs:
        ix.close()
