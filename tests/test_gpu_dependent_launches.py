"""Kernels that are launched while the one before them ends: chains on two streams at once, calls back to back, and a
captured call give what one call alone gives, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage,rescore", [("f32", 0), ("bf16", 40), ("fp8", 40)])
def test_queries_on_two_streams(gpu_lib, storage, rescore):
    import torch
    g = np.random.default_rng(41)
    N, nv, D, K = 300, 12, 256, 48
    db = g.random((N, nv, D), dtype=np.float32)
    cb = g.random((K, D), dtype=np.float32)
    ix = gpu_lib.Index(torch.from_numpy(db).cuda(), torch.from_numpy(cb).cuda(), N, nv, K, storage=storage, query_ma=2,
                       rescore_r=rescore)
    batches = []
    for counts in ((1,), (12, 7), (64, 20, 3, 30)):
        off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
        batches.append((torch.from_numpy(g.random((int(off[-1]), D), dtype=np.float32)).cuda(), off))
    alone = []
    for q, off in batches:
        alone.append(ix.query(q, off, topk=20))
        torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    got = []
    for rep in range(20):
        for s in streams:
            i = (rep + (s is streams[1])) % 3
            with torch.cuda.stream(s):
                got.append((i, ix.query(batches[i][0], batches[i][1], topk=20, stream=s)))
    torch.cuda.synchronize()
    for i, (ids, sc) in got:
        assert torch.equal(ids, alone[i][0]) and torch.equal(sc, alone[i][1])


@pytest.mark.parametrize("n", [1, 54, 300])
def test_captured_quantiser(gpu_lib, n):
    import torch
    g = np.random.default_rng(n)
    D, K = 512, 96
    cb = g.standard_normal((K, D)).astype(np.float32)
    ix = gpu_lib.Index(torch.from_numpy(cb[:1].copy()).cuda(), torch.from_numpy(cb).cuda(), 1, 1, K, keep_exact=False)
    x = torch.from_numpy(g.standard_normal((n, D)).astype(np.float32)).cuda()
    s = torch.cuda.Stream()
    ix.assign(x, 2, stream=s)
    s.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        out = ix.assign(x, 2, stream=s)
    for seed in range(3):
        x.copy_(torch.from_numpy(np.random.default_rng(seed).standard_normal((n, D)).astype(np.float32)))
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, ix.assign(x, 2))
