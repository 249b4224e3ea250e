"""A kernel's bounded wait that runs out is reported: by the next call on the index, by the serving loop, once; the
calls after that work as before."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def give_up(gpu_lib, tmp_path_factory):
    from paper_1604_01879_gb300 import build
    so = str(tmp_path_factory.mktemp("native") / "wait_probe.so")
    subprocess.run([build._nvcc(), *build.FLAGS, "-shared", "-o", so, os.path.join(HERE, "native", "wait_probe.cu")],
                   check=True, capture_output=True)
    fn = ctypes.CDLL(so).wait_probe
    fn.argtypes = [ctypes.c_void_p]

    def run(ix):
        assert fn(ix._h) == 0  # the wait gave up
    return run


def _index(gpu_lib):
    import torch
    g = torch.Generator(device="cuda").manual_seed(1)
    db = torch.rand((60 * 8, 64), generator=g, device="cuda")
    q = torch.rand((3 * 8, 64), generator=g, device="cuda")
    ix = gpu_lib.Index(db, db[:10].contiguous(), 60, 8, 10, storage="bf16", rescore_r=20, sif_k1=5, keep_exact=False)
    return ix, q, np.arange(4) * 8


@pytest.mark.parametrize("call", ["query", "host query", "rerank", "assign", "export"])
def test_next_call_on_the_index_reports(gpu_lib, give_up, call):
    import torch
    ix, q, off = _index(gpu_lib)
    other = _index(gpu_lib)[0]
    ids, sc = ix.query(q, off, topk=10)
    torch.cuda.synchronize()
    calls = {"query": lambda: ix.query(q, off, topk=10),
             "host query": lambda: ix.query(q.cpu().numpy(), off, topk=10,
                                            out=(np.empty((3, 10), np.int32), np.empty((3, 10), np.float32))),
             "rerank": lambda: ix.rerank(ids, sc, k1=5, topk=5), "assign": lambda: ix.assign(q), "export": ix.export_fif}
    give_up(ix)
    assert torch.equal(other.query(q, off, topk=10)[0], ids)  # another index is not affected
    with pytest.raises(gpu_lib.GiftError) as e:
        calls[call]()
    assert e.value.status == 4
    calls[call]()
    again = ix.query(q, off, topk=10)
    assert torch.equal(again[0], ids) and torch.equal(again[1], sc)


def test_serving_loop_fails_what_was_in_flight(gpu_lib, give_up):
    ix, q, _ = _index(gpu_lib)
    s = gpu_lib.Server(ix, slots=2, topk=10, rerank=False)
    v = q[:8].cpu().numpy()
    first = s.wait(s.submit(v))
    give_up(ix)
    with pytest.raises(gpu_lib.GiftError) as e:
        s.wait(s.submit(v))
    assert e.value.status == 4
    again = s.wait(s.submit(v))
    assert np.array_equal(again[0], first[0]) and np.array_equal(again[1], first[1])
    assert s.stats()["failed"] == 1
    s.close()
