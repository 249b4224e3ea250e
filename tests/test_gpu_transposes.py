"""Gradients whose transposed operands end within, at and just past the transposes' tiles (64 and 128 rows, 64
columns), from inputs in 16-byte rows and from inputs that start off them, against the float64 oracle."""
import numpy as np
import pytest

from oracle import gift_oracle as O
from tests.test_gpu_match import _tie_free

pytestmark = pytest.mark.gpu


def _placed(a, dtype, off):
    """a on the device, `off` elements past an allocation's start."""
    import torch
    buf = torch.empty(a.size + off, dtype=dtype, device="cuda")
    t = buf[off:].view(a.shape)
    t.copy_(torch.from_numpy(a))
    return t


@pytest.mark.parametrize("counts,Np,nv,din,dout", [
    ((1,), 1, 2, 16, 16),
    ((64, 1), 13, 5, 80, 48),
    ((127,), 16, 8, 144, 80),
    ((100, 29), 65, 2, 48, 144),
    ((256,), 48, 4, 64, 64),
])
@pytest.mark.parametrize("dtype,off", [("f32", 0), ("f32", 1), ("bf16", 0), ("bf16", 1)])
def test_backward_at_tile_edges(gpu_lib, counts, Np, nv, din, dout, dtype, off):
    import torch
    Q, qo, P, W, G = _tie_free(11, B=len(counts), Np=Np, nv=nv, din=din, dout=dout, margin=1e-6, counts=counts)
    td = torch.float32 if dtype == "f32" else torch.bfloat16
    qd, pd, wd = (_placed(a, td, off) for a in (Q, P, W))
    if dtype == "bf16":
        Q, P, W = (t.float().cpu().numpy() for t in (qd, pd, wd))
    # the views the oracle pairs, so that rounded inputs cannot move one
    am = torch.from_numpy(O.match_forward(Q, qo, P, W)[1].astype(np.int16)).cuda()
    dW, dQ, dP = gpu_lib.match_backward(qd, qo, pd, wd, torch.from_numpy(G).cuda(), am)
    rW, rQ, rP = O.match_backward(Q, qo, P, W, G)
    scale = max(np.abs(rQ).max(), np.abs(rP).max())
    assert np.allclose(dQ.cpu().numpy(), rQ, rtol=1e-4, atol=1e-5 * scale)
    assert np.allclose(dP.cpu().numpy(), rP, rtol=1e-4, atol=1e-5 * scale)
    assert np.allclose(dW.cpu().numpy(), rW, rtol=1e-4, atol=1e-5 * np.abs(rW).max())
