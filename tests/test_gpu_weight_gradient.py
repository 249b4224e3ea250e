"""The weight gradient with its reduction in parts, on single SMs (several tiles) and on pairs, at ragged sizes, against
float64 from a fixed argmax."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# d_out x d_in and the longer reduction, over N_p n_v views: one tile; 3 x 9 tiles of one SM; 2 x 16 and 2 x 9 of pairs
@pytest.mark.parametrize("dtype,nv,Np,din,dout", [
    ("float32", 20, 1001, 80, 48), ("bfloat16", 21, 401, 1040, 272), ("float32", 21, 401, 1040, 272),
    ("bfloat16", 64, 397, 4096, 512), ("float32", 33, 905, 2064, 512)])
def test_weight_gradient(gpu_lib, dtype, nv, Np, din, dout):
    import torch
    g = torch.Generator(device="cuda").manual_seed(nv * Np)
    counts = np.resize([20, 33, 64], 38)
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    nq, dt = int(off[-1]), getattr(torch, dtype)
    q = torch.randn((nq, din), generator=g, device="cuda").to(dt)
    p = torch.randn((Np, nv, din), generator=g, device="cuda").to(dt)
    w = (torch.randn((dout, din), generator=g, device="cuda") / din ** 0.5).to(dt)
    am = torch.randint(0, nv, (nq, Np), generator=g, device="cuda", dtype=torch.int16)
    gS = torch.randn((len(counts), Np), generator=g, device="cuda")
    dW = gpu_lib.match_backward(q, off, p, w, gS, am, (True, False, False))[0].double()

    q64, p64, w64 = q.double(), p.reshape(-1, din).double(), w.double()
    u, v = q64 @ w64.T, p64 @ w64.T
    un, vn = u.norm(dim=1, keepdim=True), v.norm(dim=1, keepdim=True)
    uh, vh = u / un, v / vn
    rows = torch.from_numpy(np.repeat(np.arange(len(counts)), counts)).cuda()
    c = gS.double()[rows] / torch.from_numpy(counts).cuda().double()[rows][:, None]
    at = torch.arange(Np, device="cuda")[None, :] * nv + am.long()
    G, H = torch.zeros_like(u), torch.zeros_like(v)
    Ga, Ha = torch.zeros_like(u), torch.zeros_like(v)  # with the absolute values of every term: what rounding scales with
    for i in range(0, nq, 64):
        s = slice(i, i + 64)
        x = vh[at[s]]
        G[s], Ga[s] = (c[s][:, :, None] * x).sum(1), (c[s].abs()[:, :, None] * x.abs()).sum(1)
        t = c[s][:, :, None] * uh[s][:, None, :]
        H.index_add_(0, at[s].reshape(-1), t.reshape(-1, dout))
        Ha.index_add_(0, at[s].reshape(-1), t.abs().reshape(-1, dout))

    def tangent(g_, ga, xh, n):
        return (g_ - (g_ * xh).sum(1, keepdim=True) * xh) / n, (ga + (ga * xh.abs()).sum(1, keepdim=True) * xh.abs()) / n
    dU, aU = tangent(G, Ga, uh, un)
    dV, aV = tangent(H, Ha, vh, vn)
    ref, scale = dU.T @ q64 + dV.T @ p64, aU.T @ q64.abs() + aV.T @ p64.abs()
    # each factor in two BF16 parts is 2^-16 off, u and v (twice each), the sums and the last product: 16 of these
    assert ((dW - ref).abs() <= 2.0 ** -12 * scale).all()
    assert (dW - ref).norm() <= 2.0 ** -12 * ref.norm()
