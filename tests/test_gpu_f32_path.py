"""The fp32 path's two GEMM tilings and its attention at the sizes where they
can go wrong: remainders of the 16 x 16 and 64 x 64 tiles, both sides of the
switch between them, K that is no multiple of 4 (single loads), operands off
16-byte alignment, more warps than key tiles, ragged queries and keys, and
both warp counts of attention.

Tolerance: fp32 accumulation of K terms against fp64: rel-L2 <= 2e-6 (the
worst case over K <= 1030 random-sign terms is about sqrt(K) 2^-24 = 1.9e-6).
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle as O  # noqa: E402
import xc_inputs as X  # noqa: E402

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2604_20289_gb300 import xcache as xb  # noqa: E402

DEV = torch.device("cuda")


def rt(name, shape, std=1.0):
    return X.random_tensor(11, name, shape, std=std, bf16=False)


def dev(a, off=0):
    """On the device, the first element `off` floats past a 16-byte boundary."""
    t = torch.zeros(a.size + 4, device=DEV)
    t[off:off + a.size] = torch.from_numpy(np.ascontiguousarray(a)).to(DEV).reshape(-1)
    return t[off:off + a.size].view(a.shape)


def rel_l2(t, want):
    return float(np.linalg.norm(t.double().cpu().numpy() - want) / np.linalg.norm(want))


# (M, N, K): 1 and 17 rows, K below and off the 64-wide step, K % 4 != 0; the
# 64 x 64 tiling with remainders in every dimension (N = 592 = 9 x 64 + 16)
@pytest.mark.parametrize("M,N,K", [(1, 16, 1), (17, 48, 70), (64, 64, 256), (33, 16, 1030), (500, 592, 72),
                                   (449, 592, 37), (640, 384, 16)])
@pytest.mark.parametrize("off", [0, 1])
def test_linear_f32_tilings(M, N, K, off):
    A, Wt, b = rt(f"A{M}{K}", (M, K)), rt(f"W{N}{K}", (N, K), 1 / math.sqrt(K)), rt(f"b{N}", (N,), 0.1)
    g, res, xin = rt(f"g{N}", (N,), 0.5), rt(f"r{M}{N}", (M, N)), rt(f"x{M}{N}", (M, N))
    out, rh = torch.full((M + 1, N), 7.0, device=DEV), torch.full((M + 1, N), 7.0, device=DEV)
    xb.op_linear("f32", xb.XC_EPI_RESID_CACHE, dev(A, off), dev(Wt, off), dev(b), out[:M], gate=dev(g), resid=dev(res),
                 xin=dev(xin), rhat=rh[:M])
    torch.cuda.synchronize()
    want = res + g * (A.astype(np.float64) @ Wt.astype(np.float64).T + b)
    assert rel_l2(out[:M], want) <= 2e-6
    assert torch.equal(rh[:M], out[:M] - dev(xin))           # r_hat from the stored output
    assert bool((out[M] == 7.0).all()) and bool((rh[M] == 7.0).all())    # nothing past the last row


# both warp counts (few and many (16-query, head) CTAs), keys below one tile
# and off it, queries off the 16-row tile
@pytest.mark.parametrize("Lq,Lk,H,hd", [(1, 1, 2, 16), (17, 33, 3, 32), (64, 192, 4, 16), (250, 95, 20, 16),
                                        (100, 300, 48, 32), (260, 130, 11, 64), (48, 700, 2, 64)])
@pytest.mark.parametrize("off", [0, 1])
def test_attention_f32_splits(Lq, Lk, H, hd, off):
    d = H * hd
    q, k, v = rt(f"q{Lq}{d}", (Lq, d), 2.0), rt(f"k{Lk}{d}", (Lk, d)), rt(f"v{Lk}{d}", (Lk, d))
    o = torch.full((Lq + 1, d), 7.0, device=DEV)
    xb.op_attention("f32", H, hd, dev(q, off), dev(k, off), dev(v, off), o[:Lq])
    torch.cuda.synchronize()
    want = O.attention(*(a.reshape(-1, H, hd).astype(np.float64) for a in (q, k, v))).reshape(Lq, d)
    assert rel_l2(o[:Lq], want) <= 2e-6
    assert bool((o[Lq] == 7.0).all())


def test_attention_f32_masked_and_extreme_scores():
    """Scores of -inf for a whole key tile (an infinite key component) weigh
    nothing, wherever the tile falls; a NaN score makes the row NaN."""
    H, hd, Lq, Lk = 1, 16, 16, 200
    q, k, v = np.abs(rt("eq", (Lq, hd))) + 0.1, rt("ek", (Lk, hd)), rt("ev", (Lk, hd))
    for lo in (32, 160):                                     # second tile, last full one
        kk = k.copy()
        kk[lo:lo + 32, 3] = -np.inf
        o = torch.empty(Lq, hd, device=DEV)
        xb.op_attention("f32", H, hd, dev(q), dev(kk), dev(v), o)
        keep = np.r_[0:lo, lo + 32:Lk]
        want = O.attention(*(a[:, None].astype(np.float64) for a in (q, k[keep], v[keep])))[:, 0]
        assert rel_l2(o, want) <= 2e-6
    kk = k.copy()
    kk[77] = np.nan
    xb.op_attention("f32", H, hd, dev(q), dev(kk), dev(v), o)
    assert bool(torch.isnan(o).all())
