"""The bf16 GEMM's tilings -- CTA pairs (256 x 256 tiles, halves in a short
last round), single CTAs with 256-, 128- and 64-wide tiles -- at the sizes where
they can go wrong: a second CTA without a row of its own, a last row tile of
few rows, one round without halves, halves beside full tiles, several rounds,
both staging depths of the gated residual, K below the ring's depth, and the
rows behind the last one left alone.  The tiling that a case is for is asserted
(on the 152-SM part that the rule was fitted to), for every epilogue.

Tolerances: both sides round the same value to bf16 (rel-L2 <= 2e-3, max error
1.5 bf16 ulps of the output scale: an fp32 sum may land on the other side of a
rounding boundary); r_hat is exact from the stored output.
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


def rt(name, shape, std=1.0, bf16=True):
    return X.random_tensor(13, name, shape, std=std, bf16=bf16)


def dev(a, bf16=True):
    t = torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
    return t.to(torch.bfloat16) if bf16 else t


def close(t, want):
    got = t.double().cpu().numpy()
    assert np.linalg.norm(got - want) <= 2e-3 * np.linalg.norm(want)
    assert np.max(np.abs(got - want)) <= 1.5 * np.max(np.abs(want)) * 2.0 ** -7
    assert xb.op_device_error() == 0


SMS = torch.cuda.get_device_properties(0).multi_processor_count
PAIR, WIDE = 256, 257


def expect(tiling, want):
    if SMS == 152:
        assert tiling == want, (tiling, want)


# (M, N, K, (tiling, full tiles, half tiles)); a last row tile of up to 128 rows
# leaves a pair's second CTA none.  Both staging depths of the gated residual:
# K < 1536 and above.
LINEAR = [
    (1300, 1792, 1600, (PAIR, 42, 0)),       # one round without halves; 20 rows in the last row tile
    (1040, 4352, 1024, (PAIR, 76, 18)),      # one round and halves; 16 rows
    (1040, 4352, 1600, (PAIR, 76, 18)),
    (1690, 2816, 1024, (PAIR, 76, 2)),       # 154 rows: both CTAs have some
    (2060, 4608, 1600, (PAIR, 152, 20)),     # two rounds and halves; 12 rows
    (2190, 4352, 1024, (PAIR, 152, 2)),      # 142 rows
    (2500, 2048, 1024, (PAIR, 76, 8)),
    (2500, 4096, 1600, (PAIR, 152, 16)),
    (2356, 2048, 3392, (WIDE, 152, 0)),      # one round of wide tiles; 52 rows in the last
    (2432, 2048, 1600, {xb.XC_EPI_RESID_CACHE: (128, 304, 0), None: (WIDE, 152, 0)}),
    (2370, 4096, 1600, {xb.XC_EPI_RESID_CACHE: (PAIR, 152, 16), None: (WIDE, 304, 0)}),
    (1300, 1024, 64, (128, 88, 0)),          # one k step
    (1300, 1024, 1600, (128, 88, 0)),
    (130, 512, 128, (64, 16, 0)),
    (1, 256, 1600, (64, 4, 0)),
]


@pytest.mark.parametrize("M,N,K,tiling", LINEAR)
@pytest.mark.parametrize("epi", [xb.XC_EPI_BIAS, xb.XC_EPI_GELU, xb.XC_EPI_RESID_GATE, xb.XC_EPI_RESID_CACHE])
def test_linear_tilings(M, N, K, tiling, epi):
    want = tiling if isinstance(tiling, tuple) else tiling.get(epi, tiling[None])
    expect(xb.debug_gemm_tiling(epi, M, N, K), want)
    A, Wt = rt(f"A{M}{K}", (M, K)), rt(f"W{N}{K}", (N, K), 1 / math.sqrt(K))
    b, g = rt(f"b{N}", (N,), 0.1, False), rt(f"g{N}", (N,), 0.5, False)
    res, xin = rt(f"r{M}{N}", (M, N)), rt(f"x{M}{N}", (M, N))
    out = torch.full((M + 130, N), 7.0, device=DEV, dtype=torch.bfloat16)
    rh = torch.full_like(out, 7.0)
    xb.op_linear("bf16", epi, dev(A), dev(Wt), dev(b, False), out[:M], gate=dev(g, False), resid=dev(res),
                 xin=dev(xin), rhat=rh[:M])
    torch.cuda.synchronize()
    y = (dev(A, False).double() @ dev(Wt, False).double().t()).cpu().numpy() + b
    if epi == xb.XC_EPI_GELU:
        y = O.gelu_tanh(y)
    elif epi != xb.XC_EPI_BIAS:
        y = res + g * y
    close(out[:M], O.to_bf16(y))
    assert bool((out[M:] == 7.0).all()) and bool((rh[M:] == 7.0).all())
    if epi == xb.XC_EPI_RESID_CACHE:
        assert torch.equal(rh[:M], (out[:M].float() - dev(xin).float()).to(torch.bfloat16))


# 2550 rows, N = 2304: pairs; 2100: pairs whose last row tile has 52 rows; 1980: wide
# single tiles
@pytest.mark.parametrize("gh,gw,tiling", [(17, 25, PAIR), (14, 25, PAIR), (15, 22, WIDE)])
@pytest.mark.parametrize("hd", [32, 64, 96, 128])
def test_qkv_rope_pairs(hd, gh, gw, tiling):
    cams, frames, d, chunk = 3, 2, 768, 5
    M, H = cams * frames * gh * gw, d // hd
    expect(xb.debug_gemm_tiling(16, M, 3 * d, d)[0], tiling)
    A, Wt, b = rt(f"qa{hd}", (M, d)), rt(f"qw{hd}", (3 * d, d), 1 / math.sqrt(d)), rt(f"qb{hd}", (3 * d,), 0.1, False)
    q, k, v = (torch.empty(M, d, device=DEV, dtype=torch.bfloat16) for _ in range(3))
    xb.op_qkv_rope("bf16", cams, frames, gh, gw, chunk, hd, 1e4, dev(A), dev(Wt), dev(b, False), q, k, v)
    torch.cuda.synchronize()
    y = A.astype(np.float64) @ Wt.astype(np.float64).T + b
    pos = O.token_positions(cams, frames, gh, gw, chunk)
    for i, t in enumerate((q, k)):
        close(t, O.to_bf16(O.apply_rope(y[:, i * d:(i + 1) * d].reshape(M, H, hd), pos, 1e4).reshape(M, d)))
    close(v, O.to_bf16(y[:, 2 * d:]))
