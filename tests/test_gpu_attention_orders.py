"""bf16 attention's work orders at the sizes where they can go wrong: units
split over several CTAs (evenly, and over all SMs with shares that touch two
units), whole units in waves with and without a last round, no workspace, a
second query tile without a row, ragged keys, one key tile; and scores that
outgrow the running max at head_dim 128, whose later tiles take no max of
their own.

Tolerance: the probabilities are rounded to bf16 before P V, 2^-9 relative
noise averaged over the keys: rel-L2 <= 5e-3 over all rows, 2e-2 for each.
"""
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


def check(q, k, v, H, hd, workspace):
    Lq, d = q.shape
    bf = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV).to(torch.bfloat16)   # noqa: E731
    o = torch.full((Lq + 64, d), 7.0, device=DEV, dtype=torch.bfloat16)
    xb.op_attention("bf16", H, hd, bf(q), bf(k), bf(v), o[:Lq], workspace=workspace)
    torch.cuda.synchronize()
    want = O.to_bf16(O.attention(*(a.reshape(-1, H, hd).astype(np.float64) for a in (q, k, v))).reshape(Lq, d))
    got = o[:Lq].double().cpu().numpy()
    assert np.linalg.norm(got - want) <= 5e-3 * np.linalg.norm(want)
    row = np.linalg.norm((got - want).reshape(Lq, H, hd), axis=2) / np.linalg.norm(want.reshape(Lq, H, hd), axis=2)
    assert row.max() <= 2e-2, row.max()
    assert bool((o[Lq:] == 7.0).all())                       # nothing past the last row
    assert xb.op_device_error() == 0


# (Lq, Lk, H, hd) on 152 SMs: 16 units in clusters; one unit in a cluster of 8;
# 90 units over all SMs (shares touch two units); 2 units of 3 tiles; whole
# units: 4 of them, 160 (a second round of 8), 240; contiguous cut: 189 units;
# clusters of 3, of 6 at hd 128; 4 units split 15 ways
@pytest.mark.parametrize("Lq,Lk,H,hd", [(840, 2520, 4, 64), (130, 5000, 1, 128), (2196, 3000, 10, 64),
                                        (300, 300, 1, 128), (100, 77, 4, 64), (2500, 500, 16, 128),
                                        (5000, 129, 12, 64), (2100, 2600, 21, 64),
                                        (1400, 1000, 7, 64), (840, 2520, 6, 128), (300, 9000, 2, 128)])
@pytest.mark.parametrize("workspace", ["auto", None])
def test_attention_orders(Lq, Lk, H, hd, workspace):
    d = H * hd
    q, k, v = (X.random_tensor(17, n + f"{r}x{d}", (r, d), std=s, bf16=True)
               for n, r, s in (("q", Lq, 1.5), ("k", Lk, 1.0), ("v", Lk, 1.0)))
    check(q, k, v, H, hd, workspace)


# Hot keys from the second tile on, each its query's direction times c: the
# score outgrows the first tile's max by c sqrt(128) / ln 2 in log2 units -- 16 c:
# 32 (no raise), 80 (raise), 240 (first pass infinite); then growing over tiles
@pytest.mark.parametrize("c", [2.0, 5.0, 15.0])
@pytest.mark.parametrize("workspace", ["auto", None])
def test_attention_hd128_outgrown_max(c, workspace):
    Lq, Lk, hd = 256, 1500, 128
    q = X.random_tensor(19, "oq", (Lq, hd), bf16=True)
    k = X.random_tensor(19, "ok", (Lk, hd), std=0.05, bf16=True)
    v = X.random_tensor(19, "ov", (Lk, hd), bf16=True)
    for rep, at in ((0.6, 200), (1.0, 700), (0.8, 1200)):    # three hot keys per query, the largest in the middle
        k[at + np.arange(Lq)] = X.bf16_representable((q * c * rep).astype(np.float32))
    check(q, k, v, 1, hd, workspace)
