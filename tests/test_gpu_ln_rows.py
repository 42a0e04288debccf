"""LayerNorm modulation with two rows per CTA (bf16, wider than 512, many rows):
an odd last row, the first row count that takes it, widths off the CTA's 128
threads; and one row per CTA beside it.

Tolerance: both sides round the same value to bf16 (rel-L2 <= 2e-3), fp32
sums of d terms against fp64 (rel-L2 <= 2e-6)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle as O  # noqa: E402
import xc_inputs as X  # noqa: E402

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2604_20289_gb300 import xcache as xb  # noqa: E402


@pytest.mark.parametrize("dtype,M,d", [("bf16", 607, 1040), ("bf16", 608, 528), ("bf16", 701, 5120), ("bf16", 1001, 1536),
                                       ("bf16", 650, 12288), ("f32", 701, 1552)])
def test_ln_two_rows(dtype, M, d):
    bf = dtype == "bf16"
    x = X.random_tensor(23, f"lx{M}{d}", (M, d), std=1.5, bf16=bf) + np.float32(0.5)
    x = X.bf16_representable(x) if bf else x
    sh, sc = (X.random_tensor(23, n + str(d), (d,), std=0.4) for n in ("sh", "sc"))
    T = torch.bfloat16 if bf else torch.float32
    dev = lambda a, t=torch.float32: torch.from_numpy(np.ascontiguousarray(a)).cuda().to(t)   # noqa: E731
    out = torch.full((M + 2, d), 7.0, device="cuda", dtype=T)
    xb.op_ln_mod(dtype, dev(x, T), dev(sh), dev(sc), out[:M], eps=1e-6)
    torch.cuda.synchronize()
    xd = x.astype(np.float64)
    y = (xd - xd.mean(1, keepdims=True)) / np.sqrt(xd.var(1, keepdims=True) + 1e-6) * (1.0 + sc) + sh
    want = O.to_bf16(y) if bf else y
    got = out[:M].double().cpu().numpy()
    assert np.linalg.norm(got - want) <= (2e-3 if bf else 2e-6) * np.linalg.norm(want)
    assert bool((out[M:] == 7.0).all())
