"""Output head on the last block's own output, both load schedules: grids of at
most two CTAs per SM (four rows' loads in flight) and larger ones, widths that
are no multiple of the 128-column chunk, row counts that are none of 32.

Tolerance: fp32 1e-5 of the row's norm (d fp32 additions); bf16 4e-3 (a
modulated value that fp32 and fp64 round apart differs by one ulp, 2^-8).
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


def cfg_of(dtype, heads, hd, cams, frames, h, w):
    return X.ModelCfg(f"head_{dtype}_{heads}x{hd}_{cams}x{frames}x{h}x{w}", 1, heads * hd, heads, hd, 256, cams, frames,
                      h, w, 2, 2, dtype=dtype)


# 10080 and 9735 tokens: more than 2 x 152 CTAs of 32 rows
@pytest.mark.parametrize("cfg", [cfg_of("f32", 4, 16, 1, 1, 3, 5), cfg_of("f32", 12, 16, 2, 1, 5, 7),
                                 cfg_of("f32", 20, 16, 1, 3, 5, 11), cfg_of("f32", 12, 16, 6, 3, 20, 28),
                                 cfg_of("bf16", 4, 64, 1, 1, 5, 13), cfg_of("bf16", 8, 64, 3, 1, 59, 55)],
                         ids=lambda c: c.name)
def test_head_of_the_last_block(cfg):
    w = X.make_weights(cfg)
    xc = xb.XCache(cfg, w)
    traj = X.Trajectory(cfg, n_chunks=1)
    f32 = cfg.dtype == "f32"
    tr = torch.empty(1, cfg.tokens, cfg.d_model, device="cuda", dtype=torch.float32 if f32 else torch.bfloat16)
    x = torch.tensor(traj.noise(0), dtype=torch.float32, device="cuda")
    v = torch.empty_like(x)
    xc.set_trace(tr)
    try:
        xc.chunk_step(x, traj.action(0), 1.0, 0, False, xb.gate_params(), v_out=v)
        xc.sync()
    finally:
        xc.set_trace(None)
    M = O.OracleModel(cfg, w)
    _, hm = M.cond(1.0, traj.action(0))
    want = M.head(tr[0].double().cpu().numpy(), hm).reshape(cfg.tokens, -1)
    got = v.double().cpu().numpy().reshape(cfg.tokens, -1)
    err = np.linalg.norm(got - want, axis=1) / np.linalg.norm(want, axis=1)
    assert err.max() <= (1e-5 if f32 else 4e-3), (err.argmax(), err.max())
