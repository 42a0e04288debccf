"""Operator calls of several host threads, each on its own stream, from the very
first call of the process on, give what the same calls give one after another:
the launch state that is asked for once per device is asked for by all of them at
once, and the threads have no CUDA context of their own yet."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

SCRIPT = """
import threading, torch
from paper_2604_20289_gb300 import xcache as xb
g = torch.Generator(device="cuda").manual_seed(3)
r = lambda *s: torch.randn(*s, generator=g, device="cuda")
calls = []
def linear(t, m, n, k, epi):      # pairs with halves, wide, 64-wide, fp32 tiles
    a, w, b = r(m, k).to(t), (r(n, k) / k ** 0.5).to(t), r(n)
    res = r(m, n).to(t)
    calls.append(lambda o, st: xb.op_linear("f32" if t == torch.float32 else "bf16", epi, a, w, b, o, gate=b, resid=res, stream=st))
    return torch.empty(m, n, device="cuda", dtype=t)
def attn(t, lq, lk, h, hd):       # cluster, contiguous, fp32
    q, k, v = (r(n, h * hd).to(t) for n in (lq, lk, lk))
    nb = xb.LIB.xc_op_attention_workspace_bytes(1, hd) if t == torch.bfloat16 else 0
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda") if nb else None
    calls.append(lambda o, st: xb.op_attention("f32" if t == torch.float32 else "bf16", h, hd, q, k, v, o, workspace=ws, stream=st))
    return torch.empty_like(q)
bf, f = torch.bfloat16, torch.float32
outs = [linear(bf, 2500, 2048, 512, 2), linear(bf, 2432, 2048, 512, 1), linear(bf, 130, 512, 128, 0),
        linear(f, 500, 512, 96, 2), attn(bf, 840, 2520, 4, 64), attn(bf, 2100, 2600, 21, 64),
        attn(bf, 840, 2520, 6, 128), attn(f, 300, 400, 4, 64)]
streams = [torch.cuda.Stream() for _ in calls]
torch.cuda.synchronize()
errors = []
start = threading.Barrier(len(calls))
def go(i):
    try:
        start.wait()
        for _ in range(5):
            calls[i](outs[i], streams[i])
    except Exception as e:
        errors.append((i, e))
ts = [threading.Thread(target=go, args=(i,)) for i in range(len(calls))]
[t.start() for t in ts]; [t.join() for t in ts]
torch.cuda.synchronize()
assert not errors, errors
for i, c in enumerate(calls):
    again = torch.empty_like(outs[i])
    c(again, None)
    torch.cuda.synchronize()
    assert torch.equal(again, outs[i]), i
assert xb.op_device_error() == 0
print("ok")
"""


def test_first_calls_from_several_threads():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    p = subprocess.run([sys.executable, "-c", SCRIPT], cwd=root, capture_output=True, text=True, timeout=300)
    assert p.returncode == 0 and p.stdout.split() == ["ok"], p.stdout + p.stderr
