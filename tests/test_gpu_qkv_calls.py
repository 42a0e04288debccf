"""QKV + RoPE operator calls that overlap: several streams, several threads and
captured calls, each with a grid, chunk and head_dim of its own, give what the
same call gives alone (bit for bit: one deterministic kernel each).
"""
import threading

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2604_20289_gb300 import xcache as xb  # noqa: E402

DEV = torch.device("cuda")
# (dtype, cams, frames, gh, gw, chunk, d, head_dim): tables of 48 to 5000 entries
SHAPES = [("bf16", 2, 3, 10, 14, 5, 256, 64), ("bf16", 1, 1, 200, 90, 0, 256, 128), ("bf16", 6, 3, 16, 28, 41, 512, 32),
          ("f32", 2, 2, 4, 5, 7, 64, 16)]


class Call:
    def __init__(self, i, shape):
        dtype, cams, frames, gh, gw, chunk, d, hd = shape
        g = torch.Generator(device=DEV).manual_seed(100 + i)
        t = torch.bfloat16 if dtype == "bf16" else torch.float32
        M = cams * frames * gh * gw
        r = lambda *s: torch.randn(*s, generator=g, device=DEV)   # noqa: E731
        self.args = (dtype, cams, frames, gh, gw, chunk, hd, 1e4, r(M, d).to(t), (r(3 * d, d) / d ** 0.5).to(t), r(3 * d))
        self.out = [torch.empty(M, d, device=DEV, dtype=t) for _ in range(3)]
        self()
        torch.cuda.synchronize()
        self.want = [o.clone() for o in self.out]

    def __call__(self, stream=None):
        xb.op_qkv_rope(*self.args, *self.out, stream=stream)

    def clear(self):
        for o in self.out:
            o.zero_()

    def good(self):
        return all(torch.equal(o, w) for o, w in zip(self.out, self.want))


@pytest.mark.parametrize("threads", [False, True])
def test_calls_on_several_streams(threads):
    calls = [Call(i, s) for i, s in enumerate(SHAPES)]
    streams = [torch.cuda.Stream() for _ in calls]
    for rep in range(10):
        for c in calls:
            c.clear()
        torch.cuda.synchronize()

        def go(c, st):
            for _ in range(20):
                c(stream=st)
        if threads:
            ts = [threading.Thread(target=go, args=a) for a in zip(calls, streams)]
            for t in ts:
                t.start()
            for t in ts:
                t.join()
        else:
            for _ in range(20):
                for c, st in zip(calls, streams):
                    c(stream=st)
        torch.cuda.synchronize()
        assert all(c.good() for c in calls), (rep, [c.good() for c in calls])
    assert xb.op_device_error() == 0


def test_captured_call_beside_direct_ones():
    calls = [Call(i, s) for i, s in enumerate(SHAPES)]
    graphs = []
    for c in calls:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            c()
        graphs.append(g)
    big = Call(9, ("bf16", 1, 1, 300, 400, 3, 256, 64))       # a table larger than all before
    for rep in range(5):
        for c in calls:
            c.clear()
        for g in graphs:
            big()
            g.replay()
            big()
        torch.cuda.synchronize()
        assert big.good() and all(c.good() for c in calls), rep
    assert xb.op_device_error() == 0
