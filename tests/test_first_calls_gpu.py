"""First calls from several threads at once, in a process of their own: every launcher sets its
kernels' attributes and asks the device once, whichever thread comes first, and each thread's
results are those of a single one, bit for bit."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = r"""
import threading
import numpy as np, torch
from paper_2410_11625_gb300 import flr, flnr
dev = "cuda"
gen = torch.Generator(dev).manual_seed(1)
x = torch.rand((2, 11, 64, 64), device=dev, generator=gen)
go = torch.rand((2, 8, 64, 64), device=dev, generator=gen)
weights = flnr.init_weights(3)
torch.cuda.synchronize()

def work(res):
    with torch.cuda.stream(torch.cuda.Stream()):
        net = flnr.FLNR(2 * 64 * 64, weights)
        g = net.forward(x)
        net.zero_grads(x)
        net.backward(go)
        fast = flr.FastFLR(q=8)
        y = x[0, 8:11].contiguous()
        o = fast.denoise(g[0], y)
        p = fast.param_grad(g[0], y, torch.ones_like(y))
        f = flr.FLR(q=8, radius=4, coef_radius=4)
        d = f.denoise(g[0], y)
        b = f.backward(g[0], y, torch.ones_like(y), need_eps=True)
        torch.cuda.current_stream().synchronize()
        res += [t.cpu() for t in (g, o, p, d, b["guide"], b["radiance"])] + [torch.from_numpy(net.grads())]
        net.close(); fast.close(); f.close()

start = threading.Barrier(6)
results = [[] for _ in range(6)]
def run(k):
    torch.cuda.set_device(0)
    start.wait()
    work(results[k])
threads = [threading.Thread(target=run, args=(k,)) for k in range(6)]
[t.start() for t in threads]
[t.join() for t in threads]
alone = []
work(alone)
for r in results:
    assert len(r) == len(alone)
    for a, b in zip(r, alone):
        assert torch.equal(a, b)
print("ok")
"""


def test_first_calls_from_several_threads():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    r = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stderr[-2000:]
