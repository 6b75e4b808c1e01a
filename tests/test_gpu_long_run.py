"""Many train steps in a row on layer streams finish: their CTA pairs start
beside other layers' blocks, at different times on the pair's two SMs.  In
processes of their own, with a limited wait: a stream that stopped would hold
up an orderly end."""

import os
import subprocess
import sys

import pytest

from tests.gpu_common import lib_ready, torch_cuda

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

_CHILD = r"""
import os, sys
sys.path.insert(0, {root!r})
import torch
from paper_2404_08573_gb300 import ff
kind, prec, steps, n, dims = {kind!r}, {prec!r}, {steps}, {n}, {dims}
layers = [ff.Layer(dims[k], dims[k + 1], prec=prec, lr=1e-3, init_seed=k, max_rows=2 * n)
          for k in range(len(dims) - 1)]
x = torch.rand(2 * n, dims[0], device="cuda")
y = torch.randint(0, 10, (2 * n,), device="cuda", dtype=torch.int32)
if kind == "po":
    net = ff.PoNet(layers, [ff.Head(d, max_rows=n) for d in dims[1:]], max_rows=n)
    step = lambda: net.train_step(x[:n], y[:n])
else:
    net = ff.Net(layers, max_B=n)
    step = lambda: net.train_step(x, y, B=n)
for s in range(steps):
    step()
    if s % 500 == 499:
        try:
            net.wait(10000)
        except ff.FFError as e:
            print("step", s, e, flush=True)
            os._exit(7)
net.sync()
torch.cuda.synchronize()
for l in layers:
    l.check()
print("done", flush=True)
"""


@pytest.mark.parametrize("kind,prec,steps,n,dims", [("ff", "bf16", 20000, 1024, (784, 2000, 2000, 2000, 2000)),
                                                    ("po", "bf16", 8000, 1024, (784, 2000, 2000, 2000, 2000)),
                                                    ("ff", "fp32", 4000, 256, (784, 2000, 2000, 2000, 2000))])
def test_layer_streams_keep_running(kind, prec, steps, n, dims):
    torch_cuda()
    lib_ready()
    r = subprocess.run([sys.executable, "-c", _CHILD.format(root=ROOT, kind=kind, prec=prec, steps=steps, n=n, dims=dims)],
                       capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout[-500:] + r.stderr[-2000:]
    assert "done" in r.stdout
