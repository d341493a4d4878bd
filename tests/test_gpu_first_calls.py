"""First calls of a process from several threads at once, each on a stream of its own: what the library looks up about the device on its
first call is never seen half done.  The maps need clusters of sixteen CTAs."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

PROGRAM = """
import threading
import torch
from paper_2205_12268_b200 import wcc
wcc.lib()
gen = torch.Generator(device="cuda").manual_seed(0)
x = torch.randn((1, 8, 256, 512), device="cuda", generator=gen)
Wt = torch.randn((8, 8), device="cuda", generator=gen)
nrm = (x * x).sum(1).reshape(1, -1)
torch.cuda.synchronize()
out = [None] * 8
gate = threading.Barrier(8)

def call(i):
    with torch.cuda.stream(torch.cuda.Stream()):
        gate.wait()
        y = wcc.forward(x, Wt, 2, 30000, 8)
        idx, tau = wcc.select_topk(nrm, 30000)
        torch.cuda.current_stream().synchronize()
        out[i] = (y, idx, tau)

threads = [threading.Thread(target=call, args=(i,)) for i in range(8)]
[t.start() for t in threads]
[t.join() for t in threads]
want = wcc.forward(x, Wt, 2, 30000, 8), *wcc.select_topk(nrm, 30000)
assert all(o is not None and all(torch.equal(a, b) for a, b in zip(o, want)) for o in out)
assert wcc.last_status() == 0
print("same")
"""


def test_first_calls_from_eight_threads():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "same", r.stderr[-2000:]
