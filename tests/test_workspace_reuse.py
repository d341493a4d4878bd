"""A workspace sized for the largest batch or map of a layer serves the smaller ones: the pipeline that is fastest for them may
need more scratch than the larger problem's."""
import os
import subprocess
import sys

import pytest
import torch

from test_gpu_layer import wcc      # noqa: F401  (fixture)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# Cin, Cout, levels, bits, dtype (0 fp32, 1 bf16), larger (N, H, W), smaller (N, H, W)
LAYERS = [
    (384, 64, 3, 8, 1, (8, 64, 128), (7, 64, 128)),        # one kernel from a number of positions on
    (503, 60, 2, 8, 0, (16, 136, 32), (8, 136, 32)),
    (335, 28, 1, 4, 1, (48, 24, 94), (24, 24, 94)),        # rows of 4m + 2: stored coefficients below it
    (160, 1024, 3, 8, 1, (1, 512, 520), (1, 64, 128)),     # no cluster-wide selection on the larger map
    (91, 2048, 3, 8, 1, (1, 512, 264), (1, 128, 264)),
]
BLOCKS = [(461, 16, 1, 8, 1, (8, 130, 72), (4, 130, 72)), (429, 19, 3, 8, 0, (16, 64, 56), (2, 64, 56))]

# Without a device every launch fails: what is returned is the host's decision (7: workspace too small, 8: a launch was reached).
HOST = """
import ctypes as C, sys
sys.path.insert(0, %r)
from paper_2205_12268_b200 import build, wcc
build.build()
L, a = wcc.lib(), [(1 << 40) * (i + 1) for i in range(5)]
k = lambda s: max(1, s[1] * s[2] // 16)
for cin, cout, lv, bits, dt, big, small in %r:
    n = L.wcc_workspace_bytes(big[0], cin, cout, big[1], big[2], lv, k(big), bits, dt)
    print(L.wcc_forward(a[0], a[1], small[0], cin, cout, small[1], small[2], lv, k(small), bits, a[2], dt, a[3], n, None))
    n = L.wcc_padded_workspace_bytes(big[0], cin, cout, big[1] - 1, big[2], lv, k(big), bits, dt)
    print(L.wcc_forward_padded(a[0], a[1], small[0], cin, cout, small[1] - 1, small[2], lv, k(small), bits, a[2], dt, a[3], n, None))
for c, e, lv, bits, dt, big, small in %r:
    n = L.wcc_block_workspace_bytes(big[0], c, e, big[1], big[2], lv, k(big), bits, dt)
    print(L.wcc_block_forward(a[0], a[1], a[1], a[1], small[0], c, e, small[1], small[2], lv, k(small), bits, a[2], dt, a[3], n, None))
    lay = (wcc.ChainLayer * 2)(wcc.ChainLayer(a[1], c, e, 0.0, 1), wcc.ChainLayer(a[1], e, c, 0.0, 0))
    n = L.wcc_chain_workspace_bytes(lay, 2, big[0], big[1], big[2], lv, k(big), bits, dt)
    print(L.wcc_chain_forward(a[0], lay, 2, small[0], small[1], small[2], lv, k(small), bits, a[2], dt, a[3], n, None))
"""


def test_accepted_by_the_host():
    r = subprocess.run([sys.executable, "-c", HOST % (ROOT, LAYERS, BLOCKS)], env=dict(os.environ, CUDA_VISIBLE_DEVICES=""),
                       capture_output=True, text=True, timeout=600, check=True)
    assert r.stdout.split() == ["8"] * (2 * len(LAYERS) + 2 * len(BLOCKS))


@pytest.mark.gpu
@pytest.mark.parametrize("cfg", LAYERS, ids=lambda c: "%dto%d_L%d_b%d" % c[:4])
def test_same_result(wcc, cfg):      # noqa: F811
    cin, cout, lv, bits, dt, big, small = cfg
    n = wcc.workspace_bytes(big[0], cin, cout, big[1], big[2], lv, big[1] * big[2] // 16, bits, dt)
    N, H, W = small
    g = torch.Generator(device="cuda").manual_seed(cin)
    x = torch.randn((N, cin, H, W), device="cuda", generator=g).to(torch.bfloat16 if dt else torch.float32)
    Wt = torch.randn((cout, cin), device="cuda", generator=g)
    want = wcc.forward(x, Wt, lv, H * W // 16, bits)
    ws = wcc.Workspace(n, x.device)
    ws.buf.fill_(0xFF)
    assert torch.equal(wcc.forward(x, Wt, lv, H * W // 16, bits, ws=ws), want)
    assert wcc.last_status() == 0
