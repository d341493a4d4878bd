"""Sizes at the ends of 32-bit counts are accepted by the host.  Run without a device, where every launch fails (8): a refusal of the
shape itself would be 2."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HOST = """
import sys
sys.path.insert(0, %r)
from paper_2205_12268_b200 import build, wcc
build.build()
L, a = wcc.lib(), [(1 << 40) * (i + 1) for i in range(5)]
for dt in (0, 1):
    print(L.wcc_haar_fwd(a[0], 1 << 30, 1, 2, 2, 1, dt, a[1], a[2], None))             # 2^30 tiles of four positions
    n = L.wcc_padded_workspace_bytes(65535, 8192, 1, 15, 1, 3, 1, 0, dt)
    print(L.wcc_forward_padded(a[0], a[1], 65535, 8192, 1, 15, 1, 3, 1, 0, a[2], dt, a[3], n, None))      # 2^33 padded rows
"""


def test_accepted_by_the_host():
    r = subprocess.run([sys.executable, "-c", HOST % ROOT], env=dict(os.environ, CUDA_VISIBLE_DEVICES=""), capture_output=True, text=True,
                       timeout=600, check=True)
    assert r.stdout.split() == ["8"] * 4
