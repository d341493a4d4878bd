"""The selection inside a layer: candidates of the threshold's histogram bin at the limits of its short way (how many one CTA may
send, how many are ranked at once, which keys belong to whom), against a plain sort.  One channel of constant 2 x 2 blocks: at one
level the norms of the low-pass quadrant are (2 v)^2, exact in fp32 for the values used, and all others are zero."""
import numpy as np
import pytest
import torch

from test_gpu_stages import wcc      # noqa: F401  (module fixture)

pytestmark = pytest.mark.gpu

# a CTA has 256 threads of 8, 16 or 32 keys, a cluster 1 to 16 CTAs: both sides of each step
SIZES = [(2, 8), (32, 64), (34, 64), (64, 66), (96, 320), (256, 256), (256, 260), (256, 512)]
CLOSE = [1, 2, 63, 64, 256, 257, 2000]       # keys in the threshold's bin


@pytest.mark.parametrize("together", [True, False])
@pytest.mark.parametrize("close", CLOSE)
@pytest.mark.parametrize("hw", SIZES)
def test_candidates_of_the_threshold_bin(wcc, hw, close, together):      # noqa: F811
    H, W = hw
    n = H * W // 4
    close = min(close, n)
    rng = np.random.default_rng(close + H)
    v = (4.0 + rng.integers(0, 4096, n) / 1024.0).astype(np.float32)     # norms of 64 to 256: above the bin below
    at = np.arange(close) + (n - close) // 2 if together else rng.choice(n, close, replace=False)
    v[at] = 1.0 + rng.integers(0, 512, close).astype(np.float32) / 2.0 ** 19            # norms of 4 to 4 + 2^-7: one bin, some of them equal
    x = torch.from_numpy(np.repeat(np.repeat(v.reshape(H // 2, W // 2), 2, 0), 2, 1)[None, None].copy()).cuda()
    Wt = torch.ones((1, 1), device="cuda")
    nrm = np.zeros((H, W), np.float32)
    nrm[:H // 2, :W // 2] = ((2 * v) * (2 * v)).reshape(H // 2, W // 2)
    order = np.argsort(-nrm.reshape(-1), kind="stable")
    for k in {n - close + 1, n - close + (close + 1) // 2, n}:
        y, t = wcc.forward(x, Wt, 1, k, 8, taps=("idx", "nrm2"))
        assert np.array_equal(t["nrm2"].cpu().numpy().reshape(H, W), nrm)
        assert np.array_equal(t["idx"].cpu().numpy()[0], np.sort(order[:k]))
        assert torch.equal(wcc.forward(x, Wt, 1, k, 8), y)               # (by the threshold alone where no ties are split)
    assert wcc.last_status() == 0
