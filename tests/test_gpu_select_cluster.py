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
CLOSE = [1, 2, 63, 64, 256, 257, 2000, 2048, 2049]       # keys in the threshold's bin


def _map_of(v, H, W):
    """Map of one channel whose low-pass quadrants hold 2 v at one level ([N, H W / 4]), and its norms [N, H W]."""
    N = v.shape[0]
    q = v.reshape(N, H // 2, W // 2)
    x = np.repeat(np.repeat(q, 2, 1), 2, 2)[:, None]
    nrm = np.zeros((N, H, W), np.float32)
    nrm[:, :H // 2, :W // 2] = (2 * q) * (2 * q)
    return torch.from_numpy(x.copy()).cuda(), nrm.reshape(N, H * W)


def _largest(nrm, k):
    """The kept positions: the k largest norms of every image, the lowest positions among equal ones, ascending."""
    return np.sort(np.argsort(-nrm, axis=1, kind="stable")[:, :k], axis=1)


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
    x, nrm = _map_of(v[None], H, W)
    Wt = torch.ones((1, 1), device="cuda")
    for k in {n - close + 1, n - close + (close + 1) // 2, n}:
        y, t = wcc.forward(x, Wt, 1, k, 8, taps=("idx", "nrm2"))
        assert np.array_equal(t["nrm2"].cpu().numpy().reshape(1, -1), nrm)
        assert np.array_equal(t["idx"].cpu().numpy(), _largest(nrm, k))
        assert torch.equal(wcc.forward(x, Wt, 1, k, 8), y)               # (by the threshold alone where no ties are split)
    assert wcc.last_status() == 0


@pytest.mark.parametrize("hw", [(32, 64), (64, 128)])
def test_crowded_bins_in_lone_ctas(wcc, hw):          # noqa: F811
    """One CTA per image, on every SM at once, more close keys than it ranks directly: the count that says so is set back only
    after all of its warps have read it."""
    H, W = hw
    n, N = H * W // 4, 320
    rng = np.random.default_rng(H)
    v = 1.0 + rng.integers(0, 512, (N, n)).astype(np.float32) / 2.0 ** 19
    v[::3, rng.choice(n, n - 257, replace=False)] += 4.0             # every third image: one key too many, the others: all of them
    x, nrm = _map_of(v.astype(np.float32), H, W)
    Wt = torch.ones((1, 1), device="cuda")
    for k in (n - 200, n - 3):
        want = _largest(nrm, k)
        for _ in range(3):
            y, t = wcc.forward(x, Wt, 1, k, 8, taps=("idx",))
            assert np.array_equal(t["idx"].cpu().numpy(), want)
        assert torch.equal(wcc.forward(x, Wt, 1, k, 8), y)
    assert wcc.last_status() == 0
