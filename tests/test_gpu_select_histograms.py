"""The selection inside a layer on histograms supplied by the test: as the first pass fills them, and such that do not match the norms (what
a workspace holds that something else writes to).  The former select as a plain sort does; the latter keep at most k positions, write
nothing beyond the lists they were given, and end."""
import numpy as np
import pytest
import torch

from test_gpu_stages import wcc      # noqa: F401  (module fixture)

pytestmark = pytest.mark.gpu

GUARD = 4096
WCC_ERR_TIMEOUT = 9


def _histograms(nrm):
    b = nrm.view(np.uint32)
    b = b[b != 0]
    return np.bincount(b >> 20, minlength=2048)[:2048], np.bincount(b >> 15, minlength=65536)[:65536]


def _select(wcc, nrm, k, h11, h16, want_rank, late=False):        # noqa: F811
    P = nrm.size
    dev = [torch.from_numpy(np.ascontiguousarray(a).astype(np.int32)).cuda() for a in (h11, h16)]
    thr = torch.zeros(4, dtype=torch.int32, device="cuda")
    rank = torch.full((P,), -2, dtype=torch.int32, device="cuda")
    idx = torch.full((k + GUARD + P,), -3, dtype=torch.int32, device="cuda")       # (room for all: an overrun is seen, not made)
    wcc.debug_select(torch.from_numpy(nrm).cuda(), k, *dev, want_rank, thr, rank, idx, late)
    assert wcc.last_status() == (WCC_ERR_TIMEOUT if late else 0)
    assert bool((idx[k:] == -3).all()), "wrote beyond its list"
    thr, rank, idx = thr.cpu().numpy().view(np.uint32), rank.cpu().numpy(), idx[:k].cpu().numpy()
    keys = np.where(nrm.view(np.uint32) == 0, np.uint32(0x80000000), nrm.view(np.uint32) | np.uint32(0x80000000))
    kept = (rank >= 0) if thr[2] else (keys >= thr[0])
    if thr[2]:
        assert rank.min() >= -1 and rank.max() < k
    if thr[2] and not late:
        assert np.array_equal(idx[rank[kept]], np.flatnonzero(kept))
    return np.flatnonzero(kept)


def _norms(P, seed):
    return (np.random.default_rng(seed).random(P) ** 3 * 50 + 1e-3).astype(np.float32)


@pytest.mark.parametrize("want_rank", [False, True])
@pytest.mark.parametrize("P", [1, 500, 2048, 2049, 8192, 16384])
def test_matching_histograms(wcc, P, want_rank):      # noqa: F811
    nrm = _norms(P, P)
    nrm[::5] = 0.0
    h = _histograms(nrm)
    for k in sorted({1, P // 3 + 1, int((nrm > 0).sum()) or 1}):
        assert np.array_equal(_select(wcc, nrm, k, *h, want_rank), np.sort(np.argsort(-nrm, kind="stable")[:k]))


@pytest.mark.parametrize("want_rank", [False, True])
@pytest.mark.parametrize("P", [2000, 5000, 16384])
def test_histograms_of_something_else(wcc, P, want_rank):      # noqa: F811
    nrm, k = _norms(P, P), P // 4
    h11, h16 = _histograms(nrm)
    none = np.zeros_like(h16)
    assert _select(wcc, nrm, k, h11, none, want_rank).size == 0                   # no fine bin holds the threshold
    top = np.zeros_like(h11), np.zeros_like(h16)                                  # more keys in the threshold's bin than there are
    b = int(np.float32(40.0).view(np.uint32)) >> 15
    top[0][b >> 5] = top[1][b] = P
    assert _select(wcc, nrm, k, *top, want_rank).size == 0
    close = (1.0 + np.arange(P) / 2.0 ** 23).astype(np.float32)                   # one bin of everything, and one key too few to find
    h11, h16 = _histograms(close)
    h11, h16 = h11 * 2, h16 * 2
    assert _select(wcc, close, P, h11, h16, want_rank).size == P
    close[: P // 2] = 0.25
    assert _select(wcc, close, P - 1, h11, h16, want_rank).size == 0
    for seed in range(4):                                                         # anything at all
        rng = np.random.default_rng(seed)
        h = rng.integers(0, 4, 2048) * rng.integers(0, P, 2048), rng.integers(0, 3, 65536) * rng.integers(0, P, 65536)
        assert _select(wcc, nrm, k, *h, True).size <= k
        _select(wcc, nrm, k, *h, False)


@pytest.mark.parametrize("want_rank", [False, True])
@pytest.mark.parametrize("P", [4096, 8192, 16384])     # clusters of two, four and eight
def test_a_wait_that_runs_out(wcc, P, want_rank):      # noqa: F811
    """One CTA of the cluster gives up its wait for candidates.  It stays until its neighbours, which heard everything, have left or need
    to hear from it: at the end of the threshold alone, in front of an ordered compaction (asked for, or ties kept in part), and where
    there are more candidates than the messages hold, in front of their spreading and of the histogram rounds."""
    plain = _norms(P, P)
    ties = plain.copy()
    ties[:: P // 50] = 7.0                             # few enough for the messages
    crowd = (1.0 + np.arange(P) / 2.0 ** 23).astype(np.float32)
    some = plain.copy()                                # too many for the messages, not for one CTA
    some[: P // 4] = (20.0 + np.arange(P // 4) / 2.0 ** 18).astype(np.float32)[: P // 4]
    some[1000:P // 4] = 0.5
    wcc.debug_set_wait_limit(300)
    try:
        for nrm, k in ((plain, P // 4), (ties, int((ties > 7).sum()) + 20), (some, int((some > 20).sum()) - 300), (crowd, P // 2)):
            h = _histograms(nrm)
            got = _select(wcc, nrm, k, *h, want_rank, late=True)
            right = np.sort(np.argsort(-nrm, kind="stable")[:k])
            assert got.size == 0 or (not want_rank and nrm is plain and np.array_equal(got, right))
    finally:
        wcc.debug_set_wait_limit(0)
    assert np.array_equal(_select(wcc, plain, P // 4, *_histograms(plain), want_rank), np.sort(np.argsort(-plain, kind="stable")[: P // 4]))
