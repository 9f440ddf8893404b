"""The counting form of the median filter against a plain sort, bit for bit.

Sizes at the edges of its 32 x 32 tiles and narrower than its window, thresholds
on both sides of tau = 1/4 (above it the kernel sorts), ranges that tie exactly
at the threshold, and values that send a block to the sorting form (infinite, NaN,
negative, tiny and huge ones).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pm():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2211_16266_gb300 as pm
    return pm


def _reference(d, r, tau):
    H, W = d.shape
    pad = np.full((H + 2 * r, W), np.nan, np.float32)
    pad[r:r + H] = d
    win = np.stack([np.roll(pad[a:a + H], -b, 1) for a in range(2 * r + 1) for b in range(-r, r + 1)])
    ok = win > 0
    n = ok.sum(0)
    s = np.sort(np.where(ok, win, np.float32(np.inf)), 0)
    m = np.take_along_axis(s, np.maximum(n - 1, 0)[None] // 2, 0)[0]
    with np.errstate(invalid="ignore", over="ignore"):
        gone = np.abs(d - m) > np.float32(tau) * m
    return np.where((d > 0) & ~gone, d, np.float32(0))


def _maps(W, H, seed):
    rng = np.random.default_rng(seed)
    smooth = (2 + 0.3 * rng.standard_normal((H, W))).astype(np.float32)
    holes = np.where(rng.random((H, W)) < 0.3, 0, smooth).astype(np.float32)
    steps = (rng.integers(60, 72, (H, W)) / np.float32(64)).astype(np.float32)  # ties with the median and at the threshold
    sparse = np.where(rng.random((H, W)) < 0.9, 0, smooth).astype(np.float32)
    strange = holes.copy()
    for v in (np.inf, -np.inf, np.nan, -1.0, 1e-41, 1e-12, 3e38, 2.0 ** 30):
        strange[rng.random((H, W)) < 0.01] = v
    scaled = (holes * np.float32(2.0 ** -29)).astype(np.float32)
    return [smooth, holes, steps, sparse, strange, scaled]


@pytest.mark.parametrize("W,H", [(64, 32), (65, 33), (31, 31), (5, 70), (1, 1), (2, 9), (127, 63)])
@pytest.mark.parametrize("r", [1, 2, 3])
def test_counts_decide_as_a_sort(pm, W, H, r):
    import torch
    with pm.Context(0) as ctx:
        for k, d in enumerate(_maps(W, H, W * 31 + H + r)):
            for tau in (1e-30, 1e-6, 0.05, 0.0625, 0.25, 0.26, 0.9):
                got = pm.pmsp_median_filter(ctx, torch.from_numpy(d).cuda(), r, tau).cpu().numpy()
                want = _reference(d, r, tau)
                assert np.array_equal(got.view(np.uint32), want.view(np.uint32)), (k, tau)
