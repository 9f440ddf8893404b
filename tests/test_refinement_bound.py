"""The bound that lets the half-sweep drop a refinement test (refine_margin and
ncc_bound in pixel_kernel.cuh), restated in numpy FP32 with the kernel's order of
operations: after any part of a window's samples it stays below the cost that all
of them give, plus the margin, on matching, unrelated, flat, offset and scaled
patches."""
import numpy as np
import pytest

F = np.float32


def _sums(w, I, J):
    """Prefix sums over the samples (axis 1), the first one centring J."""
    mu = (np.cumsum(w * I, 1, dtype=F)[:, -1] / np.cumsum(w, 1, dtype=F)[:, -1])[:, None]
    Ic = (I - mu).astype(F)
    wI, Jc = (w * Ic).astype(F), (J - J[:, :1]).astype(F)
    tw = (w * Jc).astype(F)
    s = lambda x: np.cumsum(x, 1, dtype=F)  # noqa: E731
    return s(w), s(wI), s((wI * Ic).astype(F)), s(tw), s((tw * Jc).astype(F)), s((wI * Jc).astype(F))


def _cost_bound_margin(w, I, J):
    sw, sI, sII, sJ, sJJ, sIJ = _sums(w, I, J)
    n = w.shape[1]
    Sw, SIc, SII = sw[:, -1:], sI[:, -1:], sII[:, -1:]
    with np.errstate(all="ignore"):
        varI = (Sw * SII - SIc * SIc).astype(F)
        varJ = (Sw * sJJ[:, -1:] - sJ[:, -1:] ** 2).astype(F)
        cov = (Sw * sIJ[:, -1:] - SIc * sJ[:, -1:]).astype(F)
        eps = F(1e-8) * Sw * Sw
        ncc = np.clip(cov / np.sqrt(varI * varJ), -1, 1)
        ncc = np.where(np.isnan(ncc), -1, ncc)
        cost = np.where((varI < eps) | (varJ < eps), F(2), F(1) - ncc)
        AB = (Sw / w[:, :1]) * (Sw * SII / varI)
        margin = F(5.9604645e-8) * F(14 * n + 20) * AB + F(4e-6)
        margin = np.where(margin < F(0.1), margin, np.inf)
        VI = (sw * sII - sI * sI).astype(F)
        VJ = (sw * sJJ - sJ * sJ).astype(F)
        C = (sw * sIJ - sI * sJ).astype(F)
        scale = Sw / (varI * sw)
        q = np.where(C > 0, C * (C / VJ), 0)
        m2 = 1 / ((VI - q) * scale + 1)
        m2[:, -1] = (q / VI)[:, -1]
        bound = 1 - np.where(VJ > F(1e-8) * sw * sw, np.sqrt(m2), F(1))
    return cost, bound, margin, varI < eps


@pytest.mark.parametrize("n", [9, 36, 49, 121])
def test_bound_stays_below_the_cost(n):
    rng = np.random.default_rng(n)
    T, dropped = 4000, 0
    for kind in range(8):
        I = rng.random((T, n))
        J = rng.random((T, n))
        mix = rng.random((T, 1)) ** 3
        J = np.where(rng.random((T, 1)) < 0.7, (1 - mix) * I + mix * J, J)  # matches of every quality
        if kind == 1:
            J = 1 - J
        if kind == 2:
            I = 0.5 + I * 10.0 ** rng.uniform(-4, 0, (T, 1))  # flat references
        if kind == 3:
            J = 0.7 + J * 10.0 ** rng.uniform(-4, 0, (T, 1))
        if kind == 4:
            J[:, 0] += rng.uniform(-5, 5, T)  # the centring sample apart from the rest
        if kind == 5:
            I, J = 255 * I, 255 * J
        if kind == 6:
            J = np.where(np.arange(n) < rng.integers(2, n, (T, 1)), J, I)  # right only later
        if kind == 7:
            J = np.where(np.arange(n) < rng.integers(2, n, (T, 1)), 0.4, J)  # constant at first
        w = np.exp(-rng.exponential(1.0, (T, n)) * rng.choice([0, 0.3, 2.0, 6.0], (T, 1)))
        cost, bound, margin, flat = _cost_bound_margin(w.astype(F), I.astype(F), J.astype(F))
        ok = ~flat[:, 0]  # (a flat reference is never bounded: its tests end at once)
        over = (bound - cost)[ok] > margin[ok]
        assert not over.any(), (kind, np.argwhere(over)[:3])
        dropped += int((bound[ok][:, n // 2] > margin[ok][:, 0] + 0.05).sum())
    assert dropped > T  # and it is of use: half a window lets many tests go at an incumbent of 0.05
