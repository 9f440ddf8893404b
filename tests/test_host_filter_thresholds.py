"""The consistency filter's comparisons (csrc/filter_thresholds.h) against the FP32
expressions that they stand for, on the CPU: the wrap of a column difference,
du - W floor(du / W + 1/2), and the distance test sqrt(s) < max_px. Every float
within 3000 of each threshold, the ends of the range and random values between
them decide alike. The header is built with the host compiler through a small
ctypes shim."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2211_16266_gb300", "csrc")
SHIM = os.path.join(ROOT, "tests", "host", "filter_thresholds_shim.cpp")
F = np.float32


@pytest.fixture(scope="module")
def thresholds(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("thresholds") / "libfilter_thresholds.so")
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-Wall", "-Wextra", "-Werror", "-fPIC", "-shared",
                           "-I", CSRC, "-o", so, SHIM])
    L = ctypes.CDLL(so)
    L.ft_thresholds.argtypes = [ctypes.c_int, ctypes.c_float, ctypes.POINTER(ctypes.c_float)]
    L.ft_thresholds.restype = None

    def of(width, max_px=1.0):
        out = (ctypes.c_float * 3)()
        L.ft_thresholds(width, max_px, out)
        return [F(v) for v in out]
    return of


def _around(x, n=3000):
    """The floats within n of x, by their order as integers."""
    i = np.array(x, F).view(np.int32).astype(np.int64)
    order = np.where(i < 0, -(i & 0x7fffffff), i) + np.arange(-n, n + 1)
    order = order[np.abs(order) <= 0x7f800000]
    bits = np.where(order < 0, (-order) | 0x80000000, order).astype(np.uint32)
    return bits.view(F)


@pytest.mark.parametrize("W", [2, 3, 7, 64, 255, 256, 333, 514, 1000, 1001, 1920, 2731, 3840, 4095, 8192, 16383, 16384])
def test_the_wrap_of_a_column_difference(thresholds, W):
    hi, lo, _ = thresholds(W)
    rng = np.random.default_rng(W)
    w = F(W)
    du = np.concatenate([_around(hi), _around(lo), _around(F(0)), rng.uniform(-W, W, 20000).astype(F),
                         np.array([-np.nextafter(w, F(0)), np.nextafter(w, F(0)), F(-0.5) * w, F(0.5) * w], F)])
    du = du[np.abs(du) < w]
    want = du - w * np.floor(du / w + F(0.5))
    got = np.where(du >= hi, du - w, np.where(du < lo, du + w, du))
    assert want.dtype == got.dtype == F
    assert np.array_equal(want, got)


@pytest.mark.parametrize("max_px", [1e-30, 1e-22, 1e-20, 1e-6, 0.1, 0.25, 0.3, 0.5, 0.7, 1.0, 1.5, 2.0, 3.0, 12.0, 777.7, 1e5, 1e18,
                                    1e19, 1e30, 3.4e38, np.inf])
def test_the_distance(thresholds, max_px):
    m = F(max_px)
    sq = thresholds(1920, float(m))[2]
    rng = np.random.default_rng(7)
    s = np.concatenate([_around(sq), _around(F(0)), _around(F(1)), np.array([0, np.inf, 3.4e38], F),
                        (10.0 ** rng.uniform(-44, 38, 20000)).astype(F)])
    s = s[s >= 0]
    with np.errstate(invalid="ignore"):
        assert np.array_equal(np.sqrt(s) < m, s < sq)
    assert not np.nan < sq  # a reprojection that is no number agrees with nothing
