"""Which half-sweeps go to the bounded kernel (csrc/sweep_policy.h), on the CPU: forms
that it was measured to slow down stay with the pooled kernel, those that it speeds up
do not. The header is built with the host compiler through a small ctypes shim."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2211_16266_gb300", "csrc")
SHIM = os.path.join(ROOT, "tests", "host", "sweep_policy_shim.cpp")
SMS = 152


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("sweep") / "libsweep_policy.so")
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-Wall", "-Wextra", "-Werror", "-fPIC", "-shared",
                           "-I", CSRC, "-o", so, SHIM])
    L = ctypes.CDLL(so)
    L.sw_bounded_serves.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_longlong, ctypes.c_int]
    L.sw_bounded_from.argtypes = [ctypes.c_int, ctypes.c_int]
    L.sw_bounded_from.restype = ctypes.c_longlong
    L.sw_close_cost.restype = ctypes.c_float
    return L


def _tiles(W, H):
    return ((W + 31) // 32) * ((H + 7) // 8)


@pytest.mark.parametrize("W,H,views,side,served", [
    (384, 192, 6, 6, 0), (448, 256, 4, 6, 0), (512, 256, 4, 6, 1), (514, 258, 10, 7, 1), (3840, 1920, 8, 6, 1),
    (1920, 960, 3, 7, 0), (1920, 960, 11, 6, 0), (1920, 960, 16, 6, 0), (1920, 960, 4, 6, 1), (1920, 960, 10, 6, 1),
    (1414, 706, 6, 3, 0), (1414, 706, 6, 4, 0), (1414, 706, 6, 5, 1),
    (514, 258, 4, 5, 0), (640, 320, 4, 5, 1), (514, 258, 5, 5, 1),  # few view-samples, few tiles
])
def test_runs_that_may_use_the_bounded_kernel(lib, W, H, views, side, served):
    assert lib.sw_bounded_serves(views, side, _tiles(W, H), SMS) == served


@pytest.mark.parametrize("W,H", [(512, 256), (640, 320), (1000, 502), (3840, 1920), (16384, 16384)])
def test_its_turn_needs_most_pixels_close(lib, W, H):
    half = W * H // 2  # pixels of a colour
    assert 0.8 * half <= lib.sw_bounded_from(W, H) <= 0.9 * half < 2 ** 32
    assert 0.05 <= lib.sw_close_cost() <= 0.1
