"""Resource use of the bounded half-sweep (bounded_kernel), as ptxas reports it (no
GPU): the instances run the resident blocks per SM of their view count's half-sweep
(5 of 128 threads up to 4 views, 4 up to 8, 3 above) without spills and within an
SM's shared memory.
"""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2211_16266_gb300", "csrc")


@pytest.mark.parametrize("views,blocks", [(4, 5), (6, 4), (8, 4), (10, 3)])
def test_bounded_instances_stay_within_their_budget(views, blocks, tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src = tmp_path / "bounded.cu"  # any window, 11x11 / 2, 7x7
    src.write_text('#include "pixel_kernel.cuh"\nnamespace pmsp {\n' + "".join(
        f"template __global__ void bounded_kernel<{views}, {win}>(const __grid_constant__ PixelParams);\n"
        for win in range(3)) + "}\n")
    r = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "--expt-relaxed-constexpr",
                        "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-Xptxas", "-v", "-c", str(src),
                        "-o", str(tmp_path / "k.o")], capture_output=True, text=True, check=True)
    found = 0
    for entry in r.stderr.split("Compiling entry function '")[1:]:
        if "bounded_kernel" not in entry.split("'")[0]:
            continue
        found += 1
        spills = re.search(r"(\d+) bytes spill stores, (\d+) bytes spill loads", entry)
        used = re.search(r"Used (\d+) registers.*?(\d+) bytes smem", entry)
        assert spills.groups() == ("0", "0"), entry
        assert int(used.group(1)) * 128 * blocks <= 65536, entry
        assert (int(used.group(2)) + 1024) * blocks <= 228 * 1024, entry  # 1 KB a block is the system's
    assert found == 3
