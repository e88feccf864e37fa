"""The list of the problems that a launch serves (k_device.cuh: Served) holds any slot number: a batch may have more
members than 16 bits count.  Compiled against the device header; no GPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = """
#include "k_device.cuh"
#include <climits>
#include <limits>
static_assert(std::numeric_limits<std::remove_extent_t<decltype(hn::Served::slot)>>::max() >= INT_MAX, "slot numbers");
static_assert(std::numeric_limits<std::remove_extent_t<decltype(hn::Served::level)>>::max() >= hn::kMaxLevel, "levels");
"""


def test_the_list_of_served_problems_holds_every_slot_number(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src = tmp_path / "list.cu"
    src.write_text(SOURCE)
    csrc = os.path.join(ROOT, "paper_0904_4152_gb300", "csrc")
    r = subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "--expt-relaxed-constexpr",
                        "-I", csrc, "-c", str(src), "-o", str(tmp_path / "list.o")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
