"""Sizes and positions that the library computes on the host and the device alike (csrc/sizes.cuh):
the same source built by the host compiler, at the limits of what the calls accept."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_19891_gb300", "csrc")

SOURCE = """
#include "sizes.cuh"
using namespace sfc;
extern "C" {
uint32_t c_tiles_of(uint64_t n, uint32_t per) { return tiles_of(n, per); }
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("rules")
    (d / "rules.cpp").write_text(SOURCE)
    subprocess.run([cxx, "-std=c++17", "-O2", "-shared", "-fPIC", f"-I{CSRC}", str(d / "rules.cpp"), "-o",
                    str(d / "rules.so")], check=True)
    return ctypes.CDLL(str(d / "rules.so"))


@pytest.mark.parametrize("per", [1024, 2048, 4096])
def test_tiles_cover_the_largest_arrays(rules, per):
    """Every element belongs to a tile, up to the largest n that a sort accepts (2^32 - 2)."""
    rules.c_tiles_of.restype = ctypes.c_uint32
    top = (1 << 32) - 2
    for n in (1, per - 1, per, per + 1, 8192, 10 ** 9, top - per, top - per + 1, top - per + 2, top - 1, top):
        assert rules.c_tiles_of(ctypes.c_uint64(n), ctypes.c_uint32(per)) == -(-n // per), n


def test_no_tile_count_of_the_sort_is_in_32_bits():
    """The sort's kernels and launches take their tile counts from tiles_of."""
    src = open(os.path.join(CSRC, "radix.cu")).read()
    counts = [line for line in src.splitlines() if "tiles =" in line and "small_tiles" not in line]
    assert counts and all("tiles_of(" in line or "uint64_t tiles" in line for line in counts), counts
