"""Sizes and positions that the library computes on the host and the device alike (csrc/sizes.cuh):
the same source built by the host compiler, at the limits of what the calls accept."""
import ctypes
import glob
import os
import re
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
void c_hit_sizes(uint64_t bytes, uint64_t most, uint64_t per, uint64_t warps, uint64_t* out)
{
    const HitSizes h = hit_sizes(bytes, most, per, warps);
    out[0] = h.batches;
    out[1] = h.records;
    out[2] = slab_records(h.records, most, per, warps);
}
void c_sample_positions(uint32_t samples, uint64_t n, uint64_t* out)
{
    for (uint32_t i = 0; i < samples; ++i) out[i] = sample_position(i, samples, n);
}
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


MEAN_RUN = 20   # the mean number of others in a key's run that fewer passes may leave


def _sample(rules, samples, n):
    out = np.empty(samples, np.uint64)
    rules.c_sample_positions(ctypes.c_uint32(samples), ctypes.c_uint64(n), out.ctypes.data_as(ctypes.c_void_p))
    return out


def _pairs(keys):
    c = np.unique(keys, return_counts=True)[1].astype(np.int64)
    return int((c * (c - 1) // 2).sum())


@pytest.mark.parametrize("order", ["shuffled", "sorted", "reversed", "every second"])
@pytest.mark.parametrize("n,samples", [(1 << 20, 2048), (1 << 23, 16384)])
def test_sample_sees_the_runs_whatever_the_order(rules, order, n, samples):
    """Half of the keys spread out, half in dense clusters: the passes that the sample chooses leave
    runs of at most twice the intended mean length (the estimate's spread) for every input order."""
    rng = np.random.default_rng(n)
    keys = rng.integers(0, 1 << 60, n, dtype=np.uint64)
    dense = rng.integers(0, 1 << 60, 40, dtype=np.uint64)[rng.integers(0, 40, n // 2)] >> np.uint64(34) << np.uint64(34)
    keys[n // 2:] = dense | rng.integers(0, 1 << 34, n // 2, dtype=np.uint64)
    if order == "shuffled":
        keys = keys[rng.permutation(n)]
    elif order == "every second":
        keys = np.stack([keys[: n // 2], keys[n // 2:]], 1).reshape(-1)
    else:
        keys.sort()
        keys = keys[::-1] if order == "reversed" else keys
    at = _sample(rules, samples, n)
    assert int(at.max()) < n
    most = (MEAN_RUN + 1) * samples * samples // (2 * n)
    for passes in range(2, 8):
        low = np.uint64(60 - 8 * passes)
        if _pairs(keys[at] >> low) <= most:
            break
    run = np.unique(keys >> low, return_counts=True)[1].astype(np.float64)
    assert (run * run).sum() / n <= 2 * MEAN_RUN, (passes, (run * run).sum() / n, run.max())


def test_sample_positions_stay_inside(rules):
    for n in (1, 2, 8192, 10 ** 8, (1 << 32) - 2):
        assert int(_sample(rules, 16384, n).max()) < n


@pytest.mark.parametrize("dim,groups,intervals", [(2, 4, 4), (2, 4, 25), (3, 2, 27)])
@pytest.mark.parametrize("n", [1, 10 ** 6, 10 ** 8])
def test_sizes_of_the_hit_buffers(rules, dim, groups, intervals, n):
    """Within the bytes given; when those suffice, a record for every group that a batch can report
    however the slabs are left; a few lookups over 10^8 points within 32 MB."""
    warps, per = 152 * 64, 32 * groups
    for m in (1, 3, 10, 100, 10 ** 4, 10 ** 7):
        most = m * (n // 32 // groups + 2 * intervals + 1) // 32 + 1
        for bytes_ in (1 << 20, (1 << 20) + 1024 * m, min(4096 << 20, (1 << 20) + 1024 * m + 4 * n)):
            out = np.empty(3, np.uint64)
            rules.c_hit_sizes(*(ctypes.c_uint64(v) for v in (bytes_, most, per, warps)), out.ctypes.data_as(ctypes.c_void_p))
            batches, records, slab = (int(v) for v in out)
            assert 28 * batches <= bytes_ // 4 and 8 * records <= bytes_ // 4 * 3
            assert batches >= 1 and slab in (per, 512)
            if 28 * most <= bytes_ // 4:
                assert batches == most
            if slab == per and 8 * most * per <= bytes_ // 4 * 3:
                assert records >= most * slab            # a slab for every batch
            if m == 1:
                assert 28 * batches + 8 * records <= 32 << 20


def _kernels(path):
    """Name and body of every __global__ function of a file."""
    src = open(path).read()
    for mt in re.finditer(r"__global__[^;{]*?(\w+_kernel)\s*\(", src):
        start = src.index("{", mt.end())
        depth, end = 1, start + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(src[end], 0)
            end += 1
        yield mt.group(1), src[start + 1:end - 1]


def test_kernels_of_a_chain_wait_before_anything_else():
    """Every kernel that launch_chain starts begins with the wait, and reads what the kernel (or the
    caller's kernel) before it writes through after_wait, at addresses known before the wait."""
    bodies, launched = {}, set()
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        for name, body in _kernels(path):
            bodies[os.path.basename(path), name] = body
        launched |= {(os.path.basename(path), m) for m in
                     re.findall(r"launch_chain\(\s*(\w+_kernel)", open(path).read())}
    assert len(launched) > 20
    for k in launched:
        assert bodies[k].lstrip().startswith("chain_start();"), k
    reads = {("boxes.cu", "boxes_kernel"): ["xy", "keys"], ("boxes.cu", "boxes3_kernel"): ["keys"],
             ("keygen.cu", "keys_kernel"): ["pts"], ("keygen.cu", "decode_kernel"): ["keys"],
             ("keygen.cu", "keys3_kernel"): ["pts"], ("update.cu", "ins_rank_kernel"): ["ikeys"],
             ("update.cu", "tile_starts_kernel"): ["pos"], ("update.cu", "move_kernel"): ["istart"],
             ("query.cu", "plan_kernel"): ["a.perm", "a.q", "a.delta"]}
    for k, names in reads.items():
        for p in names:
            assert f"after_wait({p})" in bodies[k] and f"__ldg({p} " not in bodies[k], (k, p)
