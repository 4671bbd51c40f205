"""The sort over leading digits and the ordering of the runs it leaves: against numpy's stable
argsort, at the sizes where tiles and rules change and for runs around the limit of each path."""
import numpy as np
import pytest
import torch

import oracle
import paper_2508_19891_gb300 as sfc
from conftest import to_dev, u32, u64

pytestmark = pytest.mark.gpu


def _check(keys, dev, ids=None):
    order = np.argsort(keys, kind="stable")
    k, i = sfc.sfc_sort_pairs(to_dev(keys.view(np.int64), dev), None if ids is None else to_dev(ids.view(np.int32), dev))
    want = order.astype(np.uint32) if ids is None else ids[order]
    assert np.array_equal(u64(k), keys[order]) and np.array_equal(u32(i), want)


@pytest.mark.parametrize("n", [1, 2, 31, 1023, 1024, 1025, 4097, 8191, 8192, 8193, 100_003, 466_944, 466_945,
                               (1 << 22) - 1, 1 << 22, 5_000_011])
@pytest.mark.parametrize("bits", [64, 60, 40])
def test_sizes(cuda, n, bits):
    rng = np.random.default_rng(n + bits)
    keys = rng.integers(0, 1 << 63, n, dtype=np.uint64) * 2 + rng.integers(0, 2, n, dtype=np.uint64)
    _check(keys >> np.uint64(64 - bits), cuda, rng.integers(0, 1 << 32, n, dtype=np.uint64).astype(np.uint32))


@pytest.mark.parametrize("runs", [(1,), (2, 3), (63, 64, 65), (511, 512, 513), (2047, 2048, 2049, 6000), (50_000,)])
@pytest.mark.parametrize("inside", ["random", "equal", "two"])
def test_runs(cuda, runs, inside):
    """Runs of equal leading bits, too rare for the sample to see, among single keys: in each the
    remaining bits are random, all equal, or one of two values."""
    rng = np.random.default_rng(sum(runs))
    n = 600_000
    keys = rng.integers(0, 1 << 60, n, dtype=np.uint64)
    at = 0
    for length in runs:
        for _ in range(3):
            top = rng.integers(0, 1 << 40, 1, dtype=np.uint64)[0] << np.uint64(20)
            low = {"random": rng.integers(0, 1 << 20, length), "equal": np.full(length, 77),
                   "two": rng.integers(5, 7, length)}[inside].astype(np.uint64)
            keys[at:at + length] = top | low
            at += length
    _check(keys[rng.permutation(n)], cuda)


@pytest.mark.parametrize("kind", ["equal", "half", "sorted", "reversed", "few", "tight"])
@pytest.mark.parametrize("n", [20_000, 700_001])
def test_skewed_keys(cuda, kind, n):
    rng = np.random.default_rng(n)
    keys = rng.integers(0, 1 << 60, n, dtype=np.uint64)
    if kind == "equal":
        keys[:] = 123456789
    elif kind == "half":
        keys[::2] = keys[0]
    elif kind in ("sorted", "reversed"):
        keys.sort()
        keys = keys[::-1].copy() if kind == "reversed" else keys
    elif kind == "few":
        keys = keys % np.uint64(7) << np.uint64(50)
    else:
        keys[::10] = (keys[0] >> np.uint64(12) << np.uint64(12)) + rng.integers(0, 1 << 12, len(keys[::10]), dtype=np.uint64)
    _check(keys, cuda)


@pytest.mark.parametrize("curve", ["z", "h"])
def test_build_with_stacks_and_a_tight_cluster(cuda, curve):
    """Points of which some lie in stacks of equal points and some in one small square, so that a
    build leaves runs of every kind: the sorted arrays equal the oracle's."""
    rng = np.random.default_rng(9)
    pts = rng.integers(0, 1 << 30, size=(300_000, 2)).astype(np.int32)
    pts[:9000] = rng.integers(0, 1 << 8, size=(9000, 2)) + (1 << 29)
    for s in range(12):
        pts[10_000 + 700 * s: 10_000 + 700 * s + 60 * (s + 1)] = pts[10_000 + 700 * s]
    pts = pts[rng.permutation(len(pts))]
    idx = sfc.sfc_build(to_dev(pts, cuda), curve)
    ref = oracle.build(pts, 30, curve)
    k, i, xy = sfc.sfc_get_sorted(idx)
    assert np.array_equal(u64(k), ref.keys) and np.array_equal(u32(i), ref.ids)
    assert np.array_equal(xy.cpu().numpy(), ref.xy)
    assert sfc.sfc_device_status(idx) == (0, 0)


@pytest.mark.parametrize("order", ["sorted", "reversed", "every second", "every 256th"])
@pytest.mark.parametrize("n", [1 << 20, 1 << 23])
def test_order_of_the_input(cuda, order, n):
    """Keys of which half lie in dense clusters, in orders that follow the curve or interleave the
    two kinds with a period that divides the array."""
    rng = np.random.default_rng(n)
    keys = rng.integers(0, 1 << 60, n, dtype=np.uint64)
    top = rng.integers(0, 1 << 60, 40, dtype=np.uint64) >> np.uint64(34) << np.uint64(34)
    dense = np.ones(n, bool) if "every" in order else rng.random(n) < 0.5
    if "every" in order:
        dense[:: 2 if order == "every second" else 256] = False
    keys[dense] = top[rng.integers(0, 40, int(dense.sum()))] | rng.integers(0, 1 << 34, int(dense.sum()), dtype=np.uint64)
    if order in ("sorted", "reversed"):
        keys.sort()
        keys = keys[::-1].copy() if order == "reversed" else keys
    _check(keys, cuda)
