"""The scan passes' items (groups of 32 sorted points, 128 in 2-D and 64 in 3-D per item, 32 items
per batch) at the sizes where their edges lie: bit-exact against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2508_19891_gb300 as sfc
from conftest import to_dev, u32, u64

pytestmark = pytest.mark.gpu


def _check(idx, qs, d, roff, rids, dev):
    off, ids = sfc.query(idx, to_dev(qs, dev), to_dev(d, dev))
    assert np.array_equal(u64(off), roff) and np.array_equal(u32(ids), rids)
    assert sfc.sfc_device_status(idx) == (0, 0)


def _radii(rng, m, side):
    """From 0 to beyond the whole set: empty windows, single groups, every group inside."""
    d = np.exp(rng.uniform(0, np.log(2.0 * side), m)).astype(np.int32)
    d[: m // 8] = 0
    d[-2:] = [2 * side, 2 ** 31 - 1]
    return d


@pytest.mark.parametrize("n", [1, 31, 32, 33, 127, 128, 129, 4095, 4096, 4097, 20_011])
@pytest.mark.parametrize("norm", ["disc", "square"])
def test_item_edges(cuda, n, norm):
    rng = np.random.default_rng(n)
    side = 4000
    pts = rng.integers(0, side, size=(n, 2)).astype(np.int32)
    pts[: n // 3] = pts[0]                               # one stack over many groups
    m = 203
    qs = rng.integers(0, side, size=(m, 2)).astype(np.int32)
    qs[::3] = pts[rng.integers(0, n, len(qs[::3]))]
    d = _radii(rng, m, side)
    ref = oracle.build(pts)
    roff, rids = oracle.query(ref, qs, d, norm=norm)
    for cover in (0, 1, 2):
        for reorder in (0, 1):
            idx = sfc.sfc_build(to_dev(pts, cuda), "z", cover_refine=cover, reorder_queries=reorder, query_norm=norm)
            _check(idx, qs, d, roff, rids, cuda)


@pytest.mark.parametrize("n", [1, 32, 63, 64, 65, 2047, 2048, 2049, 9001])
def test_item_edges_3d(cuda, n):
    rng = np.random.default_rng(n)
    side = 900
    pts = rng.integers(0, side, size=(n, 3)).astype(np.int32)
    pts[: n // 3] = pts[0]
    m = 101
    qs = rng.integers(0, side, size=(m, 3)).astype(np.int32)
    d = _radii(rng, m, side)
    d[-1] = 1 << 21
    roff, rids = oracle.query3(oracle.build3(pts), qs, d)
    for cover in (0, 1):
        idx = sfc.sfc_build3(to_dev(pts, cuda), cover_refine=cover)
        _check(idx, qs, d, roff, rids, cuda)


@pytest.mark.parametrize("reorder", [0, 1])
def test_items_past_the_budget(cuda, reorder):
    """Windows that scan far more than a 1 MB budget keeps records for (the write pass filters
    those queries again) next to small ones, on the device, in host slices and with a capacity
    that cuts the output short."""
    rng = np.random.default_rng(3)
    n, m = 150_000, 120
    pts = rng.integers(0, 1 << 20, size=(n, 2)).astype(np.int32)
    qs = rng.integers(0, 1 << 20, size=(m, 2)).astype(np.int32)
    d = rng.integers(0, 3000, m).astype(np.int32)
    d[rng.permutation(m)[:90]] = rng.integers(1 << 19, 1 << 20, 90)
    roff, rids = oracle.query(oracle.build(pts), qs, d, threads=8)
    assert len(rids) * 4 >= 32 << 20                     # the host call copies it out in slices
    idx = sfc.sfc_build(to_dev(pts, cuda), "z", mask_budget_mb=1, reorder_queries=reorder)
    _check(idx, qs, d, roff, rids, cuda)
    hoff, hids = sfc.sfc_query_batch_host(idx, qs, d, len(rids))
    assert np.array_equal(hoff, roff) and np.array_equal(hids, rids)
    cap = len(rids) // 2 + 7
    out = torch.full((len(rids),), -1, dtype=torch.int32, device=cuda)
    off = torch.empty(m + 1, dtype=torch.int64, device=cuda)
    sfc.sfc_query_batch(idx, to_dev(qs, cuda), to_dev(d, cuda), off, out, capacity=cap)
    assert np.array_equal(u64(off), roff)
    got = u32(out)
    assert np.array_equal(got[:cap], rids[:cap]) and (got[cap:] == 0xFFFFFFFF).all()
    assert sfc.sfc_device_status(idx)[1] == sfc.SFC_DEV_CAPACITY


@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 4096, 70_001])
@pytest.mark.parametrize("spread", ["stack", "two", "corner", "domain"])
def test_bounds_behind_the_directory(cuda, n, spread):
    """Array positions of interval ends for key ranges of every kind: one key only, two far apart,
    a small corner (directory parts narrower than a cell), the whole domain."""
    rng = np.random.default_rng(n)
    top = (1 << 30) - 1
    pts = {"stack": np.full((n, 2), 12345), "two": rng.integers(0, 2, size=(n, 1)) * np.array([[top, top]]),
           "corner": rng.integers(0, 50, size=(n, 2)), "domain": rng.integers(0, top + 1, size=(n, 2))}[spread].astype(np.int32)
    m = 64
    qs = np.concatenate([rng.integers(0, top + 1, size=(m // 2, 2)), pts[rng.integers(0, n, m // 2)]]).astype(np.int32)
    d = np.exp(rng.uniform(0, np.log(2.0 ** 31 - 1), m)).astype(np.int32)
    for curve in ("z", "h"):
        ref = oracle.build(pts, 30, curve)
        for cover in (0, 1, 2):
            idx = sfc.sfc_build(to_dev(pts, cuda), curve, cover_refine=cover)
            K = sfc.sfc_query_max_intervals(idx)
            lo, hi, b, e, c = sfc.sfc_query_ranges(idx, to_dev(qs, cuda), to_dev(d, cuda))
            lo, hi, b, e, c = u64(lo), u64(hi), u32(b), u32(e), u32(c)
            for i in range(m):
                for r in range(int(c[i])):
                    assert b[K * i + r] == oracle.lower_bound(ref.keys, int(lo[K * i + r]))
                    assert e[K * i + r] == oracle.lower_bound(ref.keys, int(hi[K * i + r]) + 1)


@pytest.mark.parametrize("dim", [2, 3])
def test_queries_without_records_are_filtered_again(cuda, dim):
    """Windows over most of the points under a 1 MB budget: their items outnumber the batches that
    there is room for, so some queries are certainly written by the second filter."""
    rng = np.random.default_rng(dim)
    n, m, side = (250_000, 260, 1 << 20) if dim == 2 else (200_000, 180, 1 << 18)
    pts = rng.integers(0, side, size=(n, dim)).astype(np.int32)
    qs = rng.integers(side // 3, 2 * side // 3, size=(m, dim)).astype(np.int32)
    d = rng.integers(side // 2, side, m).astype(np.int32)
    d[::9] = rng.integers(0, 50, len(d[::9]))            # small ones between them
    if dim == 2:
        roff, rids = oracle.query(oracle.build(pts), qs, d, threads=8)
        idx = sfc.sfc_build(to_dev(pts, cuda), "z", mask_budget_mb=1)
    else:
        roff, rids = oracle.query3(oracle.build3(pts), qs, d)
        idx = sfc.sfc_build3(to_dev(pts, cuda), mask_budget_mb=1)
    _check(idx, qs, d, roff, rids, cuda)
    # an item covers at most 128 (3-D: 64) scanned points, a batch 32 items, and 1 MB holds a quarter
    # of its bytes, and an eighth and 64 more, in 28-byte batches
    most = ((1 << 20) // 4 // 28) * 9 // 8 + 64
    assert sfc.sfc_query_stats(idx)["scanned"] > (128 if dim == 2 else 64) * 32 * most
