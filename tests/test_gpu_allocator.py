"""The caller's allocator (sfc_allocator) owns all of an index's device memory: with
PyTorch's caching allocator routed through the callbacks, every buffer of the index comes from
them (the library's own pool does not grow), torch counts the memory, results equal those of
an index on the library's pool and the oracle, and destroying the index hands every block back."""
import gc

import numpy as np
import pytest
import torch

import oracle
import paper_2508_19891_gb300 as sfc
import workloads as W
from conftest import to_dev, u32, u64

pytestmark = pytest.mark.gpu


def _pool_settled():
    """The library's own pool bytes once earlier tests' unreferenced indexes are gone."""
    gc.collect()
    torch.cuda.synchronize()
    return sfc.sfc_pool_bytes_in_use()


@pytest.mark.parametrize("bounds,curve", [("learned", "z"), ("binary", "h")])
def test_torch_allocator_owns_every_index_buffer(cuda, bounds, curve):
    wl = W.mixed_1e7(scale=0.02)
    pts, q, d = to_dev(wl.points, cuda), to_dev(wl.queries, cuda), to_dev(wl.delta, cuda)
    A = sfc.TorchAllocator(cuda)
    pool0 = _pool_settled()
    torch0 = torch.cuda.memory_allocated(cuda)
    idx = sfc.sfc_build(pts, curve, bounds=bounds, cover_refine=-1, allocator=A)
    sfc.sfc_autotune(idx, q, d)
    off, ids = sfc.query(idx, q, d)
    # a dynamic round (update workspaces) and the host-buffer batch (staging buffers)
    rng = np.random.default_rng(5)
    dels = torch.from_numpy(rng.choice(wl.n, 1000, replace=False).astype(np.int32)).to(cuda)
    ins = pts[:2000].clone()
    sfc.sfc_update(idx, ins, dels)
    sfc.sfc_query_batch_host(idx, wl.queries, wl.delta, int(off[-1].item()) * 2)
    assert _pool_settled() <= pool0              # nothing from the library's own pool
    assert A.allocs > 0 and A.live
    keys, iids, xy = sfc.sfc_get_sorted(idx, copy=False)
    n = keys.numel()
    assert A.owns(keys.data_ptr(), 8 * n) and A.owns(iids.data_ptr(), 4 * n) and A.owns(xy.data_ptr(), 8 * n)
    held = sum(A.live.values())
    assert torch.cuda.memory_allocated(cuda) - torch0 >= held   # torch accounts for the index
    # same answers as an index on the library's pool, and as the oracle
    ref = sfc.sfc_build(pts, curve, bounds=bounds, cover_refine=-1)
    sfc.sfc_autotune(ref, q, d)
    sfc.sfc_update(ref, ins, dels)
    off_a, ids_a = sfc.query(idx, q, d)
    off_r, ids_r = sfc.query(ref, q, d)
    assert torch.equal(off_a, off_r) and torch.equal(ids_a, ids_r)
    ref.close()
    first = wl.n
    alive = np.ones(wl.n + ins.shape[0], bool)
    alive[dels.cpu().numpy()] = False
    allpts = np.concatenate([wl.points, ins.cpu().numpy()])
    live = np.nonzero(alive)[0]
    boff, bids = oracle.brute(allpts[live], wl.queries[:200], wl.delta[:200])
    o, out = u64(off_a), u32(ids_a)
    for j in range(200):
        assert np.array_equal(np.sort(out[o[j]:o[j + 1]]), live[bids[boff[j]:boff[j + 1]]].astype(np.uint32)), j
    assert first == wl.n
    assert sfc.sfc_device_status(idx) == (0, 0)
    idx.close()
    torch.cuda.synchronize()
    assert not A.live and A.frees == A.allocs    # every block handed back
    assert _pool_settled() <= pool0


def test_torch_allocator_graph_and_3d(cuda):
    """A CUDA graph over an allocator-backed index (its buffers are reserved through the
    callbacks before capture) and a 3-D index built from host points."""
    wl = W.roads_3e7(scale=0.003)
    pts, q, d = to_dev(wl.points, cuda), to_dev(wl.queries, cuda), to_dev(wl.delta, cuda)
    A = sfc.TorchAllocator(cuda)
    pool0 = _pool_settled()
    idx = sfc.sfc_build(pts, "h", bounds="learned", allocator=A)
    off, ids = sfc.query(idx, q, d)
    goff = torch.zeros_like(off)
    gids = torch.zeros_like(ids)
    g = sfc.sfc_graph_capture(idx, pts, q, d, goff, gids)
    g.launch()
    torch.cuda.synchronize()
    assert torch.equal(goff, off) and torch.equal(gids, ids)
    g.close()
    idx.close()
    w3 = W.mixed3d(scale=0.002)
    i3 = sfc.sfc_build3_host(w3.points, allocator=A)
    o3, d3 = sfc.query(i3, to_dev(w3.queries, cuda), to_dev(w3.delta, cuda))
    roff, rids = oracle.query3(oracle.build3(w3.points), w3.queries, w3.delta)
    assert np.array_equal(u64(o3), roff) and np.array_equal(u32(d3), rids)
    i3.close()
    torch.cuda.synchronize()
    assert _pool_settled() <= pool0 and not A.live and A.frees == A.allocs


def test_allocator_out_of_memory_is_reported(cuda):
    """An allocator that has no memory makes the build fail with SFC_ERR_OOM, cleanly."""
    A = sfc.TorchAllocator(cuda)
    budget = {"left": 4}

    def stingy(nbytes, stream, ctx):
        if budget["left"] == 0:
            return None
        budget["left"] -= 1
        p = torch.cuda.caching_allocator_alloc(int(nbytes), cuda.index, int(stream or 0))
        A.live[int(p)] = int(nbytes)
        A.allocs += 1
        return int(p)

    A._alloc = sfc.SFC_ALLOC_FN(stingy)
    A.struct = sfc.sfc_allocator(A._alloc, A._free, None)
    pts = to_dev(W.uniform_1e5(scale=0.1).points, cuda)
    with pytest.raises(sfc.SfcError) as e:
        sfc.sfc_build(pts, "z", allocator=A)
    assert e.value.status == sfc.SFC_ERR_OOM
    torch.cuda.synchronize()
    assert not A.live and A.frees == A.allocs


def test_capture_after_a_batch_over_more_points_allocates_nothing(cuda):
    """An earlier batch over many points leaves room for more item batches than a smaller rebuild
    with more queries asks for: sfc_reserve sizes the rest of the workspace for that room, so the
    captured calls run no allocator callback, and replays are right."""
    gen = torch.Generator(device=cuda)
    gen.manual_seed(4)
    big = torch.randint(0, 1 << 30, (80_000_000, 2), generator=gen, device=cuda, dtype=torch.int32)
    n, m = 1_000_000, 290_000
    pts, q = big[:n].clone(), big[-m:].clone()
    d = torch.full((m,), 1 << 20, dtype=torch.int32, device=cuda)
    A = sfc.TorchAllocator(cuda)
    idx = sfc.sfc_build(big, "z", allocator=A)
    sfc.query(idx, q[:1000].contiguous(), d[:1000].contiguous())
    ref = sfc.sfc_build(pts, "z")
    want_off, want_ids = sfc.query(ref, q, d)
    off, ids = torch.zeros_like(want_off), torch.zeros_like(want_ids)
    sfc.sfc_reserve(idx, n, m)
    allocs, frees = A.allocs, A.frees
    g = sfc.sfc_graph_capture(idx, pts, q, d, off, ids)
    assert (A.allocs, A.frees) == (allocs, frees)
    for _ in range(2):
        off.zero_()
        ids.zero_()
        g.launch()
        torch.cuda.synchronize()
        assert torch.equal(off, want_off) and torch.equal(ids, want_ids)
    assert (A.allocs, A.frees) == (allocs, frees) and sfc.sfc_device_status(idx) == (0, 0)
    g.close()
    idx.close()


def test_reserved_batches_allocate_nothing_after_the_points_grow(cuda):
    """sfc_reserve_queries(m) holds after updates that grow the arrays and after a rebuild within
    them: batches of m queries run no allocator callback, eagerly and under a capture of the
    caller's own, and a capture made before such a rebuild stays valid."""
    rng = np.random.default_rng(6)
    pts = rng.integers(0, 1 << 16, size=(30_000, 2)).astype(np.int32)
    m = 500
    q, d = pts[:m].copy(), np.full(m, 900, np.int32)
    dq, dd = to_dev(q, cuda), to_dev(d, cuda)
    A = sfc.TorchAllocator(cuda)
    idx = sfc.sfc_build(to_dev(pts, cuda), "z", allocator=A)
    sfc.sfc_reserve_queries(idx, m)
    off = torch.zeros(m + 1, dtype=torch.int64, device=cuda)
    ids = torch.zeros(4_000_000, dtype=torch.int32, device=cuda)

    def check(points):
        roff, rids = oracle.query(oracle.build(points), q, d)
        assert np.array_equal(u64(off), roff) and np.array_equal(u32(ids[: len(rids)]), rids)

    for grown in (30_000, 200_000):
        ins = rng.integers(0, 1 << 16, size=(grown, 2)).astype(np.int32)
        sfc.sfc_update(idx, to_dev(ins, cuda), None)
        pts = np.concatenate([pts, ins])
        before = (A.allocs, A.frees)
        sfc.sfc_query_batch(idx, dq, dd, off, ids)
        check(pts)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            sfc.sfc_query_batch(idx, dq, dd, off, ids)
        assert (A.allocs, A.frees) == before
        off.zero_()
        ids.zero_()
        graph.replay()
        torch.cuda.synchronize()
        check(pts)
    sfc.sfc_rebuild(idx, to_dev(pts, cuda))              # the sort's own buffers
    before = (A.allocs, A.frees)
    sfc.sfc_rebuild(idx, to_dev(pts[:1000], cuda))
    sfc.sfc_query_batch(idx, dq, dd, off, ids)
    check(pts[:1000])
    sfc.sfc_rebuild(idx, to_dev(pts, cuda))
    sfc.sfc_query_batch(idx, dq, dd, off, ids)
    assert (A.allocs, A.frees) == before
    off.zero_()
    ids.zero_()
    graph.replay()
    torch.cuda.synchronize()
    check(pts)
    assert sfc.sfc_device_status(idx) == (0, 0)
    idx.close()


@pytest.mark.parametrize("dim", [2, 3])
def test_queries_fit_where_the_allocator_has_little_room(cuda, dim):
    """An allocator that has no room for a buffer of hits that grows with the points still serves a
    batch of wide windows (what finds no room is filtered again), and is not asked over and over."""
    rng = np.random.default_rng(dim)
    n, m, side = 1_000_000, 64, 1 << (30 if dim == 2 else 21)
    pts = rng.integers(0, side, size=(n, dim)).astype(np.int32)
    q = rng.integers(0, side, size=(m, dim)).astype(np.int32)
    d = rng.integers(0, side // 3, m).astype(np.int32)
    roff, rids = oracle.query(oracle.build(pts), q, d, threads=8) if dim == 2 else oracle.query3(oracle.build3(pts), q, d)
    A = sfc.TorchAllocator(cuda)
    roomy, state, refused = A._alloc, {"tight": False}, []

    def alloc(nbytes, stream, ctx):
        if state["tight"] and nbytes > 2 << 20:
            refused.append(int(nbytes))
            return None
        return roomy(nbytes, stream, ctx)

    A._alloc = sfc.SFC_ALLOC_FN(alloc)
    A.struct = sfc.sfc_allocator(A._alloc, A._free, None)
    idx = (sfc.sfc_build if dim == 2 else sfc.sfc_build3)(to_dev(pts, cuda), allocator=A)
    state["tight"] = True
    for _ in range(3):
        off, ids = sfc.query(idx, to_dev(q, cuda), to_dev(d, cuda))
        assert np.array_equal(u64(off), roff) and np.array_equal(u32(ids), rids)
    assert len(refused) == 1 and sfc.sfc_device_status(idx) == (0, 0)
    state["tight"] = False
    sfc.sfc_reserve_queries(idx, m)                      # asks again
    off, ids = sfc.query(idx, to_dev(q, cuda), to_dev(d, cuda))
    assert np.array_equal(u64(off), roff) and np.array_equal(u32(ids), rids)
    idx.close()
    torch.cuda.synchronize()
    assert not A.live


@pytest.mark.parametrize("dim,options", [(2, {}), (2, {"bounds": "learned", "occupancy_depth": 5}), (3, {})])
def test_rebuild_without_memory_leaves_an_empty_index(cuda, dim, options):
    """A rebuild that finds no memory, at whichever of its requests, returns SFC_ERR_OOM and leaves an
    empty index that answers queries and takes the next rebuild."""
    rng = np.random.default_rng(13)
    pts = rng.integers(0, 1 << 14, size=(40_000, dim)).astype(np.int32)
    q, d = to_dev(pts[:100], cuda), torch.full((100,), 300, dtype=torch.int32, device=cuda)
    A = sfc.TorchAllocator(cuda)
    roomy, left = A._alloc, [1 << 30]

    def alloc(nbytes, stream, ctx):
        left[0] -= 1
        return None if left[0] < 0 else roomy(nbytes, stream, ctx)

    A._alloc = sfc.SFC_ALLOC_FN(alloc)
    A.struct = sfc.sfc_allocator(A._alloc, A._free, None)
    idx = (sfc.sfc_build if dim == 2 else sfc.sfc_build3)(to_dev(pts[:2000], cuda), allocator=A, **options)
    failed = 0
    while True:
        left[0] = min(failed, 1)                         # one more request succeeds each time
        try:
            sfc.sfc_rebuild(idx, to_dev(pts, cuda))
            break
        except sfc.SfcError as e:
            assert e.status == sfc.SFC_ERR_OOM
            failed += 1
        finally:
            left[0] = 1 << 30
        off, ids = sfc.query(idx, q, d)
        assert not off.any().item() and ids.numel() == 0 and sfc.sfc_get_sorted(idx)[0].numel() == 0
    assert failed > 3
    off, ids = sfc.query(idx, q, d)
    ref = oracle.build(pts) if dim == 2 else oracle.build3(pts)
    roff, rids = (oracle.query if dim == 2 else oracle.query3)(ref, pts[:100], np.full(100, 300, np.int32))
    assert np.array_equal(u64(off), roff) and np.array_equal(u32(ids), rids)
    assert sfc.sfc_device_status(idx) == (0, 0)
    idx.close()
    torch.cuda.synchronize()
    assert not A.live


def test_reserve_for_fewer_queries_keeps_what_was_reserved(cuda):
    """sfc_reserve for many points and few queries, after batches of many queries: rebuilds within it
    and batches of either size allocate nothing."""
    rng = np.random.default_rng(8)
    pts = rng.integers(0, 1 << 16, size=(300_000, 2)).astype(np.int32)
    q, d = to_dev(pts[:5000], cuda), torch.full((5000,), 300, dtype=torch.int32, device=cuda)
    A = sfc.TorchAllocator(cuda)
    idx = sfc.sfc_build(to_dev(pts[:20_000], cuda), "z", allocator=A)
    sfc.query(idx, q, d)
    sfc.sfc_reserve(idx, len(pts), 10)
    before = (A.allocs, A.frees)
    sfc.sfc_rebuild(idx, to_dev(pts, cuda))
    for m in (10, 5000):
        off, ids = sfc.query(idx, q[:m].contiguous(), d[:m].contiguous())
        roff, rids = oracle.query(oracle.build(pts), pts[:m], np.full(m, 300, np.int32))
        assert np.array_equal(u64(off), roff) and np.array_equal(u32(ids), rids)
    assert (A.allocs, A.frees) == before and sfc.sfc_device_status(idx) == (0, 0)
    idx.close()
