// Dynamic setting (Sec. 2.1 "Dynamic implementation"; Sec. 3.3), batched.
//
// The paper keeps (pi(p), p) in a B-tree multimap and applies one element at a time.  Here a
// whole batch is applied to the sorted arrays at once; the result is exactly the array a
// rebuild from scratch over the live points would produce, because the order is (key, id)
// and every inserted id is larger than every existing one:
//
//   del_locate_kernel  each delete must be an issued, live id; its array position (lexicographic
//                      lower_bound of (key, id), the key from the id -> key table) goes into a
//                      bitmap, where a repeated id meets its own bit, and into the deletes' count
//                      per tile
//   (host)             one synchronisation: a bad batch is rejected before anything changes
//   scan               deletes before each tile
//   radix sort         inserts by key with ids next_id + i (keys computed from the points)
//   ins_rank_kernel    rank of each insert among the old entries: upper_bound of its key
//   tile_starts_kernel inserts ranked before each tile
//   move_kernel        surviving entry p to slot p - (deletes before p) + (inserts ranked <= p),
//                      counted tile by tile in shared memory
//   ins_place_kernel   insert j to slot r_j - (deletes before r_j, from the bitmap) + j
//   then: liveness bits, boxes and directory, and a refit of a trained model.
#include <algorithm>

#include "sfc_internal.cuh"
#include "index.cuh"

namespace sfc {

namespace {

constexpr int kT = 256;

int grid_of(uint64_t n)
{
    uint64_t g = (n + kT - 1) / kT;
    const uint64_t cap = (uint64_t)num_sms() * 16;
    return (int)std::max<uint64_t>(1, std::min(g, cap));
}

// Part of the sorted array that holds the keys equal to kk, from the key directory (boxes.cu): those
// before [lo, hi) are smaller, those from hi on larger.
__device__ __forceinline__ void key_part(const uint64_t* __restrict__ keys, uint32_t n, const uint32_t* __restrict__ dir,
                                         int bits, uint64_t kk, uint32_t& lo, uint32_t& hi)
{
    lo = hi = 0;
    if (n == 0) return;
    const uint64_t kmin = __ldg(keys), kmax = __ldg(keys + n - 1);
    if (kk < kmin) return;
    lo = hi = n;
    if (kk > kmax) return;
    const uint32_t v = (uint32_t)((kk - kmin) >> dir_shift(kmin, kmax, bits));
    lo = __ldg(dir + v);
    hi = __ldg(dir + v + 1);
}

// Old entries per tile of move_kernel: eight per thread.
constexpr int kMoveItems = 8;
constexpr int kMoveTile = kT * kMoveItems;
constexpr uint32_t kGone = 0xffffffffu;   // no slot is this large (n < 2^32 - 1)

// Checks and locates the deletes: position of (key, id) in the array sorted by (key, id), a bit per
// position and a count per tile.  In the order they are given: sorting them first, for searches over
// neighbouring lines and ascending positions, took longer than it saved (5*10^5 deletes at 5*10^7
// points: the update 636 us sorted, 592 not).
__global__ void del_locate_kernel(const uint64_t* __restrict__ keys, const uint32_t* __restrict__ ids, uint32_t n,
                                  const uint32_t* __restrict__ dir, int bits, const uint32_t* __restrict__ del, uint64_t k,
                                  const uint64_t* __restrict__ key_by_id, const uint32_t* __restrict__ alive,
                                  uint32_t next_id, uint32_t* dbits, uint32_t* dcount, uint32_t* bad)
{
    chain_start();
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < k; t += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t id = del[t];
        if (id >= next_id || !((alive[id >> 5] >> (id & 31)) & 1u)) {
            atomicOr(bad, 1u);
            continue;
        }
        const uint64_t kk = __ldg(key_by_id + id);
        uint32_t lo, hi;
        key_part(keys, n, dir, bits, kk, lo, hi);
        uint32_t len = hi - lo;
        while (len > 0) {
            const uint32_t half = len >> 1;
            const uint32_t mid = lo + half;
            const uint64_t km = __ldg(keys + mid);
            const bool less = km < kk || (km == kk && ids[mid] < id);
            lo = less ? mid + 1 : lo;
            len = less ? len - half - 1 : half;
        }
        bool ok = lo < n && keys[lo] == kk && ids[lo] == id;
        if (ok) ok = !((atomicOr(dbits + (lo >> 5), 1u << (lo & 31)) >> (lo & 31)) & 1u);   // a repeated id
        if (ok) atomicAdd(dcount + lo / kMoveTile, 1u);
        else atomicOr(bad, 1u);
    }
}

// Rank of each (sorted) insert among the old entries: all old ids are smaller, so it is the
// number of old keys <= the insert's key.
__global__ void ins_rank_kernel(const uint64_t* __restrict__ keys, uint32_t n, const uint32_t* __restrict__ dir, int bits,
                                const uint64_t* ikeys, uint64_t k, uint32_t* rank)
{
    chain_start();
    ikeys = after_wait(ikeys);
    for (uint64_t j = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; j < k; j += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t kk = ikeys[j];
        uint32_t lo, hi;
        key_part(keys, n, dir, bits, kk, lo, hi);
        uint32_t len = hi - lo;
        while (len > 0) {
            const uint32_t half = len >> 1;
            const bool le = keys[lo + half] <= kk;
            lo = le ? lo + half + 1 : lo;
            len = le ? len - half - 1 : half;
        }
        rank[j] = lo;
    }
}

// starts[t] = how many of the ascending pos[0 .. k) lie before tile t, t = 0 .. tiles.  The
// thread of pos[j] fills the tiles that begin after pos[j - 1] and not after pos[j] (j == k: the
// rest).  A position may be n (an insert after every entry).
__global__ void tile_starts_kernel(const uint32_t* pos, uint64_t k, uint32_t tiles, uint32_t* starts)
{
    chain_start();
    pos = after_wait(pos);
    for (uint64_t j = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; j <= k; j += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t t0 = j ? pos[j - 1] / kMoveTile + 1 : 0;
        const uint32_t t1 = j < k ? min(pos[j] / kMoveTile, tiles) : tiles;
        for (uint32_t t = t0; t <= t1; ++t) starts[t] = (uint32_t)j;
    }
}

// Moves a tile of old entries to their new slots.  Bound by HBM: it reads and writes each entry's
// 20 bytes once and nothing else per entry (a full-length deletion mask, shift counts and their
// scan took another 26 bytes per entry: 5*10^5 inserts and deletes at 5*10^7 points 1086 us
// before, 719 us after).  The entries are loaded before the tile's counts are scanned, so the loads
// overlap the shared-memory work.
__global__ void __launch_bounds__(kT) move_kernel(const uint64_t* __restrict__ keys, const uint32_t* __restrict__ ids,
                                                  const int2* __restrict__ xy, uint32_t n,
                                                  const uint32_t* __restrict__ dbits, const uint64_t* __restrict__ dstart,
                                                  const uint32_t* __restrict__ rank, const uint32_t* istart,
                                                  uint64_t* nkeys, uint32_t* nids, int2* nxy)
{
    chain_start();
    istart = after_wait(istart);
    __shared__ uint32_t s_ins[kMoveTile];   // inserts ranked at each entry, then its slot in the tile's output
    __shared__ uint32_t s_warp[kT / 32];
    const int tid = threadIdx.x;
    const uint32_t p0 = blockIdx.x * (uint32_t)kMoveTile;
    uint64_t key[kMoveItems];
    uint32_t id[kMoveItems];
    int2 c[kMoveItems];
#pragma unroll
    for (int i = 0; i < kMoveItems; ++i) {
        const uint32_t x = i * kT + tid;
        if (x < n - p0) {
            key[i] = __ldcs(keys + p0 + x);
            id[i] = __ldcs(ids + p0 + x);
            c[i] = __ldcs(xy + p0 + x);
        }
        s_ins[x] = 0;
    }
    const uint32_t d0 = dbits ? (uint32_t)dstart[blockIdx.x] : 0;
    const uint32_t i0 = rank ? istart[blockIdx.x] : 0, i1 = rank ? istart[blockIdx.x + 1] : 0;
    __syncthreads();
    for (uint32_t j = i0 + tid; j < i1; j += kT)
        atomicAdd(&s_ins[rank[j] - p0], 1u);
    __syncthreads();
    // this thread's stretch of eight entries, the eight bits of its deletions
    const uint32_t at = p0 + tid * kMoveItems;
    const uint32_t gone = dbits && at < n ? (dbits[at >> 5] >> (at & 31)) & 0xffu : 0u;
    uint32_t run[kMoveItems], sum = 0;
#pragma unroll
    for (int i = 0; i < kMoveItems; ++i) {
        const uint32_t v = s_ins[tid * kMoveItems + i];
        run[i] = sum + v;                // an entry comes after the inserts ranked at it
        sum += v + 1u - ((gone >> i) & 1u);
    }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if ((int)lane_id() >= o) incl += t;
    }
    if (lane_id() == 31) s_warp[tid >> 5] = incl;
    __syncthreads();
    uint32_t base = incl - sum;
#pragma unroll
    for (int w = 0; w < kT / 32; ++w) base += w < (tid >> 5) ? s_warp[w] : 0u;
#pragma unroll
    for (int i = 0; i < kMoveItems; ++i)
        s_ins[tid * kMoveItems + i] = (gone >> i) & 1u ? kGone : base + run[i];
    __syncthreads();
    const uint32_t first = p0 - d0 + i0;   // slot of the tile's first output
#pragma unroll
    for (int i = 0; i < kMoveItems; ++i) {
        const uint32_t x = i * kT + tid;
        if (x >= n - p0 || s_ins[x] == kGone) continue;
        const uint32_t dst = first + s_ins[x];
        nkeys[dst] = key[i];
        nids[dst] = id[i];
        nxy[dst] = c[i];
    }
}

__global__ void ins_place_kernel(const uint64_t* __restrict__ ikeys, const uint32_t* __restrict__ iids,
                                 const int2* __restrict__ ixy, uint64_t k, const uint32_t* __restrict__ rank,
                                 const uint32_t* __restrict__ dbits, const uint64_t* __restrict__ dstart, uint64_t* nkeys,
                                 uint32_t* nids, int2* nxy)
{
    chain_start();
    for (uint64_t j = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; j < k; j += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t r = rank[j];
        // deletes at positions < r: those before r's tile, then the tile's bits up to r
        uint32_t before = 0;
        if (dbits) {
            const uint32_t tile = r / kMoveTile;
            before = (uint32_t)dstart[tile];
            uint32_t w = tile * (kMoveTile / 32);
            for (; w + 4 <= r >> 5; w += 4) {
                const uint4 x = __ldg(reinterpret_cast<const uint4*>(dbits + w));
                before += __popc(x.x) + __popc(x.y) + __popc(x.z) + __popc(x.w);
            }
            for (; w < r >> 5; ++w) before += __popc(dbits[w]);
            before += __popc(dbits[w] & ((1u << (r & 31)) - 1u));
        }
        const uint64_t dst = (uint64_t)r - before + j;
        nkeys[dst] = ikeys[j];
        nids[dst] = iids[j];
        nxy[dst] = ixy[j];
    }
}

__global__ void alive_clear_kernel(const uint32_t* __restrict__ del, uint64_t k, uint32_t* alive)
{
    chain_start();
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < k; t += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t id = del[t];
        atomicAnd(alive + (id >> 5), ~(1u << (id & 31)));
    }
}

}  // namespace

sfc_status ensure_alive_bits(sfc_index* idx, uint64_t ids, cudaStream_t st)
{
    // ids >= next_id are never treated as live (checks compare against next_id first), so
    // new words can start all-ones: an inserted id is live as soon as next_id passes it.
    const uint64_t words = (ids + 31) / 32 + 1;
    if (words * 4 <= idx->alive.bytes) return SFC_OK;
    DevBuf nb;
    SFC_TRY(nb.ensure(words * 4, st));
    SFC_CUDA_TRY(cudaMemsetAsync(nb.ptr, 0xff, nb.bytes, st));
    if (idx->alive.ptr)
        SFC_CUDA_TRY(cudaMemcpyAsync(nb.ptr, idx->alive.ptr, idx->alive.bytes, cudaMemcpyDeviceToDevice, st));
    idx->alive.release(st);
    idx->alive = nb;
    return SFC_OK;
}

void release_index(sfc_index* idx, cudaStream_t st)
{
    idx->keys.release(st);
    idx->ids.release(st);
    idx->xy.release(st);
    idx->key_by_id.release(st);
    idx->alive.release(st);
    idx->status.release(st);
    idx->occ.release(st);
    idx->box.release(st);
    idx->dir.release(st);
    idx->xyz.release(st);
    idx->packed.release(st);
    idx->keys_in.release(st);
    release_sort_ws(idx->sort_ws, st);
    idx->scan_ws.flags.release(st);
    QueryWs& q = idx->qws;
    for (DevBuf* d : {&q.ranges, &q.qrec, &q.nitems, &q.gbase, &q.ovf, &q.counts, &q.ctr, &q.heads, &q.bhits, &q.bbase,
                      &q.recs, &q.flags, &q.qkeys, &q.qkeys_sorted, &q.perm, &q.pstart, &q.dbase})
        d->release(st);
    HostStage& h = idx->stage;
    h.q.release(st); h.delta.release(st); h.offsets.release(st); h.ids.release(st);
    h.points.release(st);
    if (h.copy) {
        cudaStreamSynchronize(h.copy);
        cudaStreamDestroy(h.copy);
        h.copy = nullptr;
        for (auto& e : h.done) {
            if (e) cudaEventDestroy(e);
            e = nullptr;
        }
    }
    ModelState& M = idx->model;
    M.state.release(st); M.samples.release(st); M.partial.release(st);
    M.tmp.release(st); M.leaves.release(st); M.fence.release(st);
    M.fence_fine.release(st);
    UpdateWs& u = idx->uws;
    u.a.release(st);
    u.e.release(st); u.f.release(st); u.g.release(st); u.h.release(st);
    u.keys.release(st); u.ids.release(st); u.xy.release(st);
    u.marks.release(st); u.dstart.release(st); u.istart.release(st);
}

sfc_status apply_update(sfc_index* idx, const int32_t* d_inserts, uint64_t k_ins, const uint32_t* d_del,
                        uint64_t k_del, uint32_t* h_first, cudaStream_t st)
{
    UpdateWs& U = idx->uws;
    const uint32_t n = (uint32_t)idx->n;
    const uint32_t next_id = idx->next_id;
    const int curve = idx->curve;
    if ((uint64_t)next_id + k_ins >= 0xffffffffull || (uint64_t)n + k_ins >= 0xffffffffull) return SFC_ERR_INVALID;
    uint32_t* status = idx->status.as<uint32_t>();
    // scratch: a = flags, e .. h = the sorted inserts and their ranks
    SFC_TRY(U.a.ensure(16, st));
    uint32_t* bad = U.a.as<uint32_t>();
    SFC_CUDA_TRY(cudaMemsetAsync(bad, 0, 16, st));
    uint32_t* dbits = nullptr;
    // tiles of old entries; the last one may be empty, it takes the inserts ranked after all of them
    const uint32_t tiles = n / kMoveTile + 1;
    if (k_del) {
        const size_t words = (size_t)tiles * (kMoveTile / 32);
        SFC_TRY(U.marks.ensure((words + tiles) * sizeof(uint32_t), st));
        SFC_TRY(U.dstart.ensure(((size_t)tiles + 1) * sizeof(uint64_t), st));
        dbits = U.marks.as<uint32_t>();
        uint32_t* dcount = dbits + words;
        SFC_CUDA_TRY(cudaMemsetAsync(dbits, 0, (words + tiles) * sizeof(uint32_t), st));
        launch_chain(del_locate_kernel, grid_of(k_del), kT, 0, st, idx->keys.as<uint64_t>(), idx->ids.as<uint32_t>(), n,
                     idx->dir.as<uint32_t>(), dir_bits(n), d_del, k_del, idx->key_by_id.as<uint64_t>(),
                     idx->alive.as<uint32_t>(), next_id, dbits, dcount, bad);
        count_launch();
        SFC_TRY(exclusive_scan_u32(dcount, tiles, U.dstart.as<uint64_t>(), idx->scan_ws, status, st));
        SFC_TRY(launch_status());
        uint32_t hbad = 0;
        SFC_CUDA_TRY(cudaMemcpyAsync(&hbad, bad, 4, cudaMemcpyDeviceToHost, st));
        SFC_CUDA_TRY(cudaStreamSynchronize(st));
        if (hbad) return SFC_ERR_NOT_FOUND;   // nothing has been changed yet
    }
    // ---- inserts: keys, sort, decoded coordinates ----
    const uint64_t new_n = (uint64_t)n - k_del + k_ins;
    const uint64_t ids_after = (uint64_t)next_id + k_ins;
    uint64_t* ikeys = nullptr;
    uint32_t* iids = nullptr;
    int2* ixy = nullptr;
    uint32_t* irank = nullptr;
    if (k_ins) {
        SFC_TRY(U.e.ensure(k_ins * 8, st));
        SFC_TRY(U.f.ensure(k_ins * 4, st));
        SFC_TRY(U.g.ensure(k_ins * 8, st));
        SFC_TRY(U.h.ensure(k_ins * 4, st));
        if (ids_after * sizeof(uint64_t) > idx->key_by_id.bytes)
            SFC_TRY(idx->key_by_id.grow(ids_after * sizeof(uint64_t) + ids_after * sizeof(uint64_t) / 2,
                                        (size_t)next_id * sizeof(uint64_t), st));
        ikeys = U.e.as<uint64_t>();
        iids = U.f.as<uint32_t>();
        ixy = U.g.as<int2>();
        irank = U.h.as<uint32_t>();
        SortSource src;
        // the id -> key table takes the inserts' keys from their sort (entries past next_id until the
        // batch is done mean nothing)
        src.keys_out = idx->key_by_id.as<uint64_t>() + next_id;
        src.points = reinterpret_cast<const int2*>(d_inserts);
        src.bits = 2 * kOmega;
        src.curve = curve;
        src.val_base = next_id;
        SortDest dst;
        dst.keys = ikeys;
        dst.vals = iids;
        dst.xy = ixy;
        dst.curve = curve;
        SFC_TRY(radix_sort(src, k_ins, dst, idx->sort_ws, status, st));
    }
    // ---- every other buffer that the batch needs (while the sort runs), before anything of the index
    // changes: a batch that finds no memory leaves it as it was; those that hold contents keep them ----
    SFC_TRY(U.keys.ensure(std::max<uint64_t>(new_n, 1) * 8, st));
    SFC_TRY(U.ids.ensure(std::max<uint64_t>(new_n, 1) * 4, st));
    SFC_TRY(U.xy.ensure(pad_groups(std::max<uint64_t>(new_n, 1)) * 8, st));
    SFC_TRY(U.istart.ensure(((size_t)tiles + 1) * sizeof(uint32_t), st));
    SFC_TRY(idx->box.grow(box_bytes(2, new_n), box_bytes(2, n), st));
    SFC_TRY(idx->dir.grow(dir_bytes(new_n), dir_bytes(n), st));
    if (k_ins) SFC_TRY(ensure_alive_bits(idx, ids_after, st));
    if (idx->model.trained) SFC_TRY(reserve_model(idx, new_n, st));
    // ---- shift counts and the new arrays ----
    uint32_t* istart = U.istart.as<uint32_t>();
    const uint64_t* keys = idx->keys.as<uint64_t>();
    const uint32_t* ids = idx->ids.as<uint32_t>();
    if (k_ins) {
        launch_chain(ins_rank_kernel, grid_of(k_ins), kT, 0, st, keys, n, idx->dir.as<uint32_t>(), dir_bits(n), ikeys, k_ins,
                     irank);
        launch_chain(tile_starts_kernel, grid_of(k_ins + 1), kT, 0, st, irank, k_ins, tiles, istart);
        count_launch(2);
    }
    SFC_TRY(launch_status());
    uint64_t* nkeys = U.keys.as<uint64_t>();
    uint32_t* nids = U.ids.as<uint32_t>();
    int2* nxy = U.xy.as<int2>();
    if (n) {
        launch_chain(move_kernel, tiles, kT, 0, st, keys, ids, idx->xy.as<int2>(), n, dbits, U.dstart.as<uint64_t>(), irank, istart,
                                          nkeys, nids, nxy);
        count_launch();
    }
    if (k_ins) {
        launch_chain(ins_place_kernel, grid_of(k_ins), kT, 0, st, ikeys, iids, ixy, k_ins, irank, dbits,
                     U.dstart.as<uint64_t>(), nkeys, nids, nxy);
        count_launch();
    }
    // ---- liveness ----
    if (k_del) {
        launch_chain(alive_clear_kernel, grid_of(k_del), kT, 0, st, d_del, k_del, idx->alive.as<uint32_t>());
        count_launch();
    }
    SFC_TRY(launch_status());
    // ---- swap in the new arrays ----
    std::swap(idx->keys, U.keys);
    std::swap(idx->ids, U.ids);
    std::swap(idx->xy, U.xy);
    idx->n = new_n;
    idx->next_id = next_id + (uint32_t)k_ins;
    if (h_first) *h_first = next_id;
    idx->qws.pending.valid = false;
    SFC_TRY(build_occupancy(idx, st));
    SFC_TRY(build_boxes(idx, st));
    follow_arrays(idx, st);
    if (idx->model.trained) {
        const int steps = std::max(20, idx->opt.train_steps / 5);
        SFC_TRY(refit_model(idx, steps, st));
    }
    return SFC_OK;
}

}  // namespace sfc

extern "C" sfc_status sfc_update(sfc_index* idx, const int32_t* d_inserts, uint64_t k_ins,
                                 const uint32_t* d_delete_ids, uint64_t k_del, uint32_t* h_first_new_id,
                                 void* stream)
{
    if (!idx || (k_ins && !d_inserts) || (k_del && !d_delete_ids) || idx->dim != 2) return SFC_ERR_INVALID;
    if (k_del > idx->n || k_ins >= 0xffffffffull) return k_del > idx->n ? SFC_ERR_NOT_FOUND : SFC_ERR_INVALID;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    idx->last_stream = st;
    sfc::AllocScope alloc_scope(idx->allocator());
    sfc::ProfScope ps(idx, "update", st);
    return sfc::apply_update(idx, d_inserts, k_ins, d_delete_ids, k_del, h_first_new_id, st);
}
