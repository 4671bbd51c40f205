// Bounding boxes of the groups of 32 consecutive points of the sorted array: group g holds the
// array positions 32 g .. 32 g + 31.  Points that follow each other on the curve lie close
// together, so a group's box is small and most groups that a query's ranges touch are wholly
// outside or wholly inside its window (of the groups touched on mixed points with cover 1, 53%
// and 19%): the count pass then needs neither their points nor their tests.  Rebuilt with the
// sorted array, half a byte per point (one byte in 3-D).
//
// One pass over the coordinates, bound by HBM: a warp takes four groups at a time, one coalesced
// load each, and reduces them with the warp's min / max instructions (10^8 points: 0.15 ms, 5.7
// TB/s, 0.18 ms with the directory below, against the 7 ms that the count pass of 10^7 queries saves).
//
// The same launch fills the key directory that the bound searches of the plan start from: a thread
// finds each entry by binary search (neighbouring threads walk nearly the same path, so 2^18
// entries take a few microseconds beside the boxes).
#include <algorithm>

#include "sfc_internal.cuh"
#include "index.cuh"

namespace sfc {

namespace {

constexpr int kT = 256;
constexpr int kU = 4;   // groups per warp and iteration

// One step of the directory's search: the answer in [lo, lo + len] given the keys at lo + len / 4,
// lo + len / 2 and the place between that and the end.  The three are counted, not tested one after
// another, so that their loads are in flight together.
__device__ __forceinline__ void narrow(uint32_t& lo, uint32_t& len, uint64_t ka, uint64_t kb, uint64_t kc, uint64_t t)
{
    const uint32_t q = len >> 2, h = len >> 1, c = (uint32_t)(ka < t) + (kb < t) + (kc < t);
    const uint32_t from = c == 0 ? 0 : (c & 1 ? q : 0) + (c & 2 ? h : 0) + 1;
    const uint32_t to = c == 3 ? len : (c == 0 ? q : h + (c == 2 ? q : 0));
    lo += from;
    len = to - from;
}

// Entries [0, 2^bits] of the directory, by the blocks [0, blocks) of a launch.
__device__ __forceinline__ void fill_directory(const uint64_t* keys, uint32_t n, int bits, uint32_t blocks, uint32_t* dir)
{
    // the first step's probes are the same for every entry: loaded with the ends of the range
    const uint64_t kmin = keys[0], kmax = keys[n - 1];
    const uint64_t k1 = keys[n >> 2], k2 = keys[n >> 1], k3 = keys[(n >> 2) + (n >> 1)];
    const int shift = dir_shift(kmin, kmax, bits);
    for (uint32_t v = blockIdx.x * kT + threadIdx.x; v <= 1u << bits; v += blocks * kT) {
        const uint64_t t = kmin + ((uint64_t)v << shift);   // at most 2 kmax: 64 bits hold it
        // three probes a step: the latency of the steps, not the loads, sets the time of short arrays
        uint32_t lo = 0, len = n;   // the answer lies in [lo, lo + len]
        narrow(lo, len, k1, k2, k3, t);
        while (len > 0)
            narrow(lo, len, keys[lo + (len >> 2)], keys[lo + (len >> 1)], keys[lo + (len >> 1) + (len >> 2)], t);
        dir[v] = lo;
    }
}

// Blocks [0, dblocks) fill the directory, the others the boxes.
__global__ void __launch_bounds__(kT) boxes_kernel(const int2* xy, const uint64_t* keys, uint32_t n, uint32_t groups,
                                                   int bits, uint32_t dblocks, uint32_t* dir, int4* box)
{
    chain_start();
    xy = after_wait(xy);
    keys = after_wait(keys);
    if (blockIdx.x < dblocks) {
        fill_directory(keys, n, bits, dblocks, dir);
        return;
    }
    const unsigned lane = lane_id();
    const uint32_t warps = (gridDim.x - dblocks) * (kT / 32);
    for (uint32_t g0 = ((blockIdx.x - dblocks) * (kT / 32) + (threadIdx.x >> 5)) * kU; g0 < groups; g0 += warps * kU) {
        int2 p[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u)   // past the end the last point stands in: it changes no box
            p[u] = xy[min((uint64_t)(g0 + u) * 32 + lane, (uint64_t)n - 1)];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int4 b = make_int4(__reduce_min_sync(0xffffffffu, p[u].x), __reduce_min_sync(0xffffffffu, p[u].y),
                                     __reduce_max_sync(0xffffffffu, p[u].x), __reduce_max_sync(0xffffffffu, p[u].y));
            if (lane == u && g0 + u < groups) box[g0 + u] = b;
        }
    }
}

// 3-D: decodes the sorted keys into the 16-byte records and the packed coordinates on the way (a
// decoding kernel of its own and boxes read back from its records: 78 us more at 10^7 points).
__global__ void __launch_bounds__(kT) boxes3_kernel(const uint64_t* keys, uint32_t n, uint32_t groups, int bits,
                                                    uint32_t dblocks, uint32_t* dir, int4* xyz, uint2* packed, int4* box)
{
    chain_start();
    keys = after_wait(keys);
    if (blockIdx.x < dblocks) {
        fill_directory(keys, n, bits, dblocks, dir);
        return;
    }
    const unsigned lane = lane_id();
    const uint32_t warps = (gridDim.x - dblocks) * (kT / 32);
    for (uint32_t g0 = ((blockIdx.x - dblocks) * (kT / 32) + (threadIdx.x >> 5)) * kU; g0 < groups; g0 += warps * kU) {
        uint64_t k[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u)
            k[u] = keys[min((uint64_t)(g0 + u) * 32 + lane, (uint64_t)n - 1)];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const uint64_t i = (uint64_t)(g0 + u) * 32 + lane;
            const uint32_t x = gather3_bits(k[u]), y = gather3_bits(k[u] >> 1), z = gather3_bits(k[u] >> 2);
            if (i < n) {
                xyz[i] = make_int4((int)x, (int)y, (int)z, 0);
                packed[i] = pack3(x, y, z);
            }
            const int4 lo = make_int4((int)__reduce_min_sync(0xffffffffu, x), (int)__reduce_min_sync(0xffffffffu, y),
                                      (int)__reduce_min_sync(0xffffffffu, z), 0);
            const int4 hi = make_int4((int)__reduce_max_sync(0xffffffffu, x), (int)__reduce_max_sync(0xffffffffu, y),
                                      (int)__reduce_max_sync(0xffffffffu, z), 0);
            if (lane < 2 && g0 + u < groups) box[2 * (uint64_t)(g0 + u) + lane] = lane ? hi : lo;
        }
    }
}

}  // namespace

// Padded to whole items (four groups): a lane loads its item's boxes together.
size_t box_bytes(int dim, uint64_t n) { return (n + 127) / 128 * 4 * (dim == 3 ? 2 : 1) * sizeof(int4); }

size_t dir_bytes(uint64_t n) { return ((size_t)(1u << dir_bits(n)) + 1) * sizeof(uint32_t); }

sfc_status build_boxes(sfc_index* idx, cudaStream_t st)
{
    const uint64_t n = idx->n;
    if (n == 0) return SFC_OK;
    SFC_TRY(idx->box.ensure(box_bytes(idx->dim, n), st));
    SFC_TRY(idx->dir.ensure(dir_bytes(n), st));
    const uint32_t groups = (uint32_t)((n + 31) / 32);
    const uint32_t per_block = (kT / 32) * kU;
    const int bits = dir_bits(n);
    // of the eight blocks that an SM holds, two fill the directory beside six that stream a large
    // array (the directory's latency then hides behind the boxes); short arrays take what it needs
    const bool large = n >= 1ull << 24;
    const uint32_t dblocks = std::min((1u << bits) / kT + 1, (uint32_t)num_sms() * (large ? 2 : 4));
    const uint32_t grid = dblocks + std::min((groups + per_block - 1) / per_block, (uint32_t)num_sms() * (large ? 6 : 8));
    if (idx->dim == 3)
        launch_chain(boxes3_kernel, grid, kT, 0, st, idx->keys.as<uint64_t>(), (uint32_t)n, groups, bits, dblocks,
                     idx->dir.as<uint32_t>(), idx->xyz.as<int4>(), idx->packed.as<uint2>(), idx->box.as<int4>());
    else
        launch_chain(boxes_kernel, grid, kT, 0, st, idx->xy.as<int2>(), idx->keys.as<uint64_t>(), (uint32_t)n, groups, bits, dblocks,
                                          idx->dir.as<uint32_t>(), idx->box.as<int4>());
    count_launch();
    return launch_status();
}

}  // namespace sfc
