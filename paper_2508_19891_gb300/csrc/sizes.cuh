// Sizes and positions that the host and the device compute alike.  Plain C++ without CUDA headers,
// so that a host compiler can build it too.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define SFC_HD __host__ __device__ __forceinline__
#else
#define SFC_HD inline
#endif

namespace sfc {

// Tiles of `per` elements that n elements make.  In 64 bits: n + per - 1 passes 2^32 for the largest
// arrays that a sort takes (n < 2^32 - 1).
SFC_HD uint32_t tiles_of(uint64_t n, uint32_t per) { return (uint32_t)((n + per - 1) / per); }

// Position of sample number i of `samples` among n elements (n < 2^32; a multiple of 32 samples): each 32
// consecutive samples fall into one of samples / 32 equal parts of the array, anywhere in it, by a fixed
// hash of i (the finaliser of SplitMix64, Steele, Lea & Flood 2014).  Two samples of a part meet in a
// run as often as two of its keys do, whatever the order of the input.  (At positions n i / S two
// samples of sorted input share a run only if it is n / S long, and input that interleaves kinds of
// points with a period of n / S shows one kind alone: 10^7 mixed points given in curve order were built
// in 827 us, 518 now as when shuffled; 2^24 keys of which every second lies in one dense part were
// sorted in 8.7 ms, 1.0 now.)  A part is what a warp loads at once: 16,384 samples of 6.4*10^6 points
// scattered over the whole array took 5 us longer, for their address translations.
SFC_HD uint64_t sample_position(uint32_t i, uint32_t samples, uint64_t n)
{
    uint64_t z = (i + 1ull) * 0x9e3779b97f4a7c15ull;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    const uint64_t parts = samples / 32, part = i / 32, first = n * part / parts;
    return first + ((((z ^ (z >> 31)) >> 32) * (n * (part + 1) / parts - first)) >> 32);
}

// Buffers of the hits of a query batch: per-batch heads and hit counts, and records.
struct HitSizes {
    uint64_t batches, records;
};
constexpr uint64_t kHitBatchBytes = 28, kHitRecordBytes = 8;
constexpr uint32_t kSlab = 512;   // records that a warp reserves at a time from a large buffer

// Records from which on an eighth of the buffer covers every warp's slab.
SFC_HD uint64_t large_records(uint64_t warps) { return warps * kSlab * 8; }

// Records that a warp reserves at a time: one batch's most (per_batch) where the buffer is small or has
// that many for every batch there can be, so that none goes without; else kSlab.
SFC_HD uint32_t slab_records(uint64_t records, uint64_t most_batches, uint64_t per_batch, uint64_t warps)
{
    return records < large_records(warps) || records / per_batch >= most_batches ? (uint32_t)per_batch : kSlab;
}

// Sizes within `bytes`, a quarter of them for the batches: at most what most_batches (the most that the
// batch can have) can use.  (One lookup over 10^8 points: 26 MB; 2^23 records on top of what it can
// use made that 117 MB.)
SFC_HD HitSizes hit_sizes(uint64_t bytes, uint64_t most_batches, uint64_t per_batch, uint64_t warps)
{
    HitSizes s;
    s.batches = bytes / 4 / kHitBatchBytes;
    if (s.batches > most_batches) s.batches = most_batches;
    uint64_t most = most_batches * per_batch;   // one batch a slab
    if (most >= large_records(warps)) most = 2 * most + warps * kSlab;   // slabs with unused ends
    s.records = bytes / 4 * 3 / kHitRecordBytes;
    if (s.records > most) s.records = most;
    return s;
}

}  // namespace sfc
