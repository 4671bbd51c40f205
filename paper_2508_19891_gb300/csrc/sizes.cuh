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

// Position of sample number i among n elements (n < 2^32): a fixed hash of i (the finaliser of
// SplitMix64, Steele, Lea & Flood 2014), scaled to n.  Every sample falls anywhere, independently of
// the others, so pairs of samples meet in a run as often as pairs of keys do whatever the order of
// the input.  (At positions n i / S two samples of sorted input share a run only if it is n / S long,
// and input that interleaves kinds of points with a period of n / S shows one kind alone.)
SFC_HD uint64_t sample_position(uint32_t i, uint64_t n)
{
    uint64_t z = (i + 1ull) * 0x9e3779b97f4a7c15ull;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return (((z ^ (z >> 31)) >> 32) * n) >> 32;
}

}  // namespace sfc
