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

}  // namespace sfc
