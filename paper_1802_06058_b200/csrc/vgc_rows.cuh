// Which row of a plane a position lies in (plain C++ on the host): p / width with one multiplication, for every plane that 32-bit
// positions can address.
#pragma once

#include <cstdint>

#ifndef __CUDACC__
#define __host__
#define __device__
#define __forceinline__ inline
#endif

namespace vgc {

// magic = ceil(2^(31 + l) / width), l = ceil(log2 width): magic * width - 2^(31 + l) lies in [0, width), so at most 2^l, and
// p * magic >> (31 + l) is p / width for all p < 2^31 (Granlund, Montgomery: Division by invariant integers using
// multiplication, theorem 4.2 with 31-bit numerators).  A magic number of 2^32 / width without the shift is exact for
// p * width < 2^32 only: 1024 positions of a 4096 x 4096 plane were given the wrong row.
struct RowDivisor {
    uint32_t magic;
    int shift;               // l - 1
};

// width >= 2
inline RowDivisor row_divisor(uint32_t width)
{
    int l = 1;
    while ((1ull << l) < width) ++l;
    return RowDivisor{(uint32_t)(((1ull << (31 + l)) + width - 1) / width), l - 1};
}

// p < 2^31
__host__ __device__ __forceinline__ uint32_t row_of(uint32_t p, uint32_t magic, int shift)
{
#ifdef __CUDA_ARCH__
    return __umulhi(p, magic) >> shift;
#else
    return (uint32_t)((uint64_t)p * magic >> 32) >> shift;
#endif
}

}  // namespace vgc
