// Division of indices by a number known beforehand: a high product, an addition and a
// shift (Granlund and Montgomery, "Division by Invariant Integers using
// Multiplication", 1994, the unsigned form).
#pragma once

#include <cstdint>

#ifndef SPH_HD
#ifdef __CUDACC__
#define SPH_HD __host__ __device__ __forceinline__
#else
#define SPH_HD inline
#endif
#endif

namespace sph {

struct Divisor {
    uint32_t m;  // floor(2^32 (2^s - d) / d) + 1
    int32_t s;   // ceil(log2 d)
};

inline Divisor divisor(int32_t d)  // d >= 1
{
    int32_t s = 0;
    while (((int64_t)1 << s) < d)
        ++s;
    const uint64_t excess = ((uint64_t)1 << s) - (uint64_t)d;
    return {(uint32_t)((excess << 32) / (uint64_t)d + 1), s};
}

// a / d for 0 <= a < 2^31.
SPH_HD int32_t divide(int32_t a, Divisor d)
{
#ifdef __CUDA_ARCH__
    const uint32_t h = __umulhi((uint32_t)a, d.m);
#else
    const uint32_t h = (uint32_t)(((uint64_t)(uint32_t)a * d.m) >> 32);
#endif
    return (int32_t)((h + (uint32_t)a) >> d.s);
}

}  // namespace sph
