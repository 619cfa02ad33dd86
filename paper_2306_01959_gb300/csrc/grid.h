// The cell of a coordinate along one axis.  Host and device, so that it is tested on
// the host.
#pragma once

#include <cstdint>
#include <cstring>

#ifndef __CUDA_ARCH__
#include <cmath>
#endif

#ifndef SPH_HD
#ifdef __CUDACC__
#define SPH_HD __host__ __device__ __forceinline__
#else
#define SPH_HD inline
#endif
#endif

namespace sph {

SPH_HD uint64_t double_u64(double x)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t u;
    std::memcpy(&u, &x, 8);
    return u;
#endif
}
SPH_HD int32_t double_hi(double x) { return (int32_t)(double_u64(x) >> 32); }
SPH_HD uint32_t double_lo(double x) { return (uint32_t)double_u64(x); }
SPH_HD int bits_of(uint32_t v)  // bits of v, 0 for 0
{
#ifdef __CUDA_ARCH__
    return 32 - __clz((int)v);
#else
    return v ? 32 - __builtin_clz(v) : 0;
#endif
}
// x 2^e for a normal x and a normal result.
SPH_HD double scale2(double x, int e)
{
#ifdef __CUDA_ARCH__
    return __hiloint2double(__double2hiint(x) + e * 0x100000, __double2loint(x));
#else
    return std::ldexp(x, e);
#endif
}

// Cell from the coordinate in cells; false outside [0, n).  One FP64 conversion
// (rounding down) instead of a floor, two comparisons and a conversion: the kernels
// that bin every particle are bound by the FP64 pipe (mixed update of 0.9 M particles
// 69 -> 54 us, of 1.77 M 140 -> 107 us).  The conversion saturates; a NaN, which it would
// turn into 0, is told by its bits.
SPH_HD bool cell_of(double f, int n, int &c)
{
#ifdef __CUDA_ARCH__
    c = __double2int_rd(f);
#else
    const double g = std::floor(f);
    c = g >= 2147483647.0 ? 0x7fffffff : (g <= -2147483648.0 ? (int)0x80000000 : (g == g ? (int)g : 0));
#endif
    return (unsigned)c < (unsigned)n && (double_hi(f) & 0x7ff00000) != 0x7ff00000;
}

// The cell along one axis as the definition states it, floor of the rounded quotient
// d / cs with d = x - lo, from the product with 1/cs.  Adding 1.5 2^36 leaves the
// coordinate in cells as an integer of 2^-16 in the low word (up to 2^16 cells; the high
// word tells what is outside).  The product and the quotient differ by less than 2^-36
// there, so that only a coordinate within 2^-16 of a face k is in question.  The
// remainder d - k cs is exact there, and the quotient rounds to k or above unless the
// remainder is below minus half the spacing of the doubles under k, times cs (never equal
// to it: that takes 54 bits).  A particle on a face (a lattice plane, where product and
// quotient may round to either side) is binned alike by every kernel.  Mixed update of
// 2.0 M particles with h = 1.5 dp, a third of whose lattice planes lie on faces: 107 us by
// the product alone, 170 with the division next to faces, 122 with the remainder; of
// 0.9 M with h = 2.08 dp 54, 48 and 48 us.
SPH_HD bool cell_of_product(double d, double cs, double inv_cs, int n, int &c)
{
#ifdef __CUDA_ARCH__
    const double q = fma(d, inv_cs, 0x1.8p36);
#else
    const double q = std::fma(d, inv_cs, 0x1.8p36);
#endif
    const uint32_t lo = double_lo(q);
    if (n > 0xffff)
        return cell_of(d / cs, n, c);
    c = (int)(lo >> 16);
    if (((lo + 1u) & 0xffffu) <= 2u) {
        const int k = (int)((lo + 1u) >> 16);
        if (double_hi(q) != 0x42380000 || k == 0)
            return cell_of(d / cs, n, c);
#ifdef __CUDA_ARCH__
        const double r = fma(-(double)k, cs, d);
#else
        const double r = std::fma(-(double)k, cs, d);
#endif
        c = r >= -scale2(cs, bits_of((uint32_t)(k - 1)) - 54) ? k : k - 1;
    }
    return double_hi(q) == 0x42380000 && c < n;
}

}  // namespace sph
