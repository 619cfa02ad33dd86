// Fixed-point arithmetic of the FP64 pair pass (pair_fp64.cu): positions, squared
// distances, t^3 = (1 - q/2)^3 and the reciprocal of the viscosity's denominator in
// 64-bit integers.  Host and device, so that it is tested on the host.
//
// Unit: 2^-s with 2h in [2^62, 2^63) units.  Positions are kept modulo 2^64: the
// difference of two particles within the support is below 2^63 and so exact however
// long the tank is, and a position is rounded (by 2^-63 of 2h at most) only within
// 2h / 512 of a coordinate plane, where doubles are finer still.
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

SPH_HD uint64_t double_bits(double x)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t u;
    std::memcpy(&u, &x, 8);
    return u;
#endif
}
SPH_HD double bits_double(uint64_t u)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    double x;
    std::memcpy(&x, &u, 8);
    return x;
#endif
}
SPH_HD uint64_t mulhi_u64(uint64_t a, uint64_t b)
{
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}
SPH_HD int64_t mulhi_s64(int64_t a, int64_t b)
{
#ifdef __CUDA_ARCH__
    return __mul64hi(a, b);
#else
    return (int64_t)(((__int128)a * b) >> 64);
#endif
}
SPH_HD uint32_t mulhi_u32(uint32_t a, uint32_t b)
{
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}
SPH_HD int clz64(uint64_t a)
{
#ifdef __CUDA_ARCH__
    return __clzll((long long)a);
#else
    return a ? __builtin_clzll(a) : 64;
#endif
}
// v 2^32 / sqrt(hi) and 2^30 / hi style starts: the FP32 approximations scaled to an
// integer, saturating.  On the host a relative error like the hardware's (at most
// 2^-22.9) can be put on them.
#ifndef __CUDA_ARCH__
inline double &host_approx_error()
{
    static double e = 0.0;
    return e;
}
inline uint32_t host_saturate(double x) { return x >= 4294967295.0 ? 0xffffffffu : (uint32_t)x; }
#endif
SPH_HD uint32_t rsqrt_start(uint32_t hi)
{
#ifdef __CUDA_ARCH__
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"((float)hi));
    return __float2uint_rz(y * 140737488355328.f);  // 2^47
#else
    return host_saturate((float)(1.0 / std::sqrt((double)(float)hi) * (1.0 + host_approx_error())) * 140737488355328.0);
#endif
}
SPH_HD uint32_t rcp_start(uint32_t hi)
{
#ifdef __CUDA_ARCH__
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"((float)hi));
    return __float2uint_rz(y * 4611686018427387904.f);  // 2^62
#else
    return host_saturate((float)(1.0 / (double)(float)hi * (1.0 + host_approx_error())) * 4611686018427387904.0);
#endif
}

// m 2^(biased - 1086) for a normalised m (top bit set), rounded to nearest.
SPH_HD double norm_to_double(uint64_t m, int biased)
{
    return bits_double((m >> 11) + ((m >> 10) & 1u) + ((uint64_t)(int64_t)(biased - 1) << 52));
}

// An integer, rounded to nearest.
SPH_HD double int_to_double(int64_t v)
{
    const uint64_t u = v < 0 ? 0ull - (uint64_t)v : (uint64_t)v;
    const int n = clz64(u);
    const double x = norm_to_double(u << (n & 63), 1086 - n);
    return u ? bits_double(double_bits(x) | ((uint64_t)v & 0x8000000000000000ull)) : 0.0;
}

// x 2^s modulo 2^64, rounded to nearest.
SPH_HD int64_t fixed_position(double x, int s)
{
    const uint64_t b = double_bits(x);
    const uint64_t m = (b & 0xfffffffffffffull) | 1ull << 52;
    const int sh = (int)((b >> 52) & 0x7ff) - 1075 + s;
    const uint64_t u = sh >= 0 ? (sh < 64 ? m << (sh & 63) : 0ull)
                               : (sh > -64 ? ((m >> ((-sh - 1) & 63)) + 1) >> 1 : 0ull);
    return (int64_t)((b >> 63) ? 0ull - u : u);
}

// |r_ij|^2 in units of 2^64 times the square of the position's: integer part (below
// 2^62 within the support) and 32 fraction bits, of which the sums below lose less
// than three of the second lowest.
struct Fixed2 {
    uint64_t R;
    uint32_t f;
};
SPH_HD Fixed2 fixed_dist2(int64_t dx, int64_t dy, int64_t dz)
{
    uint64_t p = 0, m = 0;
    uint32_t l = 0;
    const int64_t d[3] = {dx, dy, dz};
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int a = 0; a < 3; ++a) {
        const uint64_t u = d[a] < 0 ? 0ull - (uint64_t)d[a] : (uint64_t)d[a];
        const uint32_t lo = (uint32_t)u, hi = (uint32_t)(u >> 32);
        p += (uint64_t)hi * hi;
        m += (uint64_t)lo * hi;  // (the hi sum to less than 1.74 2^31: no overflow)
        l += mulhi_u32(lo, lo) >> 2;
    }
    m += (uint64_t)l << 1;
    return Fixed2{p + (m >> 31), (uint32_t)m << 1};
}

// R:f shifted left by n in [1, 31].
SPH_HD uint64_t shift_in(uint64_t R, uint32_t f, int n) { return (R << n) | (f >> (32 - n)); }

// t^3 = (1 - q/2)^3, 0 beyond the support, for 2^48 <= R: |r| from one third-order step
// (Householder's method: S (1 + E/2 + 3/8 E^2) in the residual E of the start), t as a
// 62-bit fraction, normalised before it is cubed.  kh: 2^126 / 2h.
SPH_HD double fixed_t3(Fixed2 d, uint64_t kh)
{
    const int n = clz64(d.R) & ~1;              // 2 .. 14
    const uint64_t m = shift_in(d.R, d.f, n);   // [2^62, 2^64): v = m / 2^62 in [1, 4)
    const uint32_t Y = rsqrt_start((uint32_t)(m >> 32));  // 2^32 / sqrt(v)
    const uint64_t S = (m >> 32) * Y + mulhi_u32((uint32_t)m, Y);  // sqrt(v), 62 fraction bits
    const int64_t E = (int64_t)((1ull << 62) - ((S >> 32) * Y + mulhi_u32((uint32_t)S, Y)));  // 1 - v y^2
    const int32_t e = (int32_t)(E >> 12);
    const int64_t g = (E >> 1) + ((3 * (((int64_t)e * e) >> 38)) >> 3);  // E / 2 + 3/8 E^2
    const uint64_t q = S + (uint64_t)(mulhi_s64((int64_t)S, (int64_t)((uint64_t)g << 22)) >> 20);
    const uint64_t r = q >> (n / 2 - 1);  // |r_ij|
    const int64_t t = (int64_t)((1ull << 62) - mulhi_u64(r, kh));
    const uint64_t tp = t > 0 ? (uint64_t)t : 0ull;
    const int k = clz64(tp);
    const uint64_t u = tp << (k & 63);
    const uint64_t c = mulhi_u64(mulhi_u64(u, u), u);  // t^3 = c 2^(-3k - 58)
    const int kc = clz64(c);                          // 0 .. 2
    const double x = norm_to_double(c << (kc & 63), 1028 - kc - 3 * k);
    return t > 0 ? x : 0.0;
}

// 1 / (V d) for V = R + f 2^-32 with 2^49 <= R < 2^63 and a normal d = (1 + x) 2^(ex - 1023),
// ex in [128, 1792), from d's bits: the product of the two mantissas, W in [1/4, 1), its
// reciprocal by one third-order step from the FP32 approximation (Householder's again),
// rounded once.
SPH_HD double fixed_rcp(Fixed2 V, double d)
{
    const uint64_t b = double_bits(d);
    const int ex = (int)(b >> 52);
    const int n = clz64(V.R);  // 1 .. 14
    const uint64_t w = mulhi_u64(shift_in(V.R, V.f, n), (b << 11) | 1ull << 63);  // W, 64 fraction bits
    const uint32_t Y = rcp_start((uint32_t)(w >> 32));                            // 2^30 / W
    const int64_t E = (int64_t)((1ull << 62) - ((w >> 32) * Y + mulhi_u32((uint32_t)w, Y)));  // 1 - W Y
    const int32_t e = (int32_t)(E >> 12);
    const int64_t g = E + (((int64_t)e * e) >> 38);  // E + E^2
    const uint64_t z = ((uint64_t)Y << 31) +
                       (uint64_t)(mulhi_s64((int64_t)((uint64_t)Y << 30), (int64_t)((uint64_t)g << 21)) >> 18);  // 2^61 / W
    const int k = clz64(z);
    return norm_to_double(z << (k & 63), 1086 - k + n + 897 - ex);
}

}  // namespace sph
