// Device helpers shared by the kernels: cell coordinates, the Tait equation of
// state (Eq. 8), the sound speed and small warp utilities.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "grid.h"
#include "internal.h"

namespace sph {

// Cell coordinates with the exact IEEE division (x - lo) / cs, as the
// definition of the grid states it; false when outside the grid.
__device__ __forceinline__ bool cell_coords_exact(const Inst &I, double x, double y, double z, int &cx, int &cy,
                                                  int &cz)
{
    const bool ix = cell_of((x - I.lo[0]) / I.cs, I.n[0], cx), iy = cell_of((y - I.lo[1]) / I.cs, I.n[1], cy),
               iz = cell_of((z - I.lo[2]) / I.cs, I.n[2], cz);
    return ix && iy && iz;
}

// The cells of cell_coords_exact, at the cost of three products.
__device__ __forceinline__ bool cell_coords_fast(const Inst &I, double x, double y, double z, int &cx, int &cy,
                                                 int &cz)
{
    const bool ix = cell_of_product(x - I.lo[0], I.cs, I.inv_cs, I.n[0], cx),
               iy = cell_of_product(y - I.lo[1], I.cs, I.inv_cs, I.n[1], cy),
               iz = cell_of_product(z - I.lo[2], I.cs, I.inv_cs, I.n[2], cz);
    return ix && iy && iz;
}

// x offset of a particle in its cell (mixed form).
__device__ __forceinline__ float x_offset(const Inst &I, double x, int cx) { return (float)(x - (I.olo[0] + cx * I.oc)); }

// Streaming multiprocessors of the current device (queried once per device;
// grids of the memory-bound kernels are capped at a multiple of it).
inline int sm_count()
{
    static int cached[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64)
        dev = 0;
    if (!cached[dev]) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1)
            n = 1;
        cached[dev] = n;
    }
    return cached[dev];
}

__device__ __forceinline__ double pow7(double x)
{
    double x2 = x * x;
    return x2 * x2 * x2 * x;
}

// Eq. 8 in double.
__device__ __forceinline__ double tait_d(const Inst &I, double rho)
{
    double x = rho / I.rho0;
    double p = I.gamma == 7.0 ? pow7(x) : pow(x, I.gamma);
    return I.B * (p - 1.0);
}

// Eq. 8 in float from the density offset d = rho - rho0:
// (1 + x)^7 - 1 expanded by the binomial theorem, which keeps full relative
// precision for small x = d / rho0.
__device__ __forceinline__ float tait_f(const Inst &I, float d)
{
    float x = d * I.inv_rho0f;
    if (I.gamma == 7.0)
        return I.Bf * x * (7.f + x * (21.f + x * (35.f + x * (35.f + x * (21.f + x * (7.f + x))))));
    return I.Bf * expm1f(I.gammaf * log1pf(x));
}

// c_i: sqrt(dP/drho) of Eq. 8, c0 (rho/rho0)^((gamma-1)/2), or c0.
__device__ __forceinline__ double sound_d(const Inst &I, double rho)
{
    if (I.csound == SPH_CSOUND_CONSTANT)
        return I.c0;
    double x = rho / I.rho0;
    if (I.gamma == 7.0)
        return I.c0 * x * x * x;
    return I.c0 * pow(x, 0.5 * (I.gamma - 1.0));
}

// Barrier of a cooperative grid (every CTA resident): a counter that each CTA
// raises once per barrier, waited on until it reaches (barriers passed) x (CTAs).
// The release makes the CTA's writes before its barrier visible, the acquire those
// of the others to the CTA after its own; both stand for the whole CTA, whose
// threads are ordered with thread 0 by the CTA barriers around it.  The wait is
// bounded: after `limit` polls thread 0 records ST_TIMEOUT in *status, and the
// barrier returns false to every thread of the CTA; the caller returns then, and
// every other CTA runs out at its next barrier.
__device__ __forceinline__ bool grid_barrier(unsigned *bar, unsigned &target, long long limit, int32_t *status,
                                             int *s_ok)
{
    __syncthreads();
    target += gridDim.x;
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
        bool ok = true;
        for (long long polls = 0;; ++polls) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
            if ((int)(v - target) >= 0)  // (the counter may wrap)
                break;
            if (polls >= limit) {
                atomicOr(status, ST_TIMEOUT);
                ok = false;
                break;
            }
            if (polls > 64)
                __nanosleep(20);
        }
        *s_ok = ok;
    }
    __syncthreads();
    return *s_ok != 0;
}

// Max of a non-negative double through its bit pattern (order preserving for
// x >= 0; a NaN result propagates as the largest pattern).
__device__ __forceinline__ void atomic_max_pos(unsigned long long *addr, double x)
{
    atomicMax(addr, (unsigned long long)__double_as_longlong(x));
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Maximum of non-negative doubles by their bit patterns, which order alike (the
// integer units instead of the FP64 pipe).
__device__ __forceinline__ long long warp_max_bits(long long v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Warp totals of K values (K a power of two, at most 32) by a value-splitting
// butterfly: at each of the first log2 K levels a lane keeps half of its
// values and adds its partner's copies of them, the remaining levels add the
// one value left, so K values cost K FP64 additions per lane (5 K for K
// separate butterflies).  On return v[k] of lane 0 holds the total of value k
// (other lanes: undefined), times `scale`.  The order of the additions is fixed.
template <int K>
__device__ __forceinline__ void warp_totals(double (&v)[K], double scale = 1.0)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = K, o = 16; k > 1; k >>= 1, o >>= 1) {
        const bool upper = (lane & o) != 0;
        const int half = k >> 1;
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const double keep = upper ? v[i + half] : v[i];
            const double send = upper ? v[i] : v[i + half];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
#pragma unroll
    for (int o = 16 / K; o > 0; o >>= 1)
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    // lane (32 / K) k holds the total of value k
    const double mine = scale * v[0];
#pragma unroll
    for (int k = 0; k < K; ++k)
        v[k] = __shfl_sync(0xffffffffu, mine, k * (32 / K));
}

__device__ __forceinline__ int warp_sum(int v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Instance owning a global cell id (instances hold consecutive cell ranges).
__device__ __forceinline__ int inst_of_cell(const Inst *inst, int ninst, int32_t c)
{
    int lo = 0, hi = ninst - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (inst[mid].cell_base <= c)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// Instance owning a global tile id.
__device__ __forceinline__ int inst_of_tile(const Inst *inst, int ninst, int32_t t)
{
    int lo = 0, hi = ninst - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (inst[mid].tile_base <= t)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ void decompose(const Inst &I, int32_t c, int &cx, int &cy, int &cz)
{
    const int lc = c - I.cell_base, t = divide(lc, I.by_nx);
    cx = lc - t * I.n[0];
    cz = divide(t, I.by_ny);
    cy = t - cz * I.n[1];
}

}  // namespace sph
