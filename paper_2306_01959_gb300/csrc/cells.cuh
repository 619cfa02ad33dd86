// Device bodies of the neighbour-structure phases: the scan of the per-cell
// counts into cell starts and the list of non-empty cells, the counting-sort
// scatter, and the per-cell sort fused with the gather of the sorted particle
// data (including the Tait pressure, Eq. 8).  The kernels of cells.cu run them
// one launch per phase; the persistent kernel of persist.cu runs them between
// grid barriers.  Each body takes the index of the unit it works on (tile,
// block or thread) and the number of such units, not blockIdx/gridDim.  Their
// pointers carry no __restrict__: in the persistent kernel the arrays they read
// were written by other CTAs earlier in the same launch, so the loads must not
// take the read-only (non-coherent) path.
#pragma once

#include <type_traits>

#include "device.cuh"
#include "fixed.h"

namespace sph {

// ---------------------------------------------------------------------------
// Scan of the per-cell counts.  Value per cell: (nonempty << 32) | count, so
// that one exclusive scan yields both the cell start and the index of the
// cell in the list of non-empty cells.  The out-of-domain bucket C is never
// marked non-empty.
// ---------------------------------------------------------------------------
constexpr int kScanThreads = 256;

__device__ __forceinline__ uint64_t scan_value(const uint32_t *count, int64_t c, int64_t C)
{
    if (c > C)
        return 0;
    uint32_t n = count[c];
    return ((uint64_t)(n > 0 && c < C) << 32) | n;
}

__device__ __forceinline__ uint64_t block_exclusive_scan(uint64_t v, uint64_t *warp_tot, uint64_t &total)
{
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint64_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o)
            x += y;
    }
    if (lane == 31)
        warp_tot[w] = x;
    __syncthreads();
    if (w == 0) {
        int nw = blockDim.x >> 5;
        uint64_t t = lane < nw ? warp_tot[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint64_t y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o)
                t += y;
        }
        if (lane < nw)
            warp_tot[lane] = t;
    }
    __syncthreads();
    uint64_t before = w > 0 ? warp_tot[w - 1] : 0;
    total = warp_tot[(blockDim.x >> 5) - 1];
    __syncthreads();
    return before + x - v;
}

// Tile `tile` of the cell counts (kScanTile cells, NT threads): its total goes to
// blocks[tile].
template <int NT = kScanThreads>
__device__ __forceinline__ void scan_reduce_tile(const uint32_t *count, uint64_t *blocks,
                                                 int64_t C, int64_t tile)
{
    constexpr int kScanItems = kScanTile / NT;
    __shared__ uint64_t warp_tot[32];
    int64_t base = tile * kScanTile + threadIdx.x * kScanItems;
    uint64_t s = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k)
        s += scan_value(count, base + k, C);
    uint64_t total;
    block_exclusive_scan(s, warp_tot, total);
    if (threadIdx.x == 0)
        blocks[tile] = total;
}

// Exclusive scan of the nb tile totals, by one block.
__device__ __forceinline__ void scan_blocks_block(uint64_t *blocks, int nb)
{
    __shared__ uint64_t warp_tot[32];
    uint64_t carry = 0;
    for (int base = 0; base < nb; base += blockDim.x) {
        int i = base + threadIdx.x;
        uint64_t v = i < nb ? blocks[i] : 0;
        uint64_t total;
        uint64_t ex = block_exclusive_scan(v, warp_tot, total);
        if (i < nb)
            blocks[i] = carry + ex;
        carry += total;
    }
}

// Tile `tile`: cell starts, non-empty cell list, and (last cell) the counts.
template <int NT = kScanThreads>
__device__ __forceinline__ void scan_final_tile(const uint32_t *count,
                                                const uint64_t *blocks, int32_t *cell_start,
                                                int32_t *active, int32_t *misc, int64_t C,
                                                int64_t tile)
{
    constexpr int kScanItems = kScanTile / NT;
    __shared__ uint64_t warp_tot[32];
    int64_t base = tile * kScanTile + threadIdx.x * kScanItems;
    uint64_t v[kScanItems];
    uint64_t s = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        v[k] = scan_value(count, base + k, C);
        s += v[k];
    }
    uint64_t total;
    uint64_t run = blocks[tile] + block_exclusive_scan(s, warp_tot, total);
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        int64_t c = base + k;
        if (c <= C) {
            cell_start[c] = (int32_t)(uint32_t)run;
            if ((v[k] >> 32) && check_ok((int64_t)(run >> 32) < C, &misc[2]))
                active[(uint32_t)(run >> 32)] = (int32_t)c;
            if (c == C) {
                misc[0] = (int32_t)(uint32_t)run;        // in-domain particles
                misc[1] = (int32_t)(run >> 32);          // non-empty cells
                misc[4] = 0;                             // tiles, listed with the sort
                cell_start[C + 1] = (int32_t)(uint32_t)(run + (v[k] & 0xffffffffu));
            }
        }
        run += v[k];
    }
}

// Counting-sort scatter over particles [thread0, N) with stride `stride`, entry(id)
// of each to its slot; decrementing the counters returns them to zero.
template <class T, class F>
__device__ __forceinline__ void scatter_entries(const uint32_t *key, uint32_t *count, const int32_t *cell_start, T *tmp,
                                                int32_t *misc, int64_t N, uint32_t C, int64_t thread0, int64_t stride,
                                                F &&entry)
{
    for (int64_t id = thread0; id < N; id += stride) {
        uint32_t c = key[id];
        if (c > C) {  // (C: the out-of-domain bucket)
            atomicOr(&misc[2], ST_OVERFLOW);
            continue;
        }
        uint32_t v = atomicSub(&count[c], 1u);
        int64_t slot = (int64_t)cell_start[c] + (int64_t)v - 1;
        if (v == 0u || slot < 0 || slot >= N) {  // counters out of step with the keys
            atomicOr(&misc[2], ST_OVERFLOW);
            continue;
        }
        tmp[slot] = entry(id);
    }
}

// The scatter of particle ids.
__device__ __forceinline__ void scatter_range(const uint32_t *key, uint32_t *count, const int32_t *cell_start,
                                              int32_t *tmp, int32_t *misc, int64_t N, uint32_t C, int64_t thread0,
                                              int64_t stride)
{
    scatter_entries(key, count, cell_start, tmp, misc, N, C, thread0, stride, [](int64_t id) { return (int32_t)id; });
}

// ---------------------------------------------------------------------------
// Per-cell sort + gather, one thread per particle: its rank within its cell is
// the number of smaller keys among the cell's scattered ones.  The FP64 form
// orders each cell by particle id, which gives the (cell, id) order of the
// method's definition.  The mixed form orders each cell by (x offset, id): rows
// of cells along x are then sorted by x, which the mixed pair kernel uses to cut
// its candidate ranges; the key travels with the scatter (x offset above id), so
// that ranking reads one short contiguous run.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t orderable(float f)
{
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

template <int MODE>
__device__ __forceinline__ void scatter_phase(const Bufs &b, int64_t N, int64_t thread0, int64_t stride)
{
    if (MODE == SPH_FP64)
        scatter_range(b.key, b.count, b.cell_start, b.ptmp, b.misc, N, (uint32_t)b.C, thread0, stride);
    else
        scatter_entries(b.key, b.count, b.cell_start, b.pkey, b.misc, N, (uint32_t)b.C, thread0, stride, [&](int64_t id) {
            return ((uint64_t)orderable(b.xof[id]) << 32) | (uint32_t)id;
        });
}

template <int MODE>
__device__ __forceinline__ void sort_reorder_range(const Bufs &b, int32_t ninst, int32_t thread0, int32_t stride)
{
    using Key = typename std::conditional<MODE == SPH_FP64, int32_t, uint64_t>::type;
    const Key *keys = MODE == SPH_FP64 ? reinterpret_cast<const Key *>(b.ptmp) : reinterpret_cast<const Key *>(b.pkey);
    const int32_t n_in = min(b.misc[0], b.N);
    for (int32_t slot = thread0; slot < n_in; slot += stride) {
        const Key key = keys[slot];
        const int32_t id = (int32_t)(uint32_t)(key & 0xffffffffu);
        if (!check_ok((uint32_t)id < (uint32_t)b.N, &b.misc[2]))
            continue;
        const int32_t c = (int32_t)b.key[id];
        if (!check_ok((uint32_t)c < (uint32_t)b.C, &b.misc[2]))
            continue;
        const dvec4 p = b.pos[id];
        const uint8_t type = b.type[id];
        const int32_t s0 = b.cell_start[c], s1 = b.cell_start[c + 1];
        const Inst &I = b.inst[b.inst_of[id]];
        if (!check_ok(s0 >= 0 && s0 <= slot && slot < s1 && s1 <= n_in, &b.misc[2]))
            continue;  // (the slot of a particle lies in its cell's run)
        int32_t s = s0;
        for (int32_t k = s0; k < s1; ++k)
            s += keys[k] < key;
        b.perm[s] = id;
        b.scell[s] = c;
        b.sflag[s] = type;
        if (b.xbuild)
            b.xbuild[id] = p;  // neighbour lists: reference of the displacement test
        if (MODE == SPH_FP64) {
            const dvec4 v = reinterpret_cast<const dvec4 *>(b.vel)[id];
            reinterpret_cast<dvec4 *>(b.sA)[s] = make_dvec4(__longlong_as_double(fixed_position(p.x, I.fx_shift)),
                                                            __longlong_as_double(fixed_position(p.y, I.fx_shift)),
                                                            __longlong_as_double(fixed_position(p.z, I.fx_shift)), v.w);
            reinterpret_cast<dvec4 *>(b.sB)[s] = make_dvec4(v.x, v.y, v.z, tait_d(I, v.w));
            b.sC[s] = make_double2(1.0 / v.w, sound_d(I, v.w));
            b.sD[s] = make_float4((float)p.x, (float)p.y, (float)p.z, type == T_FLUID ? 1.f : 0.f);
        } else {
            const float4 v = reinterpret_cast<const float4 *>(b.vel)[id];
            // offsets in the cell
            int cx, cy, cz;
            decompose(I, c, cx, cy, cz);
            const double oy0 = I.olo[1] + cy * I.oc, oz0 = I.olo[2] + cz * I.oc;
            reinterpret_cast<float4 *>(b.sA)[s] =
                make_float4(b.xof[id], (float)(p.y - oy0), (float)(p.z - oz0), v.w);
            reinterpret_cast<float4 *>(b.sB)[s] = make_float4(v.x, v.y, v.z, tait_f(I, v.w));
        }
    }
}

// ---------------------------------------------------------------------------
// The non-empty tiles of the mixed pair pass (boxes of Inst::tdim cells), from
// the cell starts: threads [thread0, ..) with stride `stride`, whole warps.
// Their order does not matter to the results; consecutive tiles mostly stay
// together.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void tile_list_range(const Bufs &b, int32_t ninst, int32_t thread0, int32_t stride)
{
    const int lane = threadIdx.x & 31;
    for (int32_t base = thread0 - lane; base < b.ntiles; base += stride) {
        const int32_t t = base + lane;
        bool used = false;
        if (t < b.ntiles) {
            const Inst &I = b.inst[inst_of_tile(b.inst, ninst, t)];
            const int32_t l = t - I.tile_base, q = l / I.ntile[0];
            const int x0 = (l - q * I.ntile[0]) * I.tdim[0], x1 = min(x0 + I.tdim[0], I.n[0]);
            const int z0 = (q / I.ntile[1]) * I.tdim[2], y0 = (q - (q / I.ntile[1]) * I.ntile[1]) * I.tdim[1];
            for (int z = z0; z < min(z0 + I.tdim[2], I.n[2]); ++z)
                for (int y = y0; y < min(y0 + I.tdim[1], I.n[1]); ++y) {
                    const int32_t row = I.cell_base + (z * I.n[1] + y) * I.n[0];
                    used = used || b.cell_start[row + x1] > b.cell_start[row + x0];
                }
        }
        const unsigned m = __ballot_sync(0xffffffffu, used);
        int32_t at = 0;
        if (lane == 0 && m)
            at = atomicAdd(&b.misc[4], __popc(m));
        at = __shfl_sync(0xffffffffu, at, 0);
        at += __popc(m & ((1u << lane) - 1u));
        if (used && at < b.ntiles)
            b.tiles[at] = t;
    }
}

}  // namespace sph
