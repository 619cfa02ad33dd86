// Cell-linked neighbour structure: binning, per-cell counts, a scan of the
// counts into cell starts and the list of non-empty cells, a counting-sort
// scatter, and a per-cell sort by particle id fused with the gather of the
// sorted particle data (including the Tait pressure, Eq. 8).
//
// The resulting order is ascending (cell, id) for every in-domain particle;
// out-of-domain particles fill the bucket after the last cell in arbitrary
// order and take no further part.
#include "cells.cuh"

namespace sph {

// With neighbour lists, `gate` is the rebuild request: these kernels run only
// when it is set (steps that reuse the lists keep the last sorted order); a
// null gate always runs.
__device__ __forceinline__ bool gated_off(const int32_t *gate) { return gate && *gate == 0; }

// ---------------------------------------------------------------------------
// Binning of the canonical state (used at creation, after a state load and,
// with neighbour lists, at a rebuild).
// ---------------------------------------------------------------------------
template <int MODE>
__global__ void k_bin(const dvec4 *__restrict__ pos, const uint16_t *__restrict__ inst_of,
                      const Inst *__restrict__ inst, uint32_t *__restrict__ key, uint32_t *__restrict__ count,
                      float *__restrict__ xof, int64_t N, uint32_t C, const int32_t *gate)
{
    if (gated_off(gate))
        return;
    for (int64_t id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; id < N; id += (int64_t)gridDim.x * blockDim.x) {
        const Inst &I = inst[inst_of[id]];
        dvec4 p = pos[id];
        int cx, cy, cz;
        uint32_t c = C;
        const bool in = MODE == SPH_FP64 ? cell_coords_exact(I, p.x, p.y, p.z, cx, cy, cz)
                                         : cell_coords_fast(I, p.x, p.y, p.z, cx, cy, cz);
        if (in)
            c = (uint32_t)(I.cell_base + (cz * I.n[1] + cy) * I.n[0] + cx);
        if (MODE == SPH_MIXED && in)
            xof[id] = x_offset(I, p.x, cx);
        key[id] = c;
        atomicAdd(&count[c], 1u);
    }
}

void launch_bin(const Bufs &b, int mode, int64_t N, int32_t C, cudaStream_t st)
{
    int blocks = (int)std::min<int64_t>((N + 255) / 256, 4096);
    if (blocks < 1)
        blocks = 1;
    if (mode == SPH_FP64)
        k_bin<SPH_FP64><<<blocks, 256, 0, st>>>(b.pos, b.inst_of, b.inst, b.key, b.count, b.xof, N, (uint32_t)C, b.lflag);
    else
        k_bin<SPH_MIXED><<<blocks, 256, 0, st>>>(b.pos, b.inst_of, b.inst, b.key, b.count, b.xof, N, (uint32_t)C, b.lflag);
}

// One launch per phase; the bodies live in cells.cuh.
__global__ void k_scan_reduce(const uint32_t *__restrict__ count, uint64_t *__restrict__ blocks, int64_t C,
                              const int32_t *gate)
{
    if (gated_off(gate))
        return;
    scan_reduce_tile(count, blocks, C, blockIdx.x);
}

__global__ void k_scan_blocks(uint64_t *__restrict__ blocks, int nb, const int32_t *gate)
{
    if (gated_off(gate))
        return;
    scan_blocks_block(blocks, nb);
}

__global__ void k_scan_final(const uint32_t *__restrict__ count, const uint64_t *__restrict__ blocks,
                             int32_t *__restrict__ cell_start, int32_t *__restrict__ active,
                             int32_t *__restrict__ misc, int64_t C, const int32_t *gate)
{
    if (gated_off(gate))
        return;
    scan_final_tile(count, blocks, cell_start, active, misc, C, blockIdx.x);
}

template <int MODE>
__global__ void k_scatter(Bufs b, int64_t N)
{
    if (gated_off(b.lflag))
        return;
    scatter_phase<MODE>(b, N, blockIdx.x * (int64_t)blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x);
}

void launch_cells(const Bufs &b, int mode, int64_t N, int32_t C, cudaStream_t st)
{
    int nb = (int)((C + 1 + kScanTile - 1) / kScanTile);
    k_scan_reduce<<<nb, kScanThreads, 0, st>>>(b.count, b.scan_blocks, C, b.lflag);
    k_scan_blocks<<<1, 1024, 0, st>>>(b.scan_blocks, nb, b.lflag);
    k_scan_final<<<nb, kScanThreads, 0, st>>>(b.count, b.scan_blocks, b.cell_start, b.active, b.misc, C, b.lflag);
    int blocks = (int)std::min<int64_t>((N + 255) / 256, 8192);
    if (blocks < 1)
        blocks = 1;
    if (mode == SPH_FP64)
        k_scatter<SPH_FP64><<<blocks, 256, 0, st>>>(b, N);
    else
        k_scatter<SPH_MIXED><<<blocks, 256, 0, st>>>(b, N);
}

// One thread per particle, gathers in flight from as many threads as fit: the
// ranking loop is short (about 9 particles per cell of size h on a lattice of
// h = 2.08 dp), so a warp per cell, as the cells of 2h had, would idle most lanes.
template <int MODE>
__global__ void __launch_bounds__(256) k_sort_reorder(Bufs b, int32_t ninst)
{
    if (gated_off(b.lflag))
        return;
    if (MODE == SPH_MIXED)
        tile_list_range(b, ninst, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
    sort_reorder_range<MODE>(b, ninst, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

void launch_reorder(const Bufs &b, int mode, int64_t N, int32_t ninst, int32_t ctas_per_sm, cudaStream_t st)
{
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((N + 255) / 256, (int64_t)sm_count() * std::max(1, ctas_per_sm)));
    if (mode == SPH_FP64)
        k_sort_reorder<SPH_FP64><<<blocks, 256, 0, st>>>(b, ninst);
    else
        k_sort_reorder<SPH_MIXED><<<blocks, 256, 0, st>>>(b, ninst);
}

}  // namespace sph
