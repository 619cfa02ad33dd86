// Persistent form of the time loop: one cooperative launch advances every
// instance of a handle (a batch of dam breaks, e.g. an alpha sweep) by nsteps
// Verlet steps of the mixed form.  Each step runs the phases of the per-phase
// launches in the same order - pair pass (Eqs. 3-8), adaptive dt (Eq. 15),
// Verlet update with rebinning (Eqs. 9-14), cell scan, scatter, per-cell sort
// and gather - with a grid-wide barrier between phases instead of a kernel
// boundary.  The phase bodies are the ones the per-phase kernels run
// (pair_mixed.cuh, step.cuh, cells.cuh), so a persistent step computes what a
// launched step computes, bit for bit.
//
// The barrier (grid_barrier, device.cuh) counts in the workspace.  Every wait is
// bounded: after spin_limit polls the CTA records ST_TIMEOUT in the device status
// (reported as SPH_ETIMEOUT) and returns, and every other CTA then runs out at its
// next barrier, so the launch always ends.  A cooperative launch guarantees that
// all CTAs are resident at once.
//
// A failed check (an index out of its range, counters out of step with the keys;
// the access is skipped) ends the launch before the next update, so that the
// remaining steps do not run on wrong data; sph_sync reports SPH_ESTATE.
//
// What each phase reads of what an earlier one wrote in the same launch, and the
// barrier in between (numbered as in the step below; the last one ends the step):
//   1 pair       sA sB scell sflag (8-9), cell_start (7), tiles misc[4] (8-9), misc[3] (3)
//   2 dt maxima  deriv mumax (1), scell sflag (8-9 of the step before)
//   3 dt         red (2); misc[2] (anywhere before)
//   4 update     dt euler misc[5] (3), deriv (1), perm (8-9), pos vel velp (own particle)
//   5 scan       count (4; the scatter of the step before leaves zeros)
//   6 scan       scan_blocks (5)
//   7 scan       scan_blocks (6), count (4)
//   8 scatter    key xof (4), cell_start (7), count (4, taken down by this phase alone)
//   9 tile list  cell_start (7), misc[4] (set to 0 in 7)
//   9 sort       pkey (8), key pos vel xof (4), cell_start misc[0] (7)
// The update (4) writes key, xof and count, the sort (9) perm, scell, sflag, sA and
// sB: none of them is read by another CTA in the same phase.
#include "cells.cuh"
#include "pair_wide.cuh"
#include "step.cuh"

namespace sph {

namespace {

constexpr int kPersistWarps = 8;  // the pair pass's default shape: 8 warps,
constexpr int kPersistGroup = 4;  // 4 particles per warp

template <bool TILED, bool DFS>
__global__ void __launch_bounds__(kPersistWarps * 32, 2)
    k_persistent_steps(Bufs b, int ninst, int nsteps, int ns, int kdiv, int max_stage, int64_t N, uint32_t C, int ntiles,
                       long long spin_limit)
{
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ typename std::conditional<TILED, PairSmem, WideSmem>::type S;
    __shared__ int s_ok;
    unsigned target = 0;
    const int tid = threadIdx.x;
    const int gthread = blockIdx.x * blockDim.x + tid, gstride = gridDim.x * blockDim.x;
    int32_t *status = &b.misc[2];
#define SPH_BARRIER()                                                       \
    if (!grid_barrier(b.bar, target, spin_limit, status, &s_ok))            \
        return;
    for (int step = 0; step < nsteps; ++step) {
        if constexpr (TILED)
            pair_mixed_body<kPersistWarps, kPersistGroup, true, false, DFS>(b, ninst, kdiv, dyn, S);
        else
            pair_wide_body<kPersistWarps, kPersistGroup, true, false, DFS>(b, ninst, kdiv, max_stage, dyn, S);
        SPH_BARRIER();
        dt_reduce_part<SPH_MIXED>(b, ninst, blockIdx.x, gridDim.x);
        SPH_BARRIER();
        if (blockIdx.x == 0) {
            dt_finalize_block(b, ninst, ns);
            if (tid == 0) {
                b.misc[3] = 0;  // the pair pass's work queue, for the next step
                b.misc[5] = (__ldcg(&b.misc[2]) & (ST_OVERFLOW | ST_BOUNDS)) != 0;
            }
        }
        SPH_BARRIER();
        // written by one thread between two barriers, so that every CTA leaves here or none
        if (b.misc[5])
            return;
        integrate_range<SPH_MIXED>(b, N, C, gthread, gstride);
        SPH_BARRIER();
        for (int t = blockIdx.x; t < ntiles; t += gridDim.x)
            scan_reduce_tile<kPersistWarps * 32>(b.count, b.scan_blocks, C, t);
        SPH_BARRIER();
        if (blockIdx.x == 0)
            scan_blocks_block(b.scan_blocks, ntiles);
        SPH_BARRIER();
        for (int t = blockIdx.x; t < ntiles; t += gridDim.x)
            scan_final_tile<kPersistWarps * 32>(b.count, b.scan_blocks, b.cell_start, b.active, b.misc, C, t);
        SPH_BARRIER();
        scatter_phase<SPH_MIXED>(b, N, gthread, gstride);
        SPH_BARRIER();
        tile_list_range(b, ninst, gthread, gstride);
        sort_reorder_range<SPH_MIXED>(b, ninst, gthread, gstride);
        SPH_BARRIER();
    }
#undef SPH_BARRIER
}

template <bool TILED, bool DFS>
cudaError_t launch_typed(const Bufs &b, int ninst, int nsteps, int ns, int cell_div, int64_t N, int32_t C,
                         long long spin_limit, cudaStream_t st)
{
    int max_stage = wide_max_stage(cell_div);
    const size_t dyn = TILED ? mixed_dyn_smem(kPersistWarps) : wide_dyn_smem(max_stage, kPersistWarps, kPersistGroup);
    static size_t dyn_set = 0;
    cudaError_t e;
    if (dyn > dyn_set) {
        e = cudaFuncSetAttribute(k_persistent_steps<TILED, DFS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
        if (e != cudaSuccess)
            return e;
        dyn_set = dyn;
    }
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_persistent_steps<TILED, DFS>, kPersistWarps * 32, dyn);
    if (e != cudaSuccess)
        return e;
    if (per_sm < 1)
        return cudaErrorLaunchOutOfResources;
    const int grid = per_sm * sm_count();
    int ntiles = (int)((C + 1 + kScanTile - 1) / kScanTile);
    uint32_t Cu = (uint32_t)C;
    void *args[] = {(void *)&b, &ninst, &nsteps, &ns, &cell_div, &max_stage, &N, &Cu, &ntiles, &spin_limit};
    e = cudaMemsetAsync(b.bar, 0, sizeof(unsigned), st);
    if (e != cudaSuccess)
        return e;
    e = cudaMemsetAsync(b.misc + 3, 0, sizeof(int32_t), st);
    if (e != cudaSuccess)
        return e;
    return cudaLaunchCooperativeKernel((const void *)k_persistent_steps<TILED, DFS>, grid, kPersistWarps * 32, args, dyn, st);
}

}  // namespace

cudaError_t launch_persistent_steps(const Bufs &b, bool tiled, int32_t ninst, int32_t nsteps, int32_t ns,
                                    int32_t cell_div, int32_t delta_mode, int64_t N, int32_t C, long long spin_limit,
                                    cudaStream_t st)
{
    const bool dfs = delta_mode == SPH_DELTA_FULL_SUPPORT;
    auto launch = tiled ? (dfs ? launch_typed<true, true> : launch_typed<true, false>)
                        : (dfs ? launch_typed<false, true> : launch_typed<false, false>);
    return launch(b, ninst, nsteps, ns, cell_div, N, C, spin_limit, st);
}

}  // namespace sph
