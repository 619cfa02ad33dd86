// Launchers of the mixed-precision pair pass (Eqs. 3-8); the kernel body, its
// work decomposition and its compensated sums are described in pair_mixed.cuh.
#include "pair_mixed.cuh"

namespace sph {

// One CTA per resident slot; the body lives in pair_mixed.cuh.
template <int NW, int G, bool COMP, bool STAT, bool DFS>
__global__ void __launch_bounds__(NW * 32, NW >= 16 ? 1 : 2) k_pair_mixed(Bufs b, int ninst, int kdiv)
{
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ PairSmem S;
    pair_mixed_body<NW, G, COMP, STAT, DFS>(b, ninst, kdiv, dyn, S);
}

template <int NW, int G, bool COMP, bool STAT, bool DFS>
static void launch_nw(const Bufs &b, int ninst, int kdiv, int ctas, cudaStream_t st)
{
    const size_t dyn = mixed_dyn_smem(NW);
    static bool dyn_set = false;  // attribute set once per instantiation, outside any capture
    if (!dyn_set) {
        cudaFuncSetAttribute(k_pair_mixed<NW, G, COMP, STAT, DFS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)dyn);
        dyn_set = true;
    }
    k_pair_mixed<NW, G, COMP, STAT, DFS><<<sm_count() * ctas, NW * 32, dyn, st>>>(b, ninst, kdiv);
}

template <bool COMP, bool STAT, bool DFS>
static void launch_comp(const Bufs &b, int ninst, int kdiv, int warps, int group, int ctas, cudaStream_t st)
{
    if (group >= 4) {
        if (warps <= 8)
            launch_nw<8, 4, COMP, STAT, DFS>(b, ninst, kdiv, ctas, st);
        else
            launch_nw<16, 4, COMP, STAT, DFS>(b, ninst, kdiv, ctas, st);
    } else {
        if (warps <= 8)
            launch_nw<8, 2, COMP, STAT, DFS>(b, ninst, kdiv, ctas, st);
        else
            launch_nw<16, 2, COMP, STAT, DFS>(b, ninst, kdiv, ctas, st);
    }
}

void launch_pair_mixed(const Bufs &b, int32_t ninst, int32_t cell_div, int32_t warps, int32_t ctas, int32_t group,
                       int32_t compensated, bool stats, int32_t delta_mode, cudaStream_t st)
{
    // defaults: the fastest launch shape measured on GB300
    if (warps <= 0)
        warps = 8;
    if (ctas <= 0)
        ctas = 2;
    if (group <= 0)
        group = 4;
    cudaMemsetAsync(b.misc + 3, 0, sizeof(int32_t), st);
    if (stats)
        cudaMemsetAsync(b.pstat, 0, 4 * sizeof(unsigned long long), st);
    if (delta_mode == SPH_DELTA_FULL_SUPPORT) {  // always compensated
        if (stats)
            launch_comp<true, true, true>(b, ninst, cell_div, warps, group, ctas, st);
        else
            launch_comp<true, false, true>(b, ninst, cell_div, warps, group, ctas, st);
    } else if (stats) {
        if (compensated)
            launch_comp<true, true, false>(b, ninst, cell_div, warps, group, ctas, st);
        else
            launch_comp<false, true, false>(b, ninst, cell_div, warps, group, ctas, st);
    } else if (compensated) {
        launch_comp<true, false, false>(b, ninst, cell_div, warps, group, ctas, st);
    } else {
        launch_comp<false, false, false>(b, ninst, cell_div, warps, group, ctas, st);
    }
}

}  // namespace sph
