#pragma once
// Mixed-precision form of the pair pass (Eqs. 3-8), device body: FP32 pair
// arithmetic on cell-relative offsets, with compensated FP32 accumulation.
//
// Work decomposition (persistent CTAs; one work item = one non-empty tile, a
// box of tdim cells):
//  1. The CTA stages the particles of the tile and of every cell within
//     cell_div cells of it into shared memory.  Rows of cells along x are
//     contiguous in the sorted order and sorted by x, so each (y, z) row is one
//     copy.  Every staged position is shifted from its own cell to the middle of
//     the tile; the FP32 offsets stay small, so relative distances
//     keep full FP32 precision however large the tank is.  The origins lie on a
//     lattice whose spacing (Inst::oc) has few mantissa bits, so the shifts are
//     exact in FP32.
//  2. A warp takes a cluster of G particles (G = 2 or 4) that follow one
//     another along x in one row of the tile: compact in space, so that the
//     candidates near any of them are mostly near all of them.  For each row of
//     cells around, a binary search gives the exact x-window of the cluster.
//  3. Lanes test the windowed candidates, 32 at a time, against the G particles
//     in packed FP32x2 arithmetic; those within 2h of any of them are compacted
//     by ballot into ONE list for the cluster.
//  4. The pair arithmetic runs over that list, one candidate per lane, for all
//     G particles at once: a candidate's data is loaded and prepared once for G
//     pair terms, and two particles share each packed FP32x2 instruction.  A
//     candidate beyond 2h of a particle has its (1 - q/2) set to zero, which
//     makes its terms exactly zero.
//  5. The 32 lane sums of the cluster are combined by a value-splitting shuffle
//     butterfly and written out; nothing is carried between warps.
// A tile whose neighbourhood exceeds the staging buffer (compressed fluid, a clump) is
// halved until its parts fit (fluid of the 0.9 M-particle obstacle case compressed to
// 1.6 times its density: 3.20 -> 1.87 ms per step, against 3.02 ms staged in chunks by
// the kernel of pair_wide.cuh; the code for it costs the others 0.4 to 3 %).  A single cell whose neighbourhood does not, or a part
// that holds values a zero weight could not cancel (non-finite or huge), takes the
// same path with the candidates read from global memory and every term masked.
//
// Why this split: one list per particle, a group's particles spread over a cell of
// 2h (pair_wide.cuh), costs four ballots and prefix counts per 32 candidates, 900
// candidate tests per particle and a load of the candidate per pair term: 1.45e9
// warp instructions on the 0.9 M-particle obstacle case.  Rows of cross-section h
// leave 640 tests, one list per cluster a quarter of the ballots, and the pair terms
// evaluated for nothing (1.4 per useful one) cost less than the tests and stores
// they replace: 0.89e9 instructions, 1.98 -> 1.17 ms per pass (8.1 M particles:
// 19.4 -> 11.1 ms; h = 1.5 dp, 2.0 M particles: 3.38 -> 1.62 ms).
// What bounds it: issue slots and fixed latencies at 16 warps per SM (128
// registers); a list step of 32 candidates takes about 170 warp instructions for 4
// pair terms, 135 of them arithmetic, a step of the sweep about 50.
//
// Compensated sums: the lane sums (at most a few tens of terms each) are
// combined across lanes with Knuth's TwoSum, carrying the rounding error of
// every addition, so the result is the compensated sum of the lane partials.
#include <type_traits>

#include "device.cuh"
#include "rows.h"

namespace sph {

constexpr int kMaxRowsM = 96;  // staged rows of a tile: (tdim_y + 2 cell_div)(tdim_z + 2 cell_div)
constexpr int kMaxHome = 16;   // rows of the tile itself
constexpr int kMaxWin = 51;    // rows within cell_div of a particle's, (2 * 3 + 1)^2, and the end of the list
constexpr int kMaxParts = 12;  // pending halves of a tile: one for each halving, at most 4 + 3 + 3 (tdim <= 12, 6, 6)
constexpr int kList = 448;     // capacity of a warp's candidate list; drained when short of room

// Dynamic shared memory of a CTA of NW warps: staged A and B (with a dummy slot
// out of everything's reach) and type flags, then the warps' lists and windows.
constexpr int kOffB = (kStage + 1) * (int)sizeof(float4);  // byte offsets in it
constexpr int kOffF = 2 * kOffB;
constexpr int kOffWarp = (kOffF + kStage + 1 + 15) / 16 * 16;
constexpr int kWarpBytes = kList * (int)sizeof(int32_t) + (kMaxWin + 1) * (int)sizeof(int2);
__host__ __device__ __forceinline__ size_t mixed_dyn_smem(int NW) { return kOffWarp + (size_t)NW * kWarpBytes; }

// A neighbourhood and the staging buffer: it fits; the box was halved; a single cell, read from global memory.
enum : int32_t { kGlobal = 0, kFits = 1, kHalved = 2 };

struct PairSmem {
    int32_t item;   // tile, -1 when the queue is exhausted
    int32_t next;   // next cluster of the tile
    int32_t fit;    // kFits, kHalved or kGlobal
    int32_t wild;   // a staged value is not finite or huge: take the masked path
    int32_t nh;     // home rows
    int32_t box;    // the part of the tile in work (box_pack), 0: all of it
    int32_t nparts, parts[kMaxParts];  // the parts to come
    unsigned long long st_ff, st_visc, st_cand;  // work counts of this CTA
    int32_t pre[kMaxRowsM + 1];  // staged index of each row's first particle
    int32_t gs[kMaxRowsM];       // its sorted index
    int32_t hoff[kMaxHome], hlen[kMaxHome + 1];  // the tile's own run of each home row, from the staged run's start
    int32_t hyz[kMaxHome];                   // y | z << 16 of the home row in the tile
    int32_t hpre[kMaxHome + 1];              // clusters before each home row
};

__device__ __forceinline__ void two_sum(float &s, float &e, float x)
{
    // Knuth's TwoSum: s + x = t + err exactly, err accumulated in e.
    float t = s + x;
    float bp = t - s;
    float err = (s - (t - bp)) + (x - bp);
    s = t;
    e += err;
}

// FP32 constants of one instance, held in registers for a work item.
struct PairConst {
    float half_inv_h, mkF, rho0, inv_rho0, dfac, eta2, c0, nah, nahc0, sup2, cs;  // nah = -alpha h
    bool csound_const;
};

__device__ __forceinline__ PairConst pair_const(const Inst &I)
{
    PairConst k;
    k.half_inv_h = 0.5f * I.inv_hf;
    k.mkF = -I.massf * I.kFf;  // m_j F = mkF (1 - q/2)^3
    k.rho0 = I.rho0f;
    k.inv_rho0 = I.inv_rho0f;
    k.dfac = I.dfac;
    k.eta2 = I.eta2f;
    k.c0 = I.c0f;
    k.nah = -I.alphaf * I.hf;
    k.nahc0 = k.nah * I.c0f;
    k.sup2 = I.sup2f;
    k.cs = I.csf;
    k.csound_const = I.csound == SPH_CSOUND_CONSTANT;
    return k;
}

// ---------------------------------------------------------------------------
// Scalar path (one particle per warp)
// ---------------------------------------------------------------------------
struct PartI {
    float x, y, z, ux, uy, uz, rho, inv_rho;
    float Pr;   // P_i / rho_i
    float ndd;  // -2 delta h c0 (rho_i - rho0)
    float nac;  // -alpha h c_i
    bool fluid;
};

__device__ __forceinline__ PartI load_part(const PairConst &k, const float4 A, const float4 B, bool fluid)
{
    PartI p;
    p.x = A.x;
    p.y = A.y;
    p.z = A.z;
    p.ux = B.x;
    p.uy = B.y;
    p.uz = B.z;
    p.rho = k.rho0 + A.w;
    p.inv_rho = __fdividef(1.f, p.rho);
    p.Pr = B.w * p.inv_rho;
    p.ndd = -k.dfac * A.w;
    const float xi = fmaf(A.w, k.inv_rho0, 1.f);
    p.nac = k.csound_const ? k.nahc0 : k.nahc0 * xi * xi * xi;
    p.fluid = fluid;
    return p;
}

struct LaneAcc {
    float drho, ax, ay, az, mumax;
    float dd;  // delta term of Eq. 7 summed apart (SPH_DELTA_FULL_SUPPORT only)
};

// Pair term of neighbour j on particle i in FP32.  dx = x_i - x_j (home-cell
// relative), du = u_i - u_j.  grad_i W_ij = F (r_i - r_j) with
// F = -kF (1 - q/2)^3; Eq. 7 continuity (standard sign) and delta term between
// fluid particles; Eqs. 4-5 viscosity when u_ij . r_ij < 0; Eq. 3 momentum.
// For j = i (dx = du = 0) every term is exactly zero.  The running maximum is
// of mu / h (the caller scales it by h).  Returns bit 0 for a fluid-fluid pair
// (delta term evaluated) and bit 1 for an approaching pair (viscosity
// evaluated).  With DFS the delta term goes to acc.dd instead of acc.drho.
template <bool DFS>
__device__ __forceinline__ int pair_term_f(const PairConst &k, const PartI &p, const float4 a, const float4 bb,
                                           bool fluid_pair, LaneAcc &acc)
{
    const float dx = p.x - a.x, dy = p.y - a.y, dz = p.z - a.z;
    const float dux = p.ux - bb.x, duy = p.uy - bb.y, duz = p.uz - bb.z;
    const float r2 = dx * dx + dy * dy + dz * dz;
    const float r = r2 * rsqrtf(r2 + 1e-30f);  // 0 for j = i
    const float t = fmaf(-k.half_inv_h, r, 1.f);
    const float mF = k.mkF * (t * t * t);  // m_j F
    const float udr = dux * dx + duy * dy + duz * dz;  // u_ij . r_ij
    const float rho_j = k.rho0 + a.w;
    const float inv_rho_j = __fdividef(1.f, rho_j);
    // continuity: m_j (u_i - u_j) . grad_i W_ij = m F udr, plus between fluid
    // particles the delta term -m F 2 delta h c0 (rho_j - rho_i) / rho_j
    const float ud = DFS ? udr : (fluid_pair ? fmaf(-fmaf(k.dfac, a.w, p.ndd), inv_rho_j, udr) : udr);
    // viscosity (Eqs. 4-5): mu = h muh
    const float muh = udr * __fdividef(1.f, r2 + k.eta2);
    // evaluated on every lane: a batch of 32 pairs almost always holds an
    // approaching pair, so a branch would only add overhead; muh < 0 exactly
    // when u_ij . r_ij < 0, so min(muh, 0) switches the term on
    const float xj = fmaf(a.w, k.inv_rho0, 1.f);
    const float nac = k.csound_const ? p.nac + k.nahc0 : fmaf(k.nahc0 * (xj * xj), xj, p.nac);  // -alpha h (c_i + c_j)
    const float visc = nac * fminf(muh, 0.f) * __fdividef(1.f, p.rho + rho_j);
    // Eq. 3: a_i -= m_j ((P_i + P_j)/(rho_i rho_j) + Pi_ij) grad_i W_ij
    const float coef = mF * fmaf(fmaf(bb.w, p.inv_rho, p.Pr), inv_rho_j, visc);
    acc.drho = fmaf(mF, ud, acc.drho);
    if (DFS)
        acc.dd = fmaf(mF, fluid_pair ? -fmaf(k.dfac, a.w, p.ndd) * inv_rho_j : 0.f, acc.dd);
    acc.ax = fmaf(-coef, dx, acc.ax);
    acc.ay = fmaf(-coef, dy, acc.ay);
    acc.az = fmaf(-coef, dz, acc.az);
    acc.mumax = fmaxf(acc.mumax, muh);
    return (fluid_pair ? 1 : 0) | (udr < 0.f ? 2 : 0);  // pair classes for the work counts
}

// Positions of the G particles of a warp, negated and packed in pairs, for the
// candidate sweep: r_j - r_i is then one packed add, and one packed FP32x2
// instruction (sm_100 and later) advances the |r_ij|^2 < (2h)^2 test of two
// particles.  For G = 1 the scalar halves are used.
template <int G>
struct SweepPos {
    float2 nx[(G + 1) / 2], ny[(G + 1) / 2], nz[(G + 1) / 2];
};

template <int G>
__device__ __forceinline__ void hit_tests(const SweepPos<G> &sp, const float4 a, float sup2, bool (&hit)[G])
{
    if constexpr (G == 1) {
        const float dx = a.x + sp.nx[0].x, dy = a.y + sp.ny[0].x, dz = a.z + sp.nz[0].x;
        hit[0] = dx * dx + dy * dy + dz * dz < sup2;
    } else {
        const float2 ax = make_float2(a.x, a.x), ay = make_float2(a.y, a.y), az = make_float2(a.z, a.z);
#pragma unroll
        for (int q = 0; q < G / 2; ++q) {
            const float2 dx = __fadd2_rn(ax, sp.nx[q]), dy = __fadd2_rn(ay, sp.ny[q]), dz = __fadd2_rn(az, sp.nz[q]);
            const float2 d2 = __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __fmul2_rn(dx, dx)));
            hit[2 * q] = d2.x < sup2;
            hit[2 * q + 1] = d2.y < sup2;
        }
    }
}

__device__ __forceinline__ float rcp_ftz(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float sqrt_ftz(float x)
{
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// A value the compiler keeps in its register instead of computing it again
// wherever it is used (lane and per-warp offsets in the inner loops).
__device__ __forceinline__ int keep(int v)
{
    asm volatile("" : "+r"(v));
    return v;
}
// Shared-memory accesses of the inner loops by 32-bit address (the window base
// stays in a register; immediate offset OFF).
template <int OFF>
__device__ __forceinline__ float4 lds_f4(uint32_t a)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4 + %5];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(a), "n"(OFF)
                 : "memory");
    return v;
}
__device__ __forceinline__ int32_t lds_i32(uint32_t a)
{
    int32_t v;
    asm volatile("ld.shared.s32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ float lds_f32(uint32_t a)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ int2 lds_i2(uint32_t a)
{
    int2 v;
    asm volatile("ld.shared.v2.s32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a) : "memory");
    return v;
}
template <int OFF>
__device__ __forceinline__ uint32_t lds_u8(uint32_t a)
{
    uint32_t v;
    asm volatile("ld.shared.u8 %0, [%1 + %2];" : "=r"(v) : "r"(a), "n"(OFF) : "memory");
    return v;
}
__device__ __forceinline__ void sts_i32(uint32_t a, int32_t v)
{
    asm volatile("st.shared.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void sts_i2(uint32_t a, int2 v)
{
    asm volatile("st.shared.v2.s32 [%0], {%1, %2};" ::"r"(a), "r"(v.x), "r"(v.y) : "memory");
}
__device__ __forceinline__ float2 dup2(float v) { return make_float2(v, v); }

// Two particles of a cluster.  Their velocities are negated, as their positions
// are in pair_cluster, so that differences are additions.
struct PackI {
    float2 d, rho, inv, Pr, nac;  // rho - rho0, rho, 1/rho, P/rho, -alpha h c
    float2 nux, nuy, nuz;
};
struct PackAcc {
    float2 drho, ax, ay, az, mu;  // in units of t^3 (the caller scales by m F(0)); mu / h
    float2 dd;                    // delta term of Eq. 7 summed apart (SPH_DELTA_FULL_SUPPORT only)
};
// One candidate.
struct CandJ {
    float x, y, z, ux, uy, uz, d, rho, inv, vd, P, nac;  // vd = 2 delta h c0 / rho, 0 for a boundary particle
};

__device__ __forceinline__ CandJ load_cand(const PairConst &k, const float4 a, const float4 b, bool fluid)
{
    CandJ j;
    const float xj = fmaf(a.w, k.inv_rho0, 1.f);
    j.x = a.x;
    j.y = a.y;
    j.z = a.z;
    j.ux = b.x;
    j.uy = b.y;
    j.uz = b.z;
    j.d = a.w;
    j.rho = k.rho0 + a.w;
    j.inv = rcp_ftz(j.rho);
    j.vd = fluid ? k.dfac * j.inv : 0.f;
    j.P = b.w;
    j.nac = k.csound_const ? k.nahc0 : k.nahc0 * xj * xj * xj;
    return j;
}

// r_ij = r_j - r_i and |r_ij|^2 for two particles i (negated positions); the
// same arithmetic in the candidate sweep and in the pair terms, so that both
// agree on which pairs lie within 2h.  The first operations take the candidate's
// scalar with each half: a packed operand (v, v) would cost two moves.
__device__ __forceinline__ float2 dist2_pack(float x, float y, float z, float2 nx, float2 ny, float2 nz, float2 &dx,
                                             float2 &dy, float2 &dz)
{
    dx = make_float2(x + nx.x, x + nx.y);
    dy = make_float2(y + ny.x, y + ny.y);
    dz = make_float2(z + nz.x, z + nz.y);
    return __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __fmul2_rn(dx, dx)));
}

// The pair terms of candidate j on two particles.  fs: see below (ALLF: all of
// the cluster are fluid), fj: the candidate is fluid.  SAFE: the terms are
// masked one by one instead of through a zero t.  Returns the masks of
// interacting pairs (bits 0, 1) and of approaching ones among them (bits 2, 3).
template <bool ALLF, bool DFS, bool SAFE>
__device__ __forceinline__ unsigned pair_terms_pack(const PairConst &k, const PackI &p, float2 nx, float2 ny, float2 nz,
                                                    const CandJ &j, float2 fs, bool fj, PackAcc &a)
{
    float2 dx, dy, dz;
    const float2 r2 = dist2_pack(j.x, j.y, j.z, nx, ny, nz, dx, dy, dz);
    // pairs of two boundary particles do not interact: fs is (2h)^2 for a fluid particle, 0 for a boundary one
    const bool p0 = r2.x < (ALLF || fj ? k.sup2 : fs.x), p1 = r2.y < (ALLF || fj ? k.sup2 : fs.y);
    float2 t = make_float2(fmaf(-k.half_inv_h, sqrt_ftz(r2.x), 1.f), fmaf(-k.half_inv_h, sqrt_ftz(r2.y), 1.f));
    t.x = p0 ? t.x : 0.f;
    t.y = p1 ? t.y : 0.f;
    const float2 t3 = __fmul2_rn(__fmul2_rn(t, t), t);  // m_j F / (m F(0))
    const float2 dux = make_float2(j.ux + p.nux.x, j.ux + p.nux.y), duy = make_float2(j.uy + p.nuy.x, j.uy + p.nuy.y),
                 duz = make_float2(j.uz + p.nuz.x, j.uz + p.nuz.y);
    const float2 udr = __ffma2_rn(duz, dz, __ffma2_rn(duy, dy, __fmul2_rn(dux, dx)));  // u_ij . r_ij
    // Eq. 7: u_ij . r_ij, plus between fluid particles the delta term 2 delta h c0 (rho_i - rho_j) / rho_j
    float2 g = make_float2(p.d.x - j.d, p.d.y - j.d);
    if (!ALLF) {
        g.x = fs.x > 0.f ? g.x : 0.f;
        g.y = fs.y > 0.f ? g.y : 0.f;
    }
    // Eqs. 4-5: mu = h muh; min(muh, 0) switches the viscosity on for approaching pairs
    float2 ire = make_float2(rcp_ftz(r2.x + k.eta2), rcp_ftz(r2.y + k.eta2));
    ire.x = p0 ? ire.x : 0.f;  // a masked pair leaves the running maximum of mu alone
    ire.y = p1 ? ire.y : 0.f;
    const float2 muh = __fmul2_rn(udr, ire);
    const float2 mn = make_float2(fminf(muh.x, 0.f), fminf(muh.y, 0.f));
    const float2 ir = make_float2(rcp_ftz(p.rho.x + j.rho), rcp_ftz(p.rho.y + j.rho));
    const float2 nac = make_float2(p.nac.x + j.nac, p.nac.y + j.nac);
    const float2 visc = __fmul2_rn(__fmul2_rn(nac, mn), ir);
    // Eq. 3: a_i += m_j F ((P_i + P_j)/(rho_i rho_j) + Pi_ij) r_ij
    float2 coef = make_float2(fmaf(fmaf(j.P, p.inv.x, p.Pr.x), j.inv, visc.x), fmaf(fmaf(j.P, p.inv.y, p.Pr.y), j.inv, visc.y));
    coef = __fmul2_rn(coef, t3);
    if (SAFE) {
        coef.x = p0 ? coef.x : 0.f;
        coef.y = p1 ? coef.y : 0.f;
        const float2 del = make_float2(g.x * j.vd, g.y * j.vd);
        float2 c = __fmul2_rn(t3, DFS ? udr : __fadd2_rn(udr, del));
        a.drho = __fadd2_rn(a.drho, make_float2(p0 ? c.x : 0.f, p1 ? c.y : 0.f));
        if (DFS) {
            c = __fmul2_rn(t3, del);
            a.dd = __fadd2_rn(a.dd, make_float2(p0 ? c.x : 0.f, p1 ? c.y : 0.f));
        }
    } else if (DFS) {
        a.drho = __ffma2_rn(t3, udr, a.drho);
        a.dd = __ffma2_rn(t3, make_float2(g.x * j.vd, g.y * j.vd), a.dd);
    } else {
        a.drho = __ffma2_rn(t3, make_float2(fmaf(g.x, j.vd, udr.x), fmaf(g.y, j.vd, udr.y)), a.drho);
    }
    a.ax = __ffma2_rn(coef, dx, a.ax);
    a.ay = __ffma2_rn(coef, dy, a.ay);
    a.az = __ffma2_rn(coef, dz, a.az);
    a.mu.x = fmaxf(a.mu.x, muh.x);
    a.mu.y = fmaxf(a.mu.y, muh.y);
    return (p0 ? 1u : 0u) | (p1 ? 2u : 0u) | (p0 && udr.x < 0.f ? 4u : 0u) | (p1 && udr.y < 0.f ? 8u : 0u);
}

// Combination of the 32 lane sums of the K = 4 G values of a cluster by a
// value-splitting butterfly: at each of the first log2 K levels a lane keeps
// half of its values and adds its partner's copies of them, so a level moves
// half as many values as the one before; the remaining levels add the one value
// left.  Lane (32 / K) m then holds, for one value `idx`, the total and (COMP)
// its error term.
template <int K, bool COMP>
__device__ __forceinline__ int warp_split_totals(float (&v)[K], float (&e)[K], int lane)
{
    int idx = 0;
#pragma unroll
    for (int k = K, o = 16; k > 1; k >>= 1, o >>= 1) {
        const bool upper = (lane & o) != 0;
        const int half = k >> 1;
        idx += upper ? half : 0;
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const float keep = upper ? v[i + half] : v[i];
            const float send = upper ? v[i] : v[i + half];
            const float recv = __shfl_xor_sync(0xffffffffu, send, o);
            if (COMP) {
                float ee = 0.f;
                if (k < K) {  // the lanes start without error terms
                    const float ke = upper ? e[i + half] : e[i];
                    const float se = upper ? e[i] : e[i + half];
                    ee = ke + __shfl_xor_sync(0xffffffffu, se, o);
                }
                float sum = keep;
                two_sum(sum, ee, recv);
                v[i] = sum;
                e[i] = ee;
            } else {
                v[i] = keep + recv;
            }
        }
    }
#pragma unroll
    for (int o = 16 / K; o > 0; o >>= 1) {
        const float recv = __shfl_xor_sync(0xffffffffu, v[0], o);
        if (COMP) {
            float ee = e[0] + __shfl_xor_sync(0xffffffffu, e[0], o);
            two_sum(v[0], ee, recv);
            e[0] = ee;
        } else {
            v[0] += recv;
        }
    }
    return idx;
}

// Geometry of the tile a CTA works on.
struct TileGeo {
    int32_t t0[3];   // first cell
    int32_t cen[3];  // origin of the frame, in half cells: the tile's centre, or a corner of its middle cell
    int mid[2];      // its distance from the first cell along y and z
    int nry;         // staged rows along y
    int32_t total;   // staged particles
    int row0, row1;  // (dy & 0xff) | dz << 8 of this lane's row around a particle's (the first 32, the next)
    float dy0, dz0;  // distance of the true cell lattice from the frame's at the frame's origin
};

// A part of a tile: first cell from the tile's and cells per axis, 4 bits each.
__device__ __forceinline__ int32_t box_pack(int ox, int oy, int oz, int dx, int dy, int dz)
{
    return ox | (oy << 4) | (oz << 8) | (dx << 12) | (dy << 16) | (dz << 20);
}
__device__ __forceinline__ int box_off(int32_t box, int a) { return (box >> (4 * a)) & 15; }
__device__ __forceinline__ int box_dim(int32_t box, int a) { return (box >> (12 + 4 * a)) & 15; }

// The two halves of a box along its longest axis (the last of the longest: the
// clusters run along x); false for a single cell.
__device__ __forceinline__ bool box_halves(int32_t box, int dx, int dy, int dz, int32_t (&half)[2])
{
    const int a = dz >= max(dx, dy) ? 2 : (dy >= dx ? 1 : 0);
    const int d = a == 2 ? dz : (a == 1 ? dy : dx), cut = d / 2;
    if (d < 2)
        return false;
    const int32_t whole = box_pack(box_off(box, 0), box_off(box, 1), box_off(box, 2), dx, dy, dz);
    half[0] = whole - ((d - cut) << (12 + 4 * a));
    half[1] = whole - (cut << (12 + 4 * a)) + (cut << (4 * a));
    return true;
}

// One cluster (G particles of one home row) by one warp.  STG: candidates from
// the staged copy; otherwise from global memory, with every term masked.
template <int NW, int G, bool COMP, bool STAT, bool DFS, bool STG>
__device__ __forceinline__ void pair_cluster(const Bufs &b, const Inst &I, const PairConst &kc, const TileGeo &T, int kdiv,
                                             int q, uint32_t st, uint32_t list, int lane, PairSmem &S,
                                             unsigned (&lc)[2], unsigned long long &wc_cand)
{
    constexpr int P = G / 2;
    const unsigned lt = (1u << lane) - 1u;
    const uint32_t win = list + kList * (uint32_t)sizeof(int32_t);  // this warp's windows follow its list
    const float4 *gA = reinterpret_cast<const float4 *>(b.sA);
    const float4 *gB = reinterpret_cast<const float4 *>(b.sB);
    const int32_t dummy = STG ? kStage : -1;
    // position and density offset of candidate t in the tile's frame
    auto ck = [&](int32_t t) -> int32_t {
        return SPH_BOUNDS_OK(STG ? t >= 0 && t <= kStage : t >= -1 && t < b.misc[0], &b.misc[2]) ? t : dummy;
    };
    auto cand_a = [&](int32_t t_) -> float4 {
        const int32_t t = ck(t_);
        if (STG)
            return lds_f4<0>(st + 16u * (uint32_t)t);
        if (t < 0)
            return make_float4(1e15f, 1e15f, 1e15f, 0.f);
        float4 a = gA[t];
        int cx, cy, cz;
        decompose(I, b.scell[t], cx, cy, cz);
        a.x += (float)(2 * cx + I.centred - T.cen[0]) * I.ohf;
        a.y += (float)(2 * cy + I.centred - T.cen[1]) * I.ohf;
        a.z += (float)(2 * cz + I.centred - T.cen[2]) * I.ohf;
        return a;
    };
    auto cand_x = [&](int32_t t) -> float { return STG ? lds_f32(st + 16u * (uint32_t)ck(t)) : cand_a(t).x; };
    auto cand_b = [&](int32_t t_) -> float4 {
        const int32_t t = ck(t_);
        if (STG)
            return lds_f4<kOffB>(st + 16u * (uint32_t)t);
        return t < 0 ? make_float4(0.f, 0.f, 0.f, 0.f) : gB[t];
    };
    auto cand_f = [&](int32_t t_) -> bool {
        const int32_t t = ck(t_);
        return STG ? lds_u8<kOffF>(st + (uint32_t)t) == T_FLUID : (t >= 0 && b.sflag[t] == T_FLUID);
    };

    // home row of cluster q, its particles
    const int nh = S.nh;
    const int rr = __popc(__ballot_sync(0xffffffffu, lane < nh && S.hpre[min(lane, nh - 1) + 1] <= q));
    const int k0 = (q - S.hpre[rr]) * G;
    const int nreal = min(G, S.hlen[rr] - k0);  // a short cluster repeats its last particle; nothing is stored for it
    if (!check_ok(rr < nh && k0 >= 0 && nreal > 0, &b.misc[2]))
        return;
    const int hy = S.hyz[rr] & 0xffff, hz = S.hyz[rr] >> 16;
    const int hrow = (hz + kdiv) * T.nry + hy + kdiv;
    // staged slot and sorted index, both from the row's one staged run
    const int32_t s0 = S.gs[hrow] + S.hoff[rr] + k0;
    const int32_t i0 = STG ? S.pre[hrow] + S.hoff[rr] + k0 : s0;
    float2 nx[P], ny[P], nz[P];
    unsigned fl = 0;  // bit g: particle g is fluid
#pragma unroll
    for (int g = 0; g < G; ++g) {
        const int32_t t = i0 + min(g, nreal - 1);
        const float4 a = cand_a(t);
        (g & 1 ? nx[g / 2].y : nx[g / 2].x) = -a.x;
        (g & 1 ? ny[g / 2].y : ny[g / 2].x) = -a.y;
        (g & 1 ? nz[g / 2].y : nz[g / 2].x) = -a.z;
        fl |= (cand_f(t) ? 1u : 0u) << g;
    }
    constexpr unsigned kAll = (1u << G) - 1u;

    // Exact x-windows: a candidate of a row can lie within 2h of particle g only
    // if |x_j - x_g| <= sqrt((2h)^2 - d^2), d the distance from g to the row's
    // y-z cross-section; the windows of the G particles are merged.  One lane per
    // row; the non-empty windows are listed in `win`.
    const int nrow = (2 * kdiv + 1) * (2 * kdiv + 1);
    int nwin = 0;
    for (int r0 = 0; r0 < nrow; r0 += 32) {
        int32_t lo = 0, hi = 0;
        if (r0 + lane < nrow) {
            const int dyz = r0 ? T.row1 : T.row0;
            const int dy = (int)(int8_t)(dyz & 0xff), dz = dyz >> 8;
            const int row = hrow + dz * T.nry + dy;
            int32_t ra = S.pre[row], rb = S.pre[row + 1];
            if (!STG) {
                rb = S.gs[row] + (rb - ra);
                ra = S.gs[row];
            }
            if (ra < rb) {
                // centre and half width of the cross-section
                const float hc = 0.5f * kc.cs, eps = 2e-6f * kc.cs;
                const float yc = (float)(2 * (hy + dy) + 1 - T.mid[0]) * hc + T.dy0;
                const float zc = (float)(2 * (hz + dz) + 1 - T.mid[1]) * hc + T.dz0;
                float xl = 3.0e38f, xh = -3.0e38f;
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    const float px = -(g & 1 ? nx[g / 2].y : nx[g / 2].x), py = -(g & 1 ? ny[g / 2].y : ny[g / 2].x),
                                pz = -(g & 1 ? nz[g / 2].y : nz[g / 2].x);
                    const float ey = fmaxf(fabsf(py - yc) - hc - eps, 0.f);
                    const float ez = fmaxf(fabsf(pz - zc) - hc - eps, 0.f);
                    const float rem = kc.sup2 - ey * ey - ez * ez;
                    if (rem > 0.f) {
                        const float w = sqrt_ftz(rem) * 1.0001f + eps;
                        xl = fminf(xl, px - w);
                        xh = fmaxf(xh, px + w);
                    }
                }
                if (xl <= xh) {
                    int32_t a0 = ra, a1 = rb;
                    while (a0 < a1) {
                        const int32_t m = (a0 + a1) >> 1;
                        if (cand_x(m) < xl)
                            a0 = m + 1;
                        else
                            a1 = m;
                    }
                    lo = a0;
                    a1 = rb;
                    while (a0 < a1) {
                        const int32_t m = (a0 + a1) >> 1;
                        if (cand_x(m) <= xh)
                            a0 = m + 1;
                        else
                            a1 = m;
                    }
                    hi = a0;
                }
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, lo < hi);
        if (lo < hi)
            sts_i2(win + 8u * (nwin + __popc(m & lt)), make_int2(lo, hi));
        nwin += __popc(m);
        if (lane == 0)
            sts_i2(win + 8u * nwin, make_int2(1, 1));  // an empty window ends the list (an odd one out is paired with it)
        __syncwarp();
        if (STAT) {
            const int c = warp_sum(hi - lo);
            if (lane == 0)
                wc_cand += (unsigned long long)c;
        }
    }
    __syncwarp();

    PackAcc acc[P];
#pragma unroll
    for (int h = 0; h < P; ++h)
        acc[h] = PackAcc{dup2(0.f), dup2(0.f), dup2(0.f), dup2(0.f), dup2(0.f), dup2(0.f)};
    int nn[G], np[G];
    unsigned nbits = 0;  // bit g: particle g has a boundary particle within 2h
#pragma unroll
    for (int g = 0; g < G; ++g)
        nn[g] = np[g] = 0;

    // Pair terms of list entries [0, n), n a multiple of 32.
    auto evaluate = [&](int n) {
        PackI pi[P];
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const int32_t t = i0 + min(g, nreal - 1);
            const float d = cand_a(t).w;
            const float4 bb = cand_b(t);
            const float rho = kc.rho0 + d, inv = rcp_ftz(rho), xi = fmaf(d, kc.inv_rho0, 1.f);
            const float nac = kc.csound_const ? kc.nahc0 : kc.nahc0 * xi * xi * xi;
            PackI &p = pi[g / 2];
#define SPH_SET(f, val) (g & 1 ? p.f.y : p.f.x) = (val)
            SPH_SET(d, d);
            SPH_SET(rho, rho);
            SPH_SET(inv, inv);
            SPH_SET(Pr, bb.w * inv);
            SPH_SET(nac, nac);
            SPH_SET(nux, -bb.x);
            SPH_SET(nuy, -bb.y);
            SPH_SET(nuz, -bb.z);
#undef SPH_SET
        }
        float2 fs[P];
#pragma unroll
        for (int h = 0; h < P; ++h)
            fs[h] = make_float2((fl >> (2 * h)) & 1u ? kc.sup2 : 0.f, (fl >> (2 * h + 1)) & 1u ? kc.sup2 : 0.f);
        auto steps = [&](auto allf) {
            constexpr bool ALLF = decltype(allf)::value;
            uint32_t at = list + 4u * lane;
            const uint32_t end = at + 4u * n;
#pragma unroll 1
            for (; at != end; at += 128u) {
                const int32_t t = lds_i32(at);
                const bool fj = cand_f(t);
                const CandJ j = load_cand(kc, cand_a(t), cand_b(t), fj);
#pragma unroll
                for (int h = 0; h < P; ++h) {
                    const unsigned m = pair_terms_pack<ALLF, DFS, !STG>(kc, pi[h], nx[h], ny[h], nz[h], j, fs[h], fj,
                                                                        acc[h]);
                    if (DFS && !fj)
                        nbits |= (m & 3u) << (2 * h);
                    if (STAT) {
                        float2 dx, dy, dz;
                        const float2 r2 = dist2_pack(j.x, j.y, j.z, nx[h], ny[h], nz[h], dx, dy, dz);
                        nn[2 * h] += r2.x < kc.sup2;
                        nn[2 * h + 1] += r2.y < kc.sup2;
                        np[2 * h] += m & 1u;
                        np[2 * h + 1] += (m >> 1) & 1u;
                        const bool f0 = (fl >> (2 * h)) & 1u, f1 = (fl >> (2 * h + 1)) & 1u;
                        const bool v0 = 2 * h < nreal, v1 = 2 * h + 1 < nreal;  // a repeated particle is not counted
                        lc[0] += (v0 && f0 && fj && (m & 1u)) + (v1 && f1 && fj && (m & 2u));
                        lc[1] += (v0 && (m & 4u)) + (v1 && (m & 8u));
                    }
                }
            }
        };
        if (fl == kAll)
            steps(std::true_type{});
        else
            steps(std::false_type{});
    };

    // Candidate sweep: two windows at a time, 16 lanes each.
    int cnt = 0;
    auto drain = [&]() {  // the full batches of the list; the rest moves to its front
        __syncwarp();
        const int full = cnt & ~31;
        evaluate(full);
        __syncwarp();
        const int32_t rest = lds_i32(list + 4u * (full + lane));
        __syncwarp();
        sts_i32(list + 4u * lane, rest);
        cnt -= full;
        __syncwarp();
    };
    constexpr int kChunk = (kList - 96) / 32;  // steps between the checks for room
    for (int w0 = 0; w0 < nwin; w0 += 2) {
        const int2 w = lds_i2(win + 8u * (w0 + (lane >> 4)));
        const int32_t last = w.y - 1;
        int32_t t = w.x + (lane & 15);
        int steps = __reduce_max_sync(0xffffffffu, (unsigned)(w.y - w.x + 15) >> 4);
        while (steps > 0) {
            const int n = min(steps, kChunk);
            steps -= n;
            // room for these steps and for the padding of the last batch
            if (cnt + 32 * n > kList - 32)
                drain();
#pragma unroll 1
            for (int k = 0; k < n; ++k, t += 16) {
                const int32_t tc = min(t, last);
                const float4 a = cand_a(tc);
                float near = 3.0e38f;
#pragma unroll
                for (int h = 0; h < P; ++h) {
                    float2 dx, dy, dz;
                    const float2 r2 = dist2_pack(a.x, a.y, a.z, nx[h], ny[h], nz[h], dx, dy, dz);
                    near = fminf(near, fminf(r2.x, r2.y));
                }
                bool take = near < kc.sup2 && t <= last;
                // clusters of boundary particles interact with fluid only
                if (!STAT && fl == 0u)
                    take = take && cand_f(tc);
                const unsigned m = __ballot_sync(0xffffffffu, take);
                const int at = cnt + __popc(m & lt);
                if (take && SPH_BOUNDS_OK(at < kList && (!STG || (t >= 0 && t < kStage)), &b.misc[2]))
                    sts_i32(list + 4u * at, t);
                cnt += __popc(m);
            }
        }
    }
    __syncwarp();
    if (SPH_BOUNDS_OK(cnt + lane < kList, &b.misc[2]))
        sts_i32(list + 4u * (cnt + lane), dummy);  // pads the last batch
    __syncwarp();
    evaluate((cnt + 31) & ~31);

    // totals and write-out
    constexpr int K = 4 * G;
    float v[K], e[K];
#pragma unroll
    for (int g = 0; g < G; ++g) {
        const PackAcc &A = acc[g / 2];
        v[4 * g + 0] = g & 1 ? A.drho.y : A.drho.x;
        v[4 * g + 1] = g & 1 ? A.ax.y : A.ax.x;
        v[4 * g + 2] = g & 1 ? A.ay.y : A.ay.x;
        v[4 * g + 3] = g & 1 ? A.az.y : A.az.x;
    }
    const int idx = warp_split_totals<K, COMP>(v, e, lane);
    const int gsel = idx >> 2, c = idx & 3;
    float sum = v[0], err = COMP ? e[0] : 0.f;
    if (DFS) {
        // the delta term only with a fluid-only support
        const unsigned nball = __reduce_or_sync(0xffffffffu, nbits);
#pragma unroll
        for (int g = 0; g < G; ++g) {
            float dv = g & 1 ? acc[g / 2].dd.y : acc[g / 2].dd.x, de = 0.f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const float recv = __shfl_xor_sync(0xffffffffu, dv, o);
                float ee = de + __shfl_xor_sync(0xffffffffu, de, o);
                two_sum(dv, ee, recv);
                de = ee;
            }
            if (gsel == g && c == 0 && !((nball >> g) & 1u)) {
                two_sum(sum, err, dv);
                err += de;
            }
        }
    }
    if ((lane & (32 / K - 1)) == 0 && gsel < nreal) {
        float val = kc.mkF * (sum + err);
        if (c == 3 && ((fl >> gsel) & 1u))
            val -= I.gf;
        reinterpret_cast<float *>(b.deriv)[4 * (size_t)(s0 + gsel) + ((c + 3) & 3)] = val;  // (a, D rho)
    }
    float mu = 0.f;
#pragma unroll
    for (int g = 0; g < G; ++g) {
        // non-negative floats order like their bits
        const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(g & 1 ? acc[g / 2].mu.y : acc[g / 2].mu.x));
        mu = lane == g ? __uint_as_float(m) : mu;
    }
    if (lane < nreal)
        reinterpret_cast<float *>(b.mumax)[s0 + lane] = I.hf * mu;
    if (STAT) {
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const int a = warp_sum(nn[g]), p = warp_sum(np[g]);
            if (lane == 0 && g < nreal) {
                // the particle's own pair comes off: a hit, and evaluated for a fluid particle
                b.nneigh[s0 + g] = a - 1;
                b.npair[s0 + g] = p - (int)((fl >> g) & 1u);
                b.ncand[s0 + g] = T.total;
                lc[0] -= (fl >> g) & 1u;  // the own pair of a fluid particle was counted
            }
        }
    }
    __syncwarp();
}

// The path of the rare tiles, kept out of line so that it costs the others no
// registers.
template <int NW, int G, bool COMP, bool STAT, bool DFS>
__device__ __noinline__ void pair_cluster_global(const Bufs &b, const Inst &I, const TileGeo &T, int kdiv, int q,
                                                 uint32_t list, int lane, PairSmem &S, unsigned (&lc)[2],
                                                 unsigned long long &wc_cand)
{
    pair_cluster<NW, G, COMP, STAT, DFS, false>(b, I, pair_const(I), T, kdiv, q, 0u, list, lane, S, lc, wc_cand);
}

// The pair pass of one CTA: pulls tiles from the work queue b.misc[3] until it
// is exhausted.  dyn: the dynamic shared memory, S: the CTA's bookkeeping.
template <int NW, int G, bool COMP, bool STAT, bool DFS>
__device__ __forceinline__ void pair_mixed_body(const Bufs &b, int ninst, int kdiv, unsigned char *dyn, PairSmem &S)
{
    float4 *stA = reinterpret_cast<float4 *>(dyn), *stB = reinterpret_cast<float4 *>(dyn + kOffB);
    uint8_t *stF = dyn + kOffF;
    const int tid = threadIdx.x, lane = keep(tid & 31), wib = keep(tid >> 5);
    const uint32_t st = keep(static_cast<uint32_t>(__cvta_generic_to_shared(dyn)));
    const uint32_t list = keep(st + kOffWarp + wib * kWarpBytes);  // this warp's list and windows
    const float4 *gA = reinterpret_cast<const float4 *>(b.sA);
    const float4 *gB = reinterpret_cast<const float4 *>(b.sB);
    const int32_t n_tiles = b.misc[4];
    unsigned lc[2] = {0u, 0u};
    unsigned long long wc_cand = 0;
    const int side = 2 * kdiv + 1;
    const int row0 = ((lane % side - kdiv) & 0xff) | ((lane / side - kdiv) << 8);
    const int row1 = (((lane + 32) % side - kdiv) & 0xff) | (((lane + 32) / side - kdiv) << 8);
    if (tid == 0) {
        S.st_ff = 0ull;
        S.st_visc = 0ull;
        S.st_cand = 0ull;
        S.nparts = 0;
        stA[kStage] = make_float4(1e15f, 1e15f, 1e15f, 0.f);  // the dummy: beyond 2h of everything
        stB[kStage] = make_float4(0.f, 0.f, 0.f, 0.f);
        stF[kStage] = T_FLUID;
    }

    for (;;) {
        if (tid == 0 && S.nparts > 0) {
            S.box = S.parts[--S.nparts];
        } else if (tid == 0) {
            S.box = 0;
            const int32_t item = atomicAdd(&b.misc[3], 1);
            int32_t t = item < n_tiles && check_ok(n_tiles <= b.ntiles, &b.misc[2]) ? b.tiles[item] : -1;
            if (!check_ok(t >= -1 && t < b.ntiles, &b.misc[2]))
                t = -1;
            S.item = t;
        }
        __syncthreads();  // and every warp is done with the previous tile
        const int32_t tile = S.item;
        if (tile < 0)
            break;
        const Inst &I = b.inst[inst_of_tile(b.inst, ninst, tile)];
        const PairConst kc = pair_const(I);
        TileGeo T;
        T.row0 = row0;
        T.row1 = row1;
        {
            const int32_t lt = tile - I.tile_base;
            const int32_t q = lt / I.ntile[0];
            T.t0[0] = (lt - q * I.ntile[0]) * I.tdim[0];
            T.t0[2] = q / I.ntile[1];
            T.t0[1] = (q - T.t0[2] * I.ntile[1]) * I.tdim[1];
            T.t0[2] *= I.tdim[2];
        }
        const int32_t box = S.box;
        int dim[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            T.t0[a] += box_off(box, a);
            dim[a] = box ? box_dim(box, a) : I.tdim[a];
            T.cen[a] = 2 * T.t0[a] + (I.centred ? dim[a] : dim[a] & ~1);
        }
        T.mid[0] = T.cen[1] - 2 * T.t0[1];
        T.mid[1] = T.cen[2] - 2 * T.t0[2];
        T.nry = dim[1] + 2 * kdiv;
        T.dy0 = (float)(0.5 * T.cen[1] * (I.cs - I.oc));
        T.dz0 = (float)(0.5 * T.cen[2] * (I.cs - I.oc));
        const int nrow = T.nry * (dim[2] + 2 * kdiv), nh = dim[1] * dim[2];
        const int x0 = max(T.t0[0] - kdiv, 0), x1 = min(T.t0[0] + dim[0] + kdiv, I.n[0]);
        // the staged rows, one thread per row: the only reads of the cell starts
        for (int r = tid; r < nrow; r += blockDim.x) {
            const int zr = r / T.nry, hz = zr - kdiv, hy = r - zr * T.nry - kdiv;
            const int z = T.t0[2] + hz, y = T.t0[1] + hy;
            const bool home = hz >= 0 && hz < dim[2] && hy >= 0 && hy < dim[1];
            RowRun run = {0, 0, 0, 0};
            if (z >= 0 && z < I.n[2] && y >= 0 && y < I.n[1]) {
                const int32_t *row = b.cell_start + (I.cell_base + (z * I.n[1] + y) * I.n[0]);
                const int32_t a = row[x0], e = row[x1];
                const int32_t ha = home ? row[T.t0[0]] : a, he = home ? row[min(T.t0[0] + dim[0], I.n[0])] : a;
                check_ok(row_run(a, e, ha, he, min(b.misc[0], b.N), run), &b.misc[2]);
            }
            S.gs[r] = run.gs;
            S.pre[r + 1] = run.n;
            if (home) {
                const int h = hz * dim[1] + hy;
                S.hoff[h] = run.hoff;
                S.hlen[h] = run.hlen;
                S.hyz[h] = hy | (hz << 16);
            }
        }
        if (tid == 0) {
            S.next = 0;
            S.wild = 0;
            S.nh = nh;
        }
        __syncthreads();
        if (wib == 0) {
            // the tile fits if no row is longer than the buffer (so that the sums cannot
            // overflow) and the sum is not either: then every slot lies in the buffer
            int carry = 0;
            bool fit = true;
            for (int r0 = 0; r0 < nrow; r0 += 32) {
                const int r = r0 + lane;
                int x = r < nrow ? S.pre[r + 1] : 0;
                fit = fit && x <= kStage;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, x, o);
                    if (lane >= o)
                        x += y;
                }
                if (r < nrow)
                    S.pre[r + 1] = carry + x;
                carry += __shfl_sync(0xffffffffu, x, 31);
            }
            fit = __all_sync(0xffffffffu, fit) && carry <= kStage;
            if (lane == 0) {
                S.pre[0] = 0;
                S.fit = fit ? kFits : kGlobal;
                int32_t half[2];
                if (!fit && box_halves(box, min(dim[0], I.n[0] - T.t0[0]), min(dim[1], I.n[1] - T.t0[1]),
                                       min(dim[2], I.n[2] - T.t0[2]), half) &&
                    check_ok(S.nparts + 2 <= kMaxParts, &b.misc[2])) {
                    S.parts[S.nparts++] = half[1];
                    S.parts[S.nparts++] = half[0];
                    S.fit = kHalved;
                }
            }
        } else if (wib == 1) {
            int x = lane < nh ? (S.hlen[lane] + G - 1) / G : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o)
                    x += y;
            }
            if (lane < nh)
                S.hpre[lane + 1] = x;
            if (lane == 0)
                S.hpre[0] = 0;
        }
        __syncthreads();
        T.total = S.pre[nrow];
        const int nclus = S.hpre[nh];
        const bool fits = S.fit == kFits;
        if (S.fit == kHalved)
            continue;
        if (fits) {
            bool wild = false;
            const float lim = 1e15f, dmin = -0.5f * kc.rho0;
            for (int r = wib; r < nrow; r += NW) {
                const int32_t p0 = S.pre[r], len = S.pre[r + 1] - p0, g0 = S.gs[r];
                if (len == 0)
                    continue;
                const int zr = r / T.nry;
                const int y = T.t0[1] + (r - zr * T.nry) - kdiv, z = T.t0[2] + zr - kdiv;
                const float sy = (float)(2 * y + I.centred - T.cen[1]) * I.ohf, sz = (float)(2 * z + I.centred - T.cen[2]) * I.ohf;
                const int32_t row = I.cell_base + (z * I.n[1] + y) * I.n[0], sx = I.centred - T.cen[0];
#pragma unroll 3
                for (int32_t l = lane; l < len; l += 32) {
                    const int32_t j = g0 + l;
                    float4 a = gA[j];
                    const float4 v = gB[j];
                    const uint8_t f = b.sflag[j];
                    a.x += (float)(2 * (b.scell[j] - row) + sx) * I.ohf;
                    a.y += sy;
                    a.z += sz;
                    // a NaN or an infinity fails the comparison too
                    wild = wild || !(fabsf(v.x) + fabsf(v.y) + fabsf(v.z) + fabsf(v.w) + fabsf(a.w) < lim && a.w > dmin);
                    const int32_t t = p0 + l;
                    if (!SPH_BOUNDS_OK(t >= 0 && t < kStage, &b.misc[2]))
                        continue;
                    stA[t] = a;
                    stB[t] = v;
                    stF[t] = f;
                }
            }
            if (wild)
                S.wild = 1;
        }
        __syncthreads();
        const bool staged = fits && !S.wild;
        for (;;) {
            int q = 0;
            if (lane == 0)
                q = atomicAdd(&S.next, 1);
            q = __shfl_sync(0xffffffffu, q, 0);
            if (q >= nclus)
                break;
            if (staged)
                pair_cluster<NW, G, COMP, STAT, DFS, true>(b, I, kc, T, kdiv, q, st, list, lane, S, lc, wc_cand);
            else
                pair_cluster_global<NW, G, COMP, STAT, DFS>(b, I, T, kdiv, q, list, lane, S, lc, wc_cand);
        }
    }
    if (!STAT)
        return;
    // work counts: lanes -> warp -> CTA -> device
    const unsigned wff = (unsigned)warp_sum((int)lc[0]), wvi = (unsigned)warp_sum((int)lc[1]);
    if (lane == 0) {
        atomicAdd(&S.st_ff, (unsigned long long)wff);
        atomicAdd(&S.st_visc, (unsigned long long)wvi);
        atomicAdd(&S.st_cand, wc_cand);
    }
    __syncthreads();
    if (tid == 0) {
        atomicAdd(&b.pstat[0], S.st_ff);
        atomicAdd(&b.pstat[1], S.st_visc);
        atomicAdd(&b.pstat[2], S.st_cand);
    }
}

}  // namespace sph
