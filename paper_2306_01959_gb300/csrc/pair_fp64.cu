// FP64 form of the pair pass (Eqs. 3-8) and the obstacle-force probe.
//
// One warp per particle i (sorted order).  The lanes sweep i's candidate
// rows: for every (dy, dz) cell offset the cells cx-k .. cx+k of that row are
// consecutive in the sorted order, so each row is one contiguous range.  A
// candidate j is a neighbour when |r_j - r_i|^2 < (2h)^2, evaluated as
// ((dx dx + dy dy) + dz dz) with every operation rounded separately, so the
// neighbour set is the same set the definition gives; an FP32 pre-test on
// FP32 copies of the positions, with radii moved out and in by their worst
// rounding error, settles every candidate certainly out of reach or certainly
// inside, so that only a thin shell around 2h takes the exact test.  Neighbours that
// interact are compacted through a per-warp queue by ballot, so that the
// expensive pair arithmetic runs on full 32-lane batches (all but the last
// batch of each particle); the lane partial sums are combined by warp shuffles.
#include "device.cuh"
#include "fixed.h"

namespace sph {

constexpr int kQ = 64;  // per-warp queue of neighbour indices

struct AccD {
    double drho, ax, ay, az;
    double dd;  // the delta term of Eq. 7, kept apart when it may be dropped (SPH_DELTA_FULL_SUPPORT)
    // running max of mu / h as the bit pattern of a double read as a signed
    // integer: non-negative doubles order like their bit patterns and negative
    // ones fall below the starting 0 (+0.0), so the integer max is the max of
    // mu started at 0, taken on the integer units instead of the FP64 pipe
    long long mumax_bits;
};

// Constants of an instance used by every pair.
struct PairConstD {
    double half_inv_h, eta2, dfac, nah;  // dfac = 2 delta h c0, nah = -alpha h
    uint64_t kh;                         // fixed-point positions only, and eta^2 in their units
    Fixed2 eta;
};

template <bool FIX>
__device__ __forceinline__ PairConstD pair_const_d(const Inst &I)
{
    return FIX ? PairConstD{I.fx_hinv, 0.0, I.fx_dfac, I.fx_nah, I.fx_kh, Fixed2{I.fx_eta, I.fx_eta_f}}
               : PairConstD{I.half_inv_h, I.eta2, I.dfac_d, I.nah, 0ull, Fixed2{0ull, 0u}};
}

// Particle i of a pair, with the products that all its pairs share, and the constants.
struct __align__(16) OwnD {
    double x, y, z, rho;
    double ux, uy, uz, inv_rho;
    double drho, prho, nac;  // -dfac rho, P / rho, nah c
    PairConstD k;
};
__device__ __forceinline__ OwnD own_d(const PairConstD &k, double x, double y, double z, double ux, double uy,
                                      double uz, double rho, double inv_rho, double P, double c)
{
    return OwnD{x, y, z, rho, ux, uy, uz, inv_rho, -k.dfac * rho, P * inv_rho, k.nah * c, k};
}

// The FP64 pipe of this GPU issues one warp operation every 64 cycles per
// scheduler, so the pair term is priced in FP64 operations alone; the library's
// reciprocal square root took about 10 of them.  This one starts from the
// hardware's 20-bit approximation and takes one step of third order (Householder's
// method, from the series of (1 - e)^-1/2 in the residual e of the approximation):
// the remaining error, e^3 < 2^-57, is below the rounding of the last operation.

// sqrt(a) for a >= 0 (5 operations); 0 for 0: the approximation is taken at
// no less than 2^-1000 (an integer maximum of the bit patterns).
__device__ __forceinline__ double sqrt3(double a)
{
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(__longlong_as_double(max(__double_as_longlong(a), 23LL << 52))));
    const double s = a * y;
    const double e = fma(-s, y, 1.0);
    return fma(s * e, fma(0.375, e, 0.5), s);
}

// ---------------------------------------------------------------------------
// Fixed-point distances (fixed.h).  The FP64 pipe is the bound and the integer pipes
// idle beside it, so the steps from the positions to t^3 = (1 - q/2)^3, |r_ij|^2 +
// eta^2 and the reciprocal, 20 of the 39 FP64 operations of a pair, run in 64-bit
// integers instead.  Differences are exact, |r_ij|^2 + eta^2 to 2^-81 and t to 2^-58,
// and each result is rounded once, so that nothing is less accurate than in doubles.
// Largest errors over pairs from 2h / 128 to 2h, 2h from 0.064 to 0.116, against
// 113-bit arithmetic (FP64 operations in brackets): r_ij 1.1e-16 of |r_ij| (1.1e-16),
// |r_ij|^2 + eta^2 3e-18 (5e-16), t^3 5.7e-17 (3.0e-16), the reciprocal of
// (|r_ij|^2 + eta^2)(rho_i + rho_j) 1.1e-16 (6.3e-16), next to the coordinate planes
// and away from them.  Closer pairs, whose |r_ij|^2 has too few bits for its root,
// take that in FP64 (R < 2^48: below 2h / 128 to 2h / 64).
// Scaling by powers of two is exact, so the sums carry the units along: with r_ij in
// units of 2^-s and |r_ij|^2 + eta^2 in 2^(64 - 2s), the constants of PairConstD absorb
// the factors and pair_sF, pair_hmu undo them.
// ---------------------------------------------------------------------------
// Geometry of a pair: r_ij, |r_ij|^2 + eta^2 and t^3, in the units of k.  The
// positions are doubles, or (FIX) 64-bit integers in the same registers, and so is
// |r_ij|^2 + eta^2 (V in place of re).
struct PairGeoD {
    double rx, ry, rz, re, t3;
    Fixed2 V;
};
template <bool FIX>
__device__ __forceinline__ PairGeoD pair_geo_d(const OwnD &o, double xj, double yj, double zj)
{
    PairGeoD p;
    if (FIX) {
        const int64_t dx = __double_as_longlong(xj) - __double_as_longlong(o.x);
        const int64_t dy = __double_as_longlong(yj) - __double_as_longlong(o.y);
        const int64_t dz = __double_as_longlong(zj) - __double_as_longlong(o.z);
        const Fixed2 d2 = fixed_dist2(dx, dy, dz);
        p.rx = int_to_double(dx);
        p.ry = int_to_double(dy);
        p.rz = int_to_double(dz);
        p.V.f = d2.f + o.k.eta.f;
        p.V.R = d2.R + o.k.eta.R + (p.V.f < d2.f);
        if (d2.R >= (1ull << 48)) {
            p.t3 = fixed_t3(d2, o.k.kh);
        } else {
            const double t = 1.0 - sqrt3(p.rx * p.rx + p.ry * p.ry + p.rz * p.rz) * o.k.half_inv_h;
            p.t3 = t * t * t;
        }
    } else {
        p.rx = xj - o.x;
        p.ry = yj - o.y;
        p.rz = zj - o.z;
        const double r2 = p.rx * p.rx + p.ry * p.ry + p.rz * p.rz;
        const double t = 1.0 - sqrt3(r2) * o.k.half_inv_h;
        p.re = r2 + o.k.eta2;
        p.t3 = t * t * t;  // m_j F / (-kF m)
    }
    return p;
}

// Eqs. 4-5: Pi_ij = -alpha c_bar mu / rho_bar (0 unless u_ij . r_ij < 0; a -0.0 gives
// a zero term), c_bar / rho_bar = (c_i + c_j) / (rho_i + rho_j), and muh = mu / h =
// (u_ij . r_ij) / (|r_ij|^2 + eta^2), 0 for an approaching pair: the running maximum
// starts there.  cs: -alpha h (c_i + c_j), rsum: rho_i + rho_j.
template <bool FIX>
__device__ __forceinline__ void pair_visc(const PairGeoD &p, double udotr, double cs, double rsum, double &visc,
                                          double &muh)
{
    const bool app = __double2hiint(udotr) < 0;
    if (FIX && (unsigned)((__double2hiint(rsum) >> 20) - 128) < 1664u) {
        // one reciprocal, of (|r_ij|^2 + eta^2)(rho_i + rho_j), and one product for both
        const double prod = udotr * fixed_rcp(p.V, rsum) * (app ? cs : rsum);
        visc = app ? prod : 0.0;
        muh = app ? 0.0 : prod;
    } else {
        // density sums that are not positive, or no number: muh does not depend on them
        const double m = udotr * __drcp_rn(FIX ? int_to_double((int64_t)p.V.R) + p.V.f * 0x1p-32 : p.re);
        visc = app ? cs * m * __drcp_rn(rsum) : 0.0;
        muh = app ? 0.0 : m;
    }
}

// Contribution of neighbour j to particle i (Eqs. 3-7), in double.
// Continuity uses the standard sign (u_i - u_j) . grad_i W_ij; the delta
// term acts between fluid particles; the viscosity of Eq. 4 applies when
// u_ij . r_ij < 0.  1/rho and c of both particles come precomputed, so a pair
// costs one square root and one reciprocal, that of (|r_ij|^2 + eta^2)(rho_i +
// rho_j): 38 FP64 operations, 19 on fixed-point positions.  m_j F = -kF m t^3 with
// t = 1 - q/2: the sums of D rho/Dt and of the acceleration are accumulated
// with t^3 in place of m_j F and the caller scales them by -kF m, and the
// running maximum is of mu / h, which the caller scales by h.  With DFS the
// delta term is summed apart (the caller drops it for a fluid particle that
// has a boundary neighbour).
template <bool DFS, bool FIX>
__device__ __forceinline__ void pair_term_d(const OwnD &o, bool fluid_i, double xj, double yj, double zj, double uxj,
                                            double uyj, double uzj, double rhoj, double inv_rhoj, double Pj,
                                            double cj, bool fluid_j, AccD &a)
{
    const PairGeoD p = pair_geo_d<FIX>(o, xj, yj, zj);
    const double rx = p.rx, ry = p.ry, rz = p.rz, t3 = p.t3;  // r_ij = r_j - r_i; grad_i W_ij = F (r_i - r_j) = -F r_ij
    double ux = uxj - o.ux, uy = uyj - o.uy, uz = uzj - o.uz;  // u_ij = u_j - u_i
    double udotr = ux * rx + uy * ry + uz * rz;  // u_ij . r_ij
    // Eq. 7: sum_j m_j (u_i - u_j) . grad_i W_ij = m_j F (u_ij . r_ij), plus the delta term
    // 2 delta h c0 (rho_j - rho_i) (r_ij . grad_i W_ij) / |r_ij|^2 m_j / rho_j, where
    // (r_ij . grad_i W_ij) / |r_ij|^2 = -F and (rho_j - rho_i) / rho_j = 1 - rho_i / rho_j
    double g = (fluid_i && fluid_j) ? fma(o.drho, inv_rhoj, o.k.dfac) : 0.0;
    if (DFS) {
        a.drho = fma(t3, udotr, a.drho);
        a.dd = fma(t3, g, a.dd);
    } else {
        a.drho = fma(t3, udotr - g, a.drho);
    }
    double visc, muh;
    pair_visc<FIX>(p, udotr, fma(o.k.nah, cj, o.nac), o.rho + rhoj, visc, muh);
    // Eq. 3: a_i -= m_j (...) grad_i W_ij = m_j (...) F r_ij, with
    // (P_i + P_j) / (rho_i rho_j) = (P_i / rho_i + P_j / rho_i) / rho_j
    double coef = fma(fma(Pj, o.inv_rho, o.prho), inv_rhoj, visc) * t3;
    a.ax += coef * rx;
    a.ay += coef * ry;
    a.az += coef * rz;
    a.mumax_bits = max(a.mumax_bits, __double_as_longlong(muh));
}

// Partner's share of a pair evaluated once (params.pair_symmetric): the terms
// of Eqs. 3, 7 and 15 for j from the same pair, added to j's accumulators in
// global memory by FP64 atomics (performed in L2).  Eq. 3 is antisymmetric
// ((P_i + P_j)/(rho_i rho_j) and Pi_ij are symmetric, r_ji = -r_ij), Eq. 7
// has the same continuity term and j's own delta term
// 2 delta h c0 (1 - rho_j / rho_i), mu is the same; units as pair_term_d
// (t^3 in place of m F, mu / h).  i's own share is accumulated in a.
__device__ __forceinline__ void pair_share_j(const OwnD &o, bool fluid_i, double xj, double yj, double zj, double uxj,
                                             double uyj, double uzj, double rhoj, double inv_rhoj, double Pj,
                                             double cj, bool fluid_j, dvec4 *jacc, long long *jmu, int32_t j,
                                             AccD &a)
{
    const PairGeoD p = pair_geo_d<true>(o, xj, yj, zj);
    const double rx = p.rx, ry = p.ry, rz = p.rz, t3 = p.t3;
    double ux = uxj - o.ux, uy = uyj - o.uy, uz = uzj - o.uz;
    double udotr = ux * rx + uy * ry + uz * rz;
    const bool ff = fluid_i && fluid_j;
    double g = ff ? fma(o.drho, inv_rhoj, o.k.dfac) : 0.0;
    double gj = ff ? fma(-o.k.dfac * rhoj, o.inv_rho, o.k.dfac) : 0.0;
    a.drho = fma(t3, udotr - g, a.drho);
    double visc, muh;
    pair_visc<true>(p, udotr, fma(o.k.nah, cj, o.nac), o.rho + rhoj, visc, muh);
    double coef = fma(fma(Pj, o.inv_rho, o.prho), inv_rhoj, visc) * t3;
    a.ax += coef * rx;
    a.ay += coef * ry;
    a.az += coef * rz;
    a.mumax_bits = max(a.mumax_bits, __double_as_longlong(muh));
    double *J = reinterpret_cast<double *>(jacc + j);
    atomicAdd(J + 0, -coef * rx);
    atomicAdd(J + 1, -coef * ry);
    atomicAdd(J + 2, -coef * rz);
    atomicAdd(J + 3, t3 * (udotr - gj));
    if (muh > 0.0)
        atomicMax(jmu + j, __double_as_longlong(muh));  // positive doubles order like their bits
}

__device__ __forceinline__ double dist2_rn(double xi, double yi, double zi, double xj, double yj, double zj)
{
    double dx = __dsub_rn(xj, xi), dy = __dsub_rn(yj, yi), dz = __dsub_rn(zj, zi);
    return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

// What the lanes of a warp share while they work on particle i.
constexpr int kRowsD = 49;  // rows of cells around one, cell_div <= 3
struct WarpD {
    OwnD own;
    double sup2, sF, hmu, g;
    float4 d;  // FP32 copy of the position, and the radius certainly inside, squared
    float filter;
    int2 rows[kRowsD];
};

// SYM: each interacting pair once (the forward half of i's neighbourhood:
// rows with dz > 0, rows with dz = 0 and dy > 0, and the home row after i),
// the partner's share by pair_share_j; k_pair_fp64_finish adds the shares.
// CNT (with SYM): also count the partners' neighbours (nneigh is read by
// sph_derivatives and the work counts, not by a time step).
// Bound by the FP64 pipe (82 % busy on 0.9 M particles, of the 84 % that FMAs alone
// reach) as long as enough warps cover the gathers and the serial integer chains of
// a batch: what the lanes of a warp share, the row ranges too, lies in shared memory,
// so that 32 warps of 64 registers fit on an SM.  0.9 M particles (11 k): 12.5 ms
// (200 us) with all of it in 124 registers and 16 warps, 10.7 (163) without the rows
// and 24 warps, 9.8 (145) with the rows and 24 warps, 8.9 (146) with 32, 9.9 (154)
// with 40, which spill.
template <bool DFS, bool SYM, bool CNT = true>
__global__ void __launch_bounds__(256, 4) k_pair_fp64(Bufs b, int ninst, int kdiv)
{
    extern __shared__ int32_t smem_q[];
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    __shared__ WarpD warps[8];
    WarpD &W = warps[wib];
    int32_t *q = smem_q + wib * kQ;  // neighbours; the sign bit marks a fluid particle
    const unsigned lt = (1u << lane) - 1u;
    const int32_t n_in = b.misc[0];
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    const dvec4 *sA = reinterpret_cast<const dvec4 *>(b.sA);
    const dvec4 *sB = reinterpret_cast<const dvec4 *>(b.sB);

    for (int32_t i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n_in; i += nwarps) {
        int nrows = 0;
        {
            const int32_t ci_cell = b.scell[i];
            const Inst &I = b.inst[inst_of_cell(b.inst, ninst, ci_cell)];
            int cx, cy, cz;
            decompose(I, ci_cell, cx, cy, cz);
            if (lane == 0) {
                const dvec4 A = sA[i], B = sB[i];
                const double2 C = b.sC[i];
                const float4 D = b.sD[i];
                W.own = own_d(pair_const_d<true>(I), A.x, A.y, A.z, B.x, B.y, B.z, A.w, C.x, B.w, C.y);
                W.d = make_float4(D.x, D.y, D.z, I.sup2_inner);
                W.filter = I.sup2_filter;
                W.sup2 = I.sup2;
                W.sF = I.pair_sF;
                W.hmu = I.pair_hmu;
                W.g = I.g;
            }
            // a lane per row of cells reads its range, so that the loads of all rows are in
            // flight together
            const int side = 2 * kdiv + 1;
            int ncand = 0;
            for (int r0 = 0; r0 < side * side; r0 += 32) {
                int32_t s0 = 0, s1 = 0;
                const int r = r0 + lane, dz = r / side - kdiv, dy = r % side - kdiv, z = cz + dz, y = cy + dy;
                if (dz <= kdiv && z >= 0 && z < I.n[2] && y >= 0 && y < I.n[1] &&
                    (!SYM || dz > 0 || (dz == 0 && dy >= 0))) {
                    const int32_t row = I.cell_base + (z * I.n[1] + y) * I.n[0];
                    s0 = b.cell_start[row + max(cx - kdiv, 0)];
                    s1 = b.cell_start[row + min(cx + kdiv, I.n[0] - 1) + 1];
                    if (SYM && dz == 0 && dy == 0)
                        s0 = i + 1;  // the home row from the home cell on (cells hold ascending ids), after i
                }
                const unsigned m = __ballot_sync(0xffffffffu, s0 < s1);
                if (s0 < s1) {
                    W.rows[nrows + __popc(m & lt)] = make_int2(s0, s1);
                    ncand += s1 - s0;
                }
                nrows += __popc(m);
            }
            ncand = warp_sum(ncand);
            if (lane == 0)
                b.ncand[i] = ncand;
        }
        __syncwarp();
        const bool fluid_i = b.sflag[i] == T_FLUID;
        AccD acc = {0.0, 0.0, 0.0, 0.0, 0.0, 0};
        bool touches_boundary = false;  // DFS: some neighbour j is a boundary particle
        int nn = 0;
        int qn = 0;
        int npair = 0;

        auto flush = [&](int cnt) {
            if (lane < cnt) {
                const int32_t qj = q[lane], j = qj & 0x7fffffff;
                const bool fluid_j = qj < 0;
                const dvec4 Aj = sA[j], Bj = sB[j];
                const double2 Cj = b.sC[j];
                if (SYM)
                    pair_share_j(W.own, fluid_i, Aj.x, Aj.y, Aj.z, Bj.x, Bj.y, Bj.z, Aj.w, Cj.x, Bj.w, Cj.y, fluid_j,
                                      b.fjacc, b.fjmu, j, acc);
                else
                    pair_term_d<DFS, true>(W.own, fluid_i, Aj.x, Aj.y, Aj.z, Bj.x, Bj.y, Bj.z, Aj.w, Cj.x, Bj.w, Cj.y,
                                          fluid_j, acc);
            }
        };

        for (int k = 0; k < nrows; ++k) {
            const int2 row = W.rows[k];
            for (int32_t base = row.x; base < row.y; base += 32) {
                int32_t j = base + lane;
                bool take = false, fluid_j = false;
                if (j < row.y && j != i) {
                    // FP32 pre-test with radii that cover every rounding of the
                    // FP32 copies: certainly inside, certainly outside, or (in a
                    // thin shell around 2h) decided by the exact FP64 test
                    const float4 Dj = b.sD[j], Di = W.d;
                    const float fx = Dj.x - Di.x, fy = Dj.y - Di.y, fz = Dj.z - Di.z;
                    const float d2f = fx * fx + fy * fy + fz * fz;
                    bool hit = d2f < Di.w;
                    if (!hit && d2f < W.filter) {
                        const dvec4 ri = b.pos[b.perm[i]], rj = b.pos[b.perm[j]];
                        hit = dist2_rn(ri.x, ri.y, ri.z, rj.x, rj.y, rj.z) < W.sup2;
                    }
                    if (hit) {
                        ++nn;
                        if (SYM && CNT)
                            atomicAdd(b.fjnn + j, 1);
                        fluid_j = Dj.w != 0.f;
                        take = fluid_i || fluid_j;
                        if (DFS)
                            touches_boundary = touches_boundary || !fluid_j;
                    }
                }
                unsigned m = __ballot_sync(0xffffffffu, take);
                if (take)
                    q[qn + __popc(m & lt)] = fluid_j ? j | (int32_t)0x80000000 : j;
                qn += __popc(m);
                npair += __popc(m);
                __syncwarp();
                if (qn >= 32) {
                    flush(32);
                    __syncwarp();
                    if (lane < qn - 32)
                        q[lane] = q[lane + 32];
                    qn -= 32;
                    __syncwarp();
                }
            }
        }
        flush(qn);
        __syncwarp();
        const double sF = W.sF;  // t^3 -> m_j F
        constexpr int K = DFS ? 8 : 4;
        double tot[K] = {acc.drho, acc.ax, acc.ay, acc.az};
        if (DFS)
            tot[4] = acc.dd;
        // lane 0 holds the totals; every operation here is paid for by the whole warp,
        // so each lane scales its one total before the exchange
        warp_totals<K>(tot, sF);
        double drho = tot[0];
        if (DFS && !__any_sync(0xffffffffu, touches_boundary))
            drho -= tot[K > 4 ? 4 : 0];
        double ax = tot[1], ay = tot[2], az = tot[3];
        double mumax = W.hmu * __longlong_as_double(warp_max_bits(acc.mumax_bits));
        int nsum = warp_sum(nn);
        if (lane == 0) {
            if (fluid_i)
                az -= W.g;
            reinterpret_cast<dvec4 *>(b.deriv)[i] = make_dvec4(ax, ay, az, drho);
            reinterpret_cast<double *>(b.mumax)[i] = mumax;
            b.nneigh[i] = nsum;
            b.npair[i] = npair;
        }
        __syncwarp();
    }
}

// Adds the partners' shares of the symmetric pass, scaled as the owner's.
template <bool CNT>
__global__ void k_pair_fp64_finish(Bufs b, int ninst)
{
    const int32_t n_in = b.misc[0];
    for (int32_t s = blockIdx.x * blockDim.x + threadIdx.x; s < n_in; s += gridDim.x * blockDim.x) {
        const Inst &I = b.inst[inst_of_cell(b.inst, ninst, b.scell[s])];
        const double sF = I.pair_sF;
        const dvec4 j = b.fjacc[s];
        dvec4 *D = reinterpret_cast<dvec4 *>(b.deriv) + s;
        const dvec4 d = *D;
        *D = make_dvec4(d.x + sF * j.x, d.y + sF * j.y, d.z + sF * j.z, d.w + sF * j.w);
        double *M = reinterpret_cast<double *>(b.mumax) + s;
        *M = fmax(*M, I.pair_hmu * __longlong_as_double(b.fjmu[s]));
        if (CNT)
            b.nneigh[s] += b.fjnn[s];
    }
}

void launch_pair_fp64(const Bufs &b, int64_t N, int32_t ninst, int32_t cell_div, int32_t warps, int32_t ctas,
                      int32_t delta_mode, bool neighbours, cudaStream_t st)
{
    if (warps <= 0 || warps > 8)
        warps = 8;  // the kernel is compiled for at most 256 threads per CTA
    if (ctas <= 0)
        ctas = 8;
    const int grid = sm_count() * ctas;
    const size_t dyn = warps * kQ * sizeof(int32_t);
    if (b.fjacc) {
        // the partners' accumulators start at zero (mu / h >= 0 as bits)
        cudaMemsetAsync(b.fjacc, 0, sizeof(dvec4) * (size_t)N, st);
        cudaMemsetAsync(b.fjmu, 0, sizeof(long long) * (size_t)N, st);
        const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((N + 255) / 256, (int64_t)sm_count() * 8));
        if (neighbours) {
            cudaMemsetAsync(b.fjnn, 0, sizeof(int32_t) * (size_t)N, st);
            k_pair_fp64<false, true, true><<<grid, warps * 32, dyn, st>>>(b, ninst, cell_div);
            k_pair_fp64_finish<true><<<blocks, 256, 0, st>>>(b, ninst);
        } else {
            k_pair_fp64<false, true, false><<<grid, warps * 32, dyn, st>>>(b, ninst, cell_div);
            k_pair_fp64_finish<false><<<blocks, 256, 0, st>>>(b, ninst);
        }
        return;
    }
    if (delta_mode == SPH_DELTA_FULL_SUPPORT)
        k_pair_fp64<true, false><<<grid, warps * 32, dyn, st>>>(b, ninst, cell_div);
    else
        k_pair_fp64<false, false><<<grid, warps * 32, dyn, st>>>(b, ninst, cell_div);
}

// ---------------------------------------------------------------------------
// Force on the obstacle (Section 3.2): sum over its particles of m a_b, a_b
// from fluid neighbours by Eq. 3 without gravity, in double on the current
// state (read through the canonical arrays, so both precision forms agree).
// ---------------------------------------------------------------------------
template <int MODE>
__device__ __forceinline__ void load_state(const Bufs &b, const Inst &I, int32_t id, double &x, double &y,
                                           double &z, double &ux, double &uy, double &uz, double &rho)
{
    dvec4 p = b.pos[id];
    x = p.x;
    y = p.y;
    z = p.z;
    if (MODE == SPH_FP64) {
        dvec4 v = reinterpret_cast<const dvec4 *>(b.vel)[id];
        ux = v.x;
        uy = v.y;
        uz = v.z;
        rho = v.w;
    } else {
        float4 v = reinterpret_cast<const float4 *>(b.vel)[id];
        ux = v.x;
        uy = v.y;
        uz = v.z;
        rho = I.rho0 + (double)v.w;
    }
}

template <int MODE>
__global__ void k_probe_force(Bufs b, int inst, int kdiv)
{
    __shared__ double part[8][3];
    const Inst &I = b.inst[inst];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    const int32_t s_begin = b.cell_start[I.cell_base], s_end = b.cell_start[I.cell_base + I.ncells];
    double fx = 0, fy = 0, fz = 0;
    for (int32_t s = s_begin + ((blockIdx.x * blockDim.x + threadIdx.x) >> 5); s < s_end; s += nwarps) {
        if (b.sflag[s] != T_OBST)
            continue;
        int32_t idb = b.perm[s];
        double xb, yb, zb, uxb, uyb, uzb, rhob;
        load_state<MODE>(b, I, idb, xb, yb, zb, uxb, uyb, uzb, rhob);
        double Pb = tait_d(I, rhob), cb = sound_d(I, rhob);
        const OwnD own =
            own_d(pair_const_d<false>(I), xb, yb, zb, uxb, uyb, uzb, rhob, 1.0 / rhob, Pb, cb);
        int cx, cy, cz;
        decompose(I, b.scell[s], cx, cy, cz);
        AccD acc = {0, 0, 0, 0, 0};
        for (int dz = -kdiv; dz <= kdiv; ++dz) {
            int z = cz + dz;
            if (z < 0 || z >= I.n[2])
                continue;
            for (int dy = -kdiv; dy <= kdiv; ++dy) {
                int y = cy + dy;
                if (y < 0 || y >= I.n[1])
                    continue;
                int x0 = max(cx - kdiv, 0), x1 = min(cx + kdiv, I.n[0] - 1);
                int32_t row = I.cell_base + (z * I.n[1] + y) * I.n[0];
                int32_t s0 = b.cell_start[row + x0], s1 = b.cell_start[row + x1 + 1];
                for (int32_t j = s0 + lane; j < s1; j += 32) {
                    if (b.sflag[j] != T_FLUID)
                        continue;
                    int32_t idj = b.perm[j];
                    double xj, yj, zj, uxj, uyj, uzj, rhoj;
                    load_state<MODE>(b, I, idj, xj, yj, zj, uxj, uyj, uzj, rhoj);
                    if (dist2_rn(xb, yb, zb, xj, yj, zj) < I.sup2)
                        pair_term_d<false, false>(own, false, xj, yj, zj, uxj, uyj, uzj, rhoj, 1.0 / rhoj,
                                                  tait_d(I, rhoj), sound_d(I, rhoj), true, acc);
                }
            }
        }
        const double sF = -I.kFm * I.mass;  // t^3 -> m_j F, times the obstacle particle's mass
        fx += sF * acc.ax;
        fy += sF * acc.ay;
        fz += sF * acc.az;
    }
    fx = warp_sum(fx);
    fy = warp_sum(fy);
    fz = warp_sum(fz);
    if (lane == 0) {
        part[wib][0] = fx;
        part[wib][1] = fy;
        part[wib][2] = fz;
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        double s = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w)
            s += part[w][threadIdx.x];
        b.diag[blockIdx.x * 3 + threadIdx.x] = s;
    }
}

__global__ void k_sum_blocks3(const double *part, int nb, double *out)
{
    if (threadIdx.x < 3) {
        double s = 0;
        for (int k = 0; k < nb; ++k)
            s += part[k * 3 + threadIdx.x];
        out[threadIdx.x] = s;
    }
}

void launch_probe_force(const Bufs &b, int mode, int32_t inst, int32_t ninst, int32_t cell_div, int64_t N,
                        cudaStream_t st)
{
    (void)ninst;
    (void)N;
    const int nb = kDiagBlocks;
    if (mode == SPH_FP64)
        k_probe_force<SPH_FP64><<<nb, 256, 0, st>>>(b, inst, cell_div);
    else
        k_probe_force<SPH_MIXED><<<nb, 256, 0, st>>>(b, inst, cell_div);
    k_sum_blocks3<<<1, 32, 0, st>>>(b.diag, nb, b.probe_out);
}

}  // namespace sph
