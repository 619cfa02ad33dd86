// Host-side scene generation and instance constants.
//
// The paper gives tank, column and obstacle sizes (Sections 3.1, 3.2) but not
// the particle layout.  The layout taken: fluid on the lattice
// ((i+1/2) dp, (j+1/2) dp, (k+1/2) dp) measured from the inner tank corner,
// the column against the x = 0 end wall; `boundary_layers` layers of fixed
// boundary particles outside the floor and the four walls, up to the tank
// height, no lid; the obstacle a filled lattice box whose lower corner is
// rounded to the lattice; an optional moving gate built the same way.
// Particle ids: fluid (x fastest, then y, then z), walls+floor (same loop
// order over the enclosing box), obstacle, gate.  Every
// particle has mass rho0 dp^3.  The cell grid spans
// [-L dp, Lt + L dp] x [-L dp, Wt + L dp] x [-L dp, Ht + 4h] with cells of
// size 2h / cell_div.
#include <cmath>
#include <cstring>

#include "internal.h"

namespace sph {

static int64_t nint(double x) { return (int64_t)std::floor(x + 0.5); }

int effective_cell_div(const sph_params &p)
{
    // automatic: cells of size 2h for the mixed form (what callers see; its tiled
    // pair pass divides them again), cells of size h for the FP64 form
    if (p.cell_div > 0)
        return p.cell_div;
    return p.precision == SPH_MIXED ? 1 : 2;
}

int validate_instance(const sph_instance &in, const sph_params &p, std::string &err)
{
    auto bad = [&](const char *m) {
        err = m;
        return SPH_EINVAL;
    };
    if (!(in.dp > 0) || !(in.h > 0) || !(in.c0 > 0) || !(in.rho0 > 0) || !(in.alpha >= 0))
        return bad("dp, h, c0, rho0 must be > 0 and alpha >= 0");
    if (!(in.h >= 0.5 * in.dp) || in.h > 8.0 * in.dp)
        return bad("h must lie in [dp/2, 8 dp]");
    for (int a = 0; a < 3; ++a) {
        if (!(in.tank[a] > 0) || !(in.column[a] >= 0))
            return bad("tank sizes must be > 0 and column sizes >= 0");
        if (nint(in.column[a] / in.dp) > nint(in.tank[a] / in.dp))
            return bad("water column does not fit in the tank");
    }
    if (in.has_obstacle) {
        int64_t o0[3], o1[3];
        for (int a = 0; a < 3; ++a) {
            if (!(in.obstacle[3 + a] > 0) || !(in.obstacle[a] >= 0))
                return bad("obstacle corner must be >= 0 and sizes > 0");
            o0[a] = nint(in.obstacle[a] / in.dp);
            o1[a] = o0[a] + nint(in.obstacle[3 + a] / in.dp);
            if (o1[a] > nint(in.tank[a] / in.dp) || o1[a] <= o0[a])
                return bad("obstacle does not fit in the tank");
        }
        bool overlap = true;
        for (int a = 0; a < 3; ++a)
            overlap = overlap && o0[a] < nint(in.column[a] / in.dp) && 0 < o1[a];
        if (overlap && nint(in.column[0] / in.dp) > 0 && nint(in.column[1] / in.dp) > 0 &&
            nint(in.column[2] / in.dp) > 0)
            return bad("obstacle overlaps the water column");
    }
    if (in.has_gate) {
        int64_t g0[3], g1[3];
        for (int a = 0; a < 3; ++a) {
            if (!(in.gate[3 + a] > 0) || !(in.gate[a] >= 0) || !std::isfinite(in.gate_velocity[a]))
                return bad("gate corner must be >= 0, sizes > 0 and the velocity finite");
            g0[a] = nint(in.gate[a] / in.dp);
            g1[a] = g0[a] + nint(in.gate[3 + a] / in.dp);
            if (g1[a] > nint(in.tank[a] / in.dp) || g1[a] <= g0[a])
                return bad("gate does not fit in the tank");
        }
        bool overlap = true;
        for (int a = 0; a < 3; ++a)
            overlap = overlap && g0[a] < nint(in.column[a] / in.dp) && 0 < g1[a];
        if (overlap && nint(in.column[0] / in.dp) > 0 && nint(in.column[1] / in.dp) > 0 &&
            nint(in.column[2] / in.dp) > 0)
            return bad("gate overlaps the water column");
    }
    if (p.boundary_layers < 1 || p.boundary_layers > 8)
        return bad("boundary_layers must be in [1, 8]");
    if (p.cell_div < 0 || p.cell_div > 3)
        return bad("cell_div must be 0 (automatic), 1, 2 or 3");
    if (p.ns < 1)
        return bad("ns must be >= 1");
    if (!(p.cfl > 0) || p.cfl > 1)
        return bad("cfl must be in (0, 1]");
    if (!(p.gamma >= 1) || !(p.delta >= 0) || !(p.g >= 0) || !(p.dt_min >= 0))
        return bad("gamma >= 1, delta >= 0, g >= 0 and dt_min >= 0 required");
    if (p.precision != SPH_FP64 && p.precision != SPH_MIXED)
        return bad("precision must be SPH_FP64 or SPH_MIXED");
    if (p.integrator != SPH_VERLET && p.integrator != SPH_SYMPLECTIC)
        return bad("integrator must be SPH_VERLET or SPH_SYMPLECTIC");
    if (p.delta_mode != SPH_DELTA_ALL_FLUID && p.delta_mode != SPH_DELTA_FULL_SUPPORT)
        return bad("delta_mode must be SPH_DELTA_ALL_FLUID or SPH_DELTA_FULL_SUPPORT");
    if (p.pair_symmetric && (p.precision != SPH_FP64 || p.delta_mode != SPH_DELTA_ALL_FLUID))
        return bad("pair_symmetric runs the FP64 form with SPH_DELTA_ALL_FLUID");
    if (!(p.list_skin >= 0) || !(p.list_skin <= 4) || p.list_capacity < 0 || p.list_capacity > 65536)
        return bad("list_skin must be in [0, 4] and list_capacity in [0, 65536]");
    if (p.list_skin > 0 && (p.precision != SPH_MIXED || p.integrator != SPH_VERLET || p.persistent ||
                            effective_cell_div(p) != 1))
        return bad("neighbour lists (list_skin > 0) run the mixed form with the Verlet scheme, per-phase "
                   "launches and cell_div 1");
    return SPH_OK;
}

// Constants of the FP64 pair pass in the units of its fixed-point positions (fixed.h).
static void fill_fixed_point(Inst &d)
{
    if (!std::isfinite(d.h))
        return;  // (refused later: such an instance has no particles)
    const int s = 62 - std::ilogb(2.0 * d.h);
    d.fx_shift = s;
    const uint64_t h2 = (uint64_t)std::ldexp(2.0 * d.h, s);  // an integer in [2^62, 2^63)
    const unsigned __int128 k = ((unsigned __int128)1 << 126) / h2;
    d.fx_kh = k >> 64 ? ~0ull : (uint64_t)k;
    const double eta = std::ldexp(d.eta2, 2 * s - 64);
    d.fx_eta = (uint64_t)eta;
    d.fx_eta_f = (uint32_t)std::ldexp(eta - (double)d.fx_eta, 32);
    d.fx_hinv = std::ldexp(d.half_inv_h, -s);
    d.fx_dfac = std::ldexp(d.dfac_d, s);
    d.fx_nah = std::ldexp(d.nah, s - 64);
    d.pair_sF = std::ldexp(-d.kFm, -s);
    d.pair_hmu = std::ldexp(d.h, s - 64);
}

void fill_inst(HostInst &hi, const sph_params &p, int fine, bool tiled)
{
    const sph_instance &in = hi.d;
    double dp = in.dp;
    int64_t L = p.boundary_layers;
    int64_t ncx = nint(in.column[0] / dp), ncy = nint(in.column[1] / dp), ncz = nint(in.column[2] / dp);
    int64_t ntx = nint(in.tank[0] / dp), nty = nint(in.tank[1] / dp), ntz = nint(in.tank[2] / dp);
    hi.nf = ncx * ncy * ncz;
    hi.nw = (ntx + 2 * L) * (nty + 2 * L) * (ntz + L) - ntx * nty * ntz;
    hi.no = in.has_obstacle
                ? nint(in.obstacle[3] / dp) * nint(in.obstacle[4] / dp) * nint(in.obstacle[5] / dp)
                : 0;
    hi.ng = in.has_gate ? nint(in.gate[3] / dp) * nint(in.gate[4] / dp) * nint(in.gate[5] / dp) : 0;

    Inst &d = hi.dev;
    std::memset(&d, 0, sizeof(d));
    double Ld = L * dp;
    double hi3[3] = {in.tank[0] + Ld, in.tank[1] + Ld, in.tank[2] + 4.0 * in.h};
    // with neighbour lists the cells hold the list radius 2h + s
    d.skin = p.list_skin * in.h;
    d.cs = (2.0 * in.h + d.skin) / effective_cell_div(p);
    d.inv_cs = 1.0 / d.cs;
    for (int a = 0; a < 3; ++a) {
        d.lo[a] = -Ld;
        d.n[a] = (int32_t)std::ceil((hi3[a] - d.lo[a]) / d.cs);
    }
    // a finer grid of the same box: halving the spacing (fine = 2) is exact, so a
    // particle's coarse cell is its fine cell divided by two
    d.cs /= fine;
    d.inv_cs *= fine;
    for (int a = 0; a < 3; ++a)
        d.n[a] *= fine;
    d.oc = d.cs;
    if (tiled) {
        int e;
        const double f = std::frexp(d.cs, &e);
        d.oc = std::ldexp(std::nearbyint(std::ldexp(f, 20)), e - 20);
    }
    d.ohf = (float)(0.5 * d.oc);
    d.centred = tiled && effective_cell_div(p) * fine == 1;
    for (int a = 0; a < 3; ++a)
        d.olo[a] = d.lo[a] + (d.centred ? 0.5 * d.oc : 0.0);
    d.ncells = d.n[0] * d.n[1] * d.n[2];
    d.by_nx = divisor(std::max(d.n[0], 1));
    d.by_ny = divisor(std::max(d.n[1], 1));
    d.h = in.h;
    d.c0 = in.c0;
    d.rho0 = in.rho0;
    d.alpha = in.alpha;
    d.delta = p.delta;
    d.gamma = p.gamma;
    d.g = p.g;
    d.cfl = p.cfl;
    d.dp = dp;
    d.mass = in.rho0 * dp * dp * dp;
    d.B = in.rho0 * in.c0 * in.c0 / p.gamma;
    d.eta2 = 0.01 * in.h * in.h;
    d.sup2 = (2.0 * in.h) * (2.0 * in.h);
    d.dt_min = p.dt_min;
    d.ztop = in.tank[2] + 4.0 * in.h;
    const double pi = 3.14159265358979323846;
    d.kW = 21.0 / (16.0 * pi * in.h * in.h * in.h);
    d.kF = 5.0 * d.kW / (in.h * in.h);
    d.half_inv_h = 0.5 / d.h;
    d.kFm = d.kF * d.mass;
    d.dfac_d = 2.0 * d.delta * d.h * d.c0;
    d.nah = -d.alpha * d.h;
    fill_fixed_point(d);
    d.csound = p.csound;
    d.delta_mode = p.delta_mode;
    d.nf = (int32_t)hi.nf;
    d.nw = (int32_t)hi.nw;
    d.no = (int32_t)hi.no;
    d.ng = (int32_t)hi.ng;
    d.np = (int32_t)(hi.nf + hi.nw + hi.no + hi.ng);
    for (int a = 0; a < 3; ++a) {
        d.gate_v[a] = in.has_gate ? in.gate_velocity[a] : 0.0;
        d.gate_vf[a] = (float)d.gate_v[a];
    }
    d.csf = (float)d.cs;
    d.hf = (float)d.h;
    d.inv_hf = (float)(1.0 / d.h);
    d.c0f = (float)d.c0;
    d.rho0f = (float)d.rho0;
    d.inv_rho0f = (float)(1.0 / d.rho0);
    d.alphaf = (float)d.alpha;
    d.massf = (float)d.mass;
    d.Bf = (float)d.B;
    d.eta2f = (float)d.eta2;
    d.sup2f = (float)d.sup2;
    d.list_r2f = (float)((2.0 * in.h + d.skin) * (2.0 * in.h + d.skin));
    d.half_skin2 = 0.25 * d.skin * d.skin;
    {
        // |x_f - x| <= |x| 2^-24 for a coordinate inside the grid; a difference
        // of two such copies is off by at most 2 coord_max 2^-24 per axis
        double coord_max = 0.0;
        for (int a = 0; a < 3; ++a)
            coord_max = std::fmax(coord_max, std::fmax(std::fabs(d.lo[a]), std::fabs(d.lo[a] + d.n[a] * d.cs)));
        const double eps = std::ldexp(coord_max, -22);  // twice the bound
        const double R = 2.0 * in.h + 2.0 * std::sqrt(3.0) * eps;
        d.sup2_filter = std::nextafter((float)(R * R * (1.0 + std::ldexp(1.0, -18))), 3.0e38f);
        const double Ri = std::fmax(2.0 * in.h - 2.0 * std::sqrt(3.0) * eps, 0.0);
        d.sup2_inner = std::nextafter((float)(Ri * Ri * (1.0 - std::ldexp(1.0, -18))), 0.0f);
    }
    d.kFf = (float)d.kF;
    d.dfac = (float)(2.0 * d.delta * d.h * d.c0);
    d.gammaf = (float)d.gamma;
    d.gf = (float)d.g;
}

// The tiled pair pass stages a tile of at least (2h)^3 with the cells within 2h of
// it: 6h each way.  On the particle lattice (the densest state of a weakly
// compressible flow, at its worst alignment) that has to fit the staging buffer,
// which it does for h < 7/3 dp; beyond, the neighbourhoods are staged in chunks by
// the other kernel (pair_wide.cuh).  Neighbour lists keep to that one too: their
// cells are wider than 2h.
bool tiles_fit(const sph_instance &in, const sph_params &p)
{
    const double n = std::floor(6.0 * in.h / in.dp * (1.0 + 1e-9)) + 1.0;
    return !(p.list_skin > 0) && n * n * n <= kStage;
}

// Cells per 2h of the tiled pass where callers see cells of 2h.  Cells of h leave fewer
// candidates to test, but hold less than 6 particles each below h = 1.75 dp, and rows of
// 2h fill the clusters better there (us per step, cells of 2h | h: 0.9 M particles h = 1.5 dp
// 772 | 890, 1.8 dp 1040 | 1036, 2.08 dp 1367 | 1292; 31 k particles 90 | 100, 91 | 94,
// 99 | 100).  The automatic size takes that below 48 k particles only (18 k at h = 1.5
// dp: 68 us, 78 with cells of h, 69 before the tiled pass): larger tanks get tiles whose
// FP32 frames are longer with cells of 2h, at 185 k particles 5 % less accurate.
int tile_cell_div(const std::vector<HostInst> &inst, int64_t n_total, bool automatic)
{
    double most = 0.0;
    for (const HostInst &hi : inst)
        most = std::max(most, hi.d.h / hi.d.dp);
    return most < 1.75 && (!automatic || n_total < 48000) ? 1 : 2;
}

// A larger tile stages fewer candidates per particle of its own (27 at (2h)^3, 18 at
// twice that length); it has to fit the staging buffer like the smallest, and there
// must be enough tiles to fill the GPU (2 CTAs on each of 152 SMs) four times over.
int64_t fill_tiles(std::vector<HostInst> &inst, int k, int64_t n_total)
{
    int64_t base = 0;
    for (HostInst &hi : inst) {
        Inst &d = hi.dev;
        const double c = d.cs / d.dp;  // cell size in particle spacings
        int best[3] = {k, k, k};
        double most = k * k * k * c * c * c;
        for (int tz = k; tz <= 2 * k; tz += k)
            for (int ty = tz; ty <= 2 * k; ty += k)
                for (int tx = k; tx <= 4 * k; ++tx) {
                    if (ty * tz > 16 || (ty + 2 * k) * (tz + 2 * k) > 96)
                        continue;
                    const double staged = (std::floor((tx + 2 * k) * c) + 1) * (std::floor((ty + 2 * k) * c) + 1) *
                                          (std::floor((tz + 2 * k) * c) + 1);
                    const double own = tx * ty * tz * c * c * c;
                    if (staged <= kStage && own * 1216 <= (double)n_total && own > most * 1.01) {
                        most = own;
                        best[0] = tx;
                        best[1] = ty;
                        best[2] = tz;
                    }
                }
        int64_t nt = 1;
        for (int a = 0; a < 3; ++a) {
            d.tdim[a] = best[a];
            d.ntile[a] = (d.n[a] + best[a] - 1) / best[a];
            nt *= d.ntile[a];
        }
        d.tile_base = (int32_t)base;
        base += nt;
    }
    return base;
}

void build_scene(const HostInst &hi, const sph_params &p, double *r, double *rho, uint8_t *type)
{
    const sph_instance &in = hi.d;
    double dp = in.dp;
    int64_t L = p.boundary_layers;
    int64_t ncx = nint(in.column[0] / dp), ncy = nint(in.column[1] / dp), ncz = nint(in.column[2] / dp);
    int64_t ntx = nint(in.tank[0] / dp), nty = nint(in.tank[1] / dp), ntz = nint(in.tank[2] / dp);
    int64_t id = 0;
    double gamma = p.gamma, g = p.g, c0 = in.c0, rho0 = in.rho0, hc = in.column[2];
    for (int64_t k = 0; k < ncz; ++k)
        for (int64_t j = 0; j < ncy; ++j)
            for (int64_t i = 0; i < ncx; ++i) {
                double z = (k + 0.5) * dp;
                r[3 * id] = (i + 0.5) * dp;
                r[3 * id + 1] = (j + 0.5) * dp;
                r[3 * id + 2] = z;
                // Eq. 8 inverted for the hydrostatic pressure rho0 g (Hc - z)
                rho[id] = p.init == SPH_INIT_HYDROSTATIC
                              ? rho0 * std::pow(1.0 + gamma * g * (hc - z) / (c0 * c0), 1.0 / gamma)
                              : rho0;
                type[id] = T_FLUID;
                ++id;
            }
    for (int64_t k = -L; k < ntz; ++k)
        for (int64_t j = -L; j < nty + L; ++j)
            for (int64_t i = -L; i < ntx + L; ++i) {
                if (i >= 0 && i < ntx && j >= 0 && j < nty && k >= 0)
                    continue;
                r[3 * id] = (i + 0.5) * dp;
                r[3 * id + 1] = (j + 0.5) * dp;
                r[3 * id + 2] = (k + 0.5) * dp;
                rho[id] = rho0;
                type[id] = T_WALL;
                ++id;
            }
    if (in.has_obstacle) {
        int64_t i0 = nint(in.obstacle[0] / dp), j0 = nint(in.obstacle[1] / dp), k0 = nint(in.obstacle[2] / dp);
        int64_t nx = nint(in.obstacle[3] / dp), ny = nint(in.obstacle[4] / dp), nz = nint(in.obstacle[5] / dp);
        for (int64_t k = k0; k < k0 + nz; ++k)
            for (int64_t j = j0; j < j0 + ny; ++j)
                for (int64_t i = i0; i < i0 + nx; ++i) {
                    r[3 * id] = (i + 0.5) * dp;
                    r[3 * id + 1] = (j + 0.5) * dp;
                    r[3 * id + 2] = (k + 0.5) * dp;
                    rho[id] = rho0;
                    type[id] = T_OBST;
                    ++id;
                }
    }
    if (in.has_gate) {
        int64_t i0 = nint(in.gate[0] / dp), j0 = nint(in.gate[1] / dp), k0 = nint(in.gate[2] / dp);
        int64_t nx = nint(in.gate[3] / dp), ny = nint(in.gate[4] / dp), nz = nint(in.gate[5] / dp);
        for (int64_t k = k0; k < k0 + nz; ++k)
            for (int64_t j = j0; j < j0 + ny; ++j)
                for (int64_t i = i0; i < i0 + nx; ++i) {
                    r[3 * id] = (i + 0.5) * dp;
                    r[3 * id + 1] = (j + 0.5) * dp;
                    r[3 * id + 2] = (k + 0.5) * dp;
                    rho[id] = rho0;
                    type[id] = T_GATE;
                    ++id;
                }
    }
}

}  // namespace sph
