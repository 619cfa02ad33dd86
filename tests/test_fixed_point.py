"""The integer arithmetic of the FP64 pair pass (csrc/fixed.h), compiled for the host
and compared with extended precision: each result is rounded once, wherever the
pair lies."""
import subprocess

import pytest

from paper_2306_01959_gb300 import build

# Bounds, with u = 2^-53 (one rounding) and the position's unit of at most 2^-62 of 2h:
# - r_ij, a component: its rounding, and one unit where doubles are finer than it;
# - |r_ij|^2 + eta^2, eta = 0.05 of 2h: a unit of each component changes it by at most
#   2 sqrt(3) r 2^-62 / (r^2 + eta^2) < 2^-56.8 relative; the sums themselves lose 2^-81;
# - t^3: its rounding, and the error of t, below 2^-59 (the units above, 2^-62 each of
#   root, product with 1/2h and residual), three times over, relative to t;
# - the reciprocal: its rounding, that of its argument above, E^3 of the start
#   (2^-68) and the truncations of its products, below 2^-57.
MAIN = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include "fixed.h"
using namespace sph;
typedef long double Q;
int main(int argc, char **argv)
{
    const double base = atof(argv[1]), h2s[] = {0.0625, 0.0625 * (1 + 1e-15), 0.083, 0.1249999, 3.1e-4, 7.7};
    std::mt19937_64 g(2306);
    std::uniform_real_distribution<double> U(0, 1);
    std::normal_distribution<double> G;
    const Q u = 0x1p-53L;
    long n = 0;
    for (double h2 : h2s) {
        const double h = 0.5 * h2, eta2 = 0.01 * h * h;
        const int s = 62 - std::ilogb(h2);
        const uint64_t H = (uint64_t)std::ldexp(h2, s);
        const unsigned __int128 k = ((unsigned __int128)1 << 126) / H;
        const uint64_t kh = k >> 64 ? ~0ull : (uint64_t)k;
        const double es = std::ldexp(eta2, 2 * s - 64);
        Fixed2 eta = {(uint64_t)es, (uint32_t)std::ldexp(es - (double)(uint64_t)es, 32)};
        for (int i = 0; i < 150000; ++i) {
            double x[2][3], d[3], m = 0;
            for (double &q : d) {
                q = G(g);
                m += q * q;
            }
            const double gap = (i & 1 ? std::exp2(-6.0 * U(g)) : 1.0 - std::exp2(-20.0 * U(g))) * h2;
            for (int a = 0; a < 3; ++a) {
                x[0][a] = base * h2 * (U(g) + (base > 1)) + (U(g) - 0.5) * h2;
                x[1][a] = x[0][a] + d[a] / std::sqrt(m) * gap;
            }
            host_approx_error() = (2 * U(g) - 1) * 1.27e-7;  // 2^-22.9
            int64_t D[3];
            Q r2 = 0;
            for (int a = 0; a < 3; ++a) {
                const Q e = (Q)x[1][a] - x[0][a];
                r2 += e * e;
                D[a] = (int64_t)((uint64_t)fixed_position(x[1][a], s) - (uint64_t)fixed_position(x[0][a], s));
                const Q err = fabsl((Q)std::ldexp(int_to_double(D[a]), -s) - e);
                if (err > u * fabsl(e) * 1.001L + ldexpl(1, -s))
                    return std::printf("r_ij\n"), 1;
            }
            const Q r = sqrtl(r2), t = 1 - r / h2, V = r2 + eta2;
            const Fixed2 f = fixed_dist2(D[0], D[1], D[2]);
            if (r >= h2 || f.R < (1ull << 48))
                continue;
            ++n;
            Fixed2 v;
            v.f = f.f + eta.f;
            v.R = f.R + eta.R + (v.f < f.f);
            const Q vv = ((Q)v.R + ldexpl(v.f, -32)) * ldexpl(1, 64 - 2 * s);
            if (fabsl(vv / V - 1) > 0x1p-56L)
                return std::printf("r^2 %Lg\n", fabsl(vv / V - 1)), 1;
            const Q e3 = fabsl((Q)fixed_t3(f, kh) / (t * t * t) - 1);
            if (e3 > u * 1.001L + 3 * 0x1p-59L / t + 0x1p-58L)
                return std::printf("t3 %Lg at t = %Lg\n", e3, t), 1;
            const double rho = 1000 * std::exp2(20 * U(g) - 10);
            const Q er = fabsl((Q)fixed_rcp(v, rho) * rho * ldexpl(V, 2 * s - 64) - 1);
            if (er > u + 0x1p-55L)
                return std::printf("reciprocal %Lg\n", er), 1;
        }
    }
    std::printf("ok %ld\n", n);
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed")
    (d / "fixed.cpp").write_text(MAIN)
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-ffp-contract=off", "-I", build.SRC, str(d / "fixed.cpp"), "-o",
                    str(d / "fixed")], check=True)
    return str(d / "fixed")


# supports from the coordinate planes: at them, near them, along a tank, and where
# positions exceed 2^63 units (from one support on) and 2^64 (from two) many times over
@pytest.mark.parametrize("base", [0, 1e-3, 1, 40, 3000])
def test_rounded_once(exe, base):
    out = subprocess.run([exe, str(base)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.startswith("ok"), out.stdout
    assert int(out.stdout.split()[1]) > 500000
