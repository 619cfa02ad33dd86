"""The cell of a coordinate by the product with 1/cs (csrc/grid.h), compiled for the host:
the floor of the rounded quotient, next to faces above all."""
import subprocess

from paper_2306_01959_gb300 import build

MAIN = r"""
#include <cstdio>
#include <limits>
#include <random>
#include "grid.h"
using namespace sph;
static long n_checked = 0;
static bool same(double d, double cs, int n)
{
    int a = -1, b = -1;
    const double inv = 1.0 / cs, f = std::floor(d / cs);
    const bool in = cell_of_product(d, cs, inv, n, a), ref = f >= 0.0 && f < n;
    (void)b;
    ++n_checked;
    if (in == ref && (!in || a == (int)f))
        return true;
    std::printf("d %.17g cs %.17g n %d: %d %d, quotient %.17g\n", d, cs, n, (int)in, a, d / cs);
    return false;
}
int main()
{
    std::mt19937_64 g(2306);
    std::uniform_real_distribution<double> U(0, 1);
    const double inf = std::numeric_limits<double>::infinity();
    for (int t = 0; t < 4000; ++t) {
        // spacings of every size, powers of two and lattice multiples among them
        double cs = std::exp2(30 * U(g) - 20);
        if (t % 4 == 1)
            cs = std::exp2(std::floor(std::log2(cs)));
        if (t % 4 == 2)
            cs = 0.01 * std::floor(1 + 400 * U(g)) / 4;
        const int n = (int)std::exp2(1 + 16.2 * U(g));  // up to 75,000: beyond 65,535 the quotient decides
        for (int k = 0; k < 400; ++k) {
            int face = (int)(U(g) * (n + 3)) - 1;
            if (k % 5 == 0)
                face = 1 << (int)(17 * U(g));
            double d = face * cs;
            const int e = (int)(U(g) * 4);
            if (e == 1)  // a few roundings off the face
                for (int s = (int)(U(g) * 9) - 4; s != 0; s += s < 0 ? 1 : -1)
                    d = std::nextafter(d, s < 0 ? -inf : inf);
            if (e == 2)
                d += cs * (U(g) - 0.5) * std::exp2(-60 * U(g));
            if (e == 3)
                d = cs * (U(g) * 1.2 - 0.1) * n;
            if (!same(d, cs, n))
                return 1;
        }
        for (double d : {0.0, -0.0, 5e-324, -5e-324, 1e300, -1e300, inf, -inf, std::nan(""), 65536 * cs, 65535 * cs,
                         -65536 * cs, std::exp2(36.0) * cs, std::exp2(37.0) * cs, std::exp2(52.0) * cs})
            if (!same(d, cs, n))
                return 1;
    }
    std::printf("ok %ld\n", n_checked);
}
"""


def test_floor_of_the_rounded_quotient(tmp_path):
    src, exe = tmp_path / "grid.cpp", tmp_path / "grid"
    src.write_text(MAIN)
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-ffp-contract=off", "-I", build.SRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.startswith("ok"), r.stdout
