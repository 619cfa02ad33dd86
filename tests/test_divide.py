"""Division by a number known beforehand (csrc/divide.h), compiled for the host."""
import subprocess

from paper_2306_01959_gb300 import build

MAIN = r"""
#include <cstdio>
#include <random>
#include "divide.h"
using namespace sph;
static bool ok(int32_t a, int32_t d) { return divide(a, divisor(d)) == a / d; }
int main()
{
    std::mt19937 g(2306);
    const int32_t top = 0x7fffffff;
    for (int32_t d = 1; d <= 3000; ++d)  // small divisors: around every kind of quotient
        for (int k = 0; k < 2000; ++k) {
            const int32_t a = k < 600 ? k : (k < 700 ? top - (k - 600) : (int32_t)(g() & top));
            const int32_t edge = a / d * d;
            if (!ok(a, d) || !ok(edge, d) || (edge && !ok(edge - 1, d)))
                return std::printf("%d / %d\n", a, d), 1;
        }
    for (int k = 0; k < 3000000; ++k) {
        const int32_t d = (int32_t)((g() & top) >> (g() % 31)) | 1, a = (int32_t)(g() & top), edge = a / d * d;
        if (!ok(a, d) || !ok(edge, d) || (edge && !ok(edge - 1, d)) || !ok(top, d) || !ok(a, top) || !ok(top, top))
            return std::printf("%d / %d\n", a, d), 1;
    }
    for (int s = 0; s < 31; ++s)
        for (int e = -1; e <= 1; ++e)
            if ((1 << s) + e >= 1 && (!ok(top, (1 << s) + e) || !ok((1 << s) + e, (1 << s) + e)))
                return std::printf("2^%d\n", s), 1;
    std::puts("ok");
}
"""


def test_quotients_are_exact(tmp_path):
    src, exe = tmp_path / "divide.cpp", tmp_path / "divide"
    src.write_text(MAIN)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", build.SRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
