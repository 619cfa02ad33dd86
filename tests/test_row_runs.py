"""The staged run of a row of cells (csrc/rows.h), compiled for the host: whatever
the cell starts hold, every index formed from a run stays in bounds."""
import os
import subprocess

from paper_2306_01959_gb300 import build

MAIN = r"""
#include <cassert>
#include <cstdio>
#include <random>
#include "rows.h"
using namespace sph;
static void check(int32_t a, int32_t e, int32_t ha, int32_t he, int32_t n)
{
    RowRun r;
    const bool ok = row_run(a, e, ha, he, n, r);
    assert(r.gs >= 0 && r.n >= 0 && r.n <= n - r.gs);            // sorted indices below n
    assert(r.hoff >= 0 && r.hlen >= 0 && r.hlen <= r.n - r.hoff);  // the tile's own run lies in it
    const bool sane = 0 <= a && a <= ha && ha <= he && he <= e && e <= n;
    assert(ok == sane);
    if (sane)
        assert(r.gs == a && r.n == e - a && r.gs + r.hoff == ha && r.hlen == he - ha);
    else
        assert(r.n == 0 && r.hlen == 0);
}
int main()
{
    std::mt19937 rng(2306);
    for (int k = 0; k < 2000000; ++k) {
        const int32_t n = rng() % 1000;
        int32_t v[4];
        for (int q = 0; q < 4; ++q)  // near the valid range, or any word
            v[q] = k & 1 ? (int32_t)(rng() % 1100) - 50 : (int32_t)rng();
        check(v[0], v[1], v[2], v[3], n);
        const int32_t a = rng() % (n + 1), ha = a + rng() % (n - a + 1), he = ha + rng() % (n - ha + 1);
        check(a, he + rng() % (n - he + 1), ha, he, n);  // a consistent row
    }
    check(0, 0x7fffffff, 0, 0x7fffffff, 0x7fffffff);
    std::puts("ok");
}
"""


def test_row_run_is_in_bounds_for_any_cell_starts(tmp_path):
    src, exe = tmp_path / "rows.cpp", tmp_path / "rows"
    src.write_text(MAIN)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ftrapv", "-I", build.SRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.strip() == "ok"


def test_cell_starts_are_read_in_one_place():
    # the staged slot and the sorted index of a cluster come from its row's one run
    text = open(os.path.join(build.SRC, "pair_mixed.cuh")).read()
    assert text.count("b.cell_start") == 1 and "row_run(" in text
