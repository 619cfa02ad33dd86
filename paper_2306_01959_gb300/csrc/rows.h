// The run of sorted particles that a tile of the mixed pair pass stages from one
// row of cells (pair_mixed.cuh), and the part of it that the tile itself owns.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define SPH_HD __host__ __device__ __forceinline__
#else
#define SPH_HD inline
#endif

namespace sph {

struct RowRun {
    int32_t gs, n;       // first sorted particle and length of the staged run
    int32_t hoff, hlen;  // the tile's own particles, from gs on
};

// The runs from the cell starts of the staged cells [a, e) and of the tile's own
// cells [ha, he) of the row, n_in sorted particles in all.  Every index that the
// pass forms comes from this one set of four values, so that whatever they hold, a
// staged slot lies in its row and a sorted index below n_in: values that no cell
// structure has give an empty run, and false.
SPH_HD bool row_run(int32_t a, int32_t e, int32_t ha, int32_t he, int32_t n_in, RowRun &r)
{
    const bool ok = a >= 0 && a <= ha && ha <= he && he <= e && e <= n_in;
    r.gs = ok ? a : 0;
    r.n = ok ? e - a : 0;
    r.hoff = ok ? ha - a : 0;
    r.hlen = ok ? he - ha : 0;
    return ok;
}

}  // namespace sph
