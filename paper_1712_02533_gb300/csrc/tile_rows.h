// Row ranges of the step kernels' tiles, for host and device alike.
#pragma once

#ifdef __CUDACC__
#define REG_HD __host__ __device__ __forceinline__
#else
#define REG_HD inline
#endif

// Node rows of one warp in a gradient tile of h rows from row tile0 of a level of n
// rows, the tile cut into `parts` runs of rows (1: one warp walks all of it).  The warp
// owns [r0, rEnd); its walk visits first .. last, one halo row on either side of them,
// and a visited row is loaded if it lies on the level.  Since n = 2^l + 1 and h divides
// 2^l, the last row of tiles owns the single row n - 1: every other warp of such a tile
// starts past the level, owns nothing and visits nothing (last < first).
struct GradRows {
    int r0, rEnd, first, last;
};

REG_HD GradRows grad_rows(int tile0, int h, int n, int part, int parts)
{
    const int len = h / parts;
    GradRows g;
    g.r0 = tile0 + part * len;
    g.rEnd = g.r0 + len < n ? g.r0 + len : n;
    g.first = g.r0 - 1;
    g.last = g.r0 < n ? g.rEnd : g.first - 1;
    return g;
}

// Whether the walk loads row r.
REG_HD bool grad_loads(const GradRows &g, int r, int n) { return r >= g.first && r <= g.last && r >= 0 && r < n; }

// Gradient tiles of an operator at a level of n rows and columns, and the most that any
// of its nl levels has, tiles of `width` owned columns by rows[k] rows: with rows set
// per level a coarser level can have more tiles than the finest.
REG_HD int grad_tiles(int n, int rows, int width) { return ((n + width - 1) / width) * ((n + rows - 1) / rows); }

REG_HD int most_grad_tiles(const int *n, const int *rows, int nl, int width)
{
    int m = 0;
    for (int k = 0; k < nl; k++) {
        const int t = grad_tiles(n[k], rows[k], width);
        m = t > m ? t : m;
    }
    return m;
}
