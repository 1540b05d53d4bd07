// Row ranges of the step kernels' tiles, for host and device alike.
#pragma once

#ifdef __CUDACC__
#define REG_HD __host__ __device__ __forceinline__
#else
#define REG_HD inline
#endif

// Node rows of one warp in a gradient tile of h rows from row tile0 of a level of n
// rows, the tile cut into `parts` runs of rows.  The warp owns r0 .. rLast; its walk
// visits r0 - 1 .. rLast + 1, one halo row on either side, and loads those of them that
// lie on the level: the first one before the walk (grad_loads_first), row r + 1 while it
// works on row r (r + 1 < n && r + 1 <= rLast + 1).  Since n = 2^l + 1 and h divides 2^l,
// the last row of tiles owns the single row n - 1: every other warp of a tile there starts
// past the level, owns nothing and visits nothing (r0 - 1 > rLast + 1).
struct GradRows {
    int r0, rLast;
};

REG_HD GradRows grad_rows(int tile0, int h, int n, int part, int parts)
{
    GradRows g;
    g.r0 = tile0 + part * (h / parts);
    g.rLast = g.r0 + h / parts - 1 < n - 1 ? g.r0 + h / parts - 1 : n - 1;
    if (g.r0 >= n) g.r0 = n + 2;
    return g;
}

REG_HD bool grad_loads_first(int r0, int n) { return r0 - 1 >= 0 && r0 - 1 < n; }

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
