// CUDA kernels of libreg (sm_103a).
//
// Grid conventions: level l is the vertex grid of n = 2^l + 1 nodes per side;
// node (r, c) is row r (x_1), column c (x_0).  Displacements are kept in grid
// units of their level (1 unit = one node spacing h = 2^-l), which keeps the
// sub-node position of a sample exact in float: the integer node index and the
// small displacement are split before they are added.  Frames are stored
// normalised per level (FE mean 0, FE standard deviation 1): NCC is invariant
// under affine changes of either image and bilinear interpolation commutes
// with them, so the energy and its gradient are those of the raw frames.
//
// Energies are sums over cells of the Q1 element integrals (exact FE mass and
// stiffness forms); per-cell values are float, per-warp and per-tile sums
// float (level-start sums: float triples), and the per-operator sum over tiles
// runs in float triples, exact to 2^-72, and goes on in double (the energies that
// the Armijo test compares).
#include <algorithm>

#include "reg_common.cuh"
#include "tile_rows.h"

namespace {

__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ double warp_sum_d(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

template <bool BF16>
__device__ __forceinline__ float ldimg(const void *p, int idx)
{
    if constexpr (BF16) {
        unsigned short raw = __ldg(reinterpret_cast<const unsigned short *>(p) + idx);
        return __uint_as_float(((unsigned)raw) << 16);
    } else {
        return __ldg(reinterpret_cast<const float *>(p) + idx);
    }
}

// Bilinear interpolant of a nodal image at grid point (c + vx, r + vy),
// clamped to the grid [0, n-1]^2 (= Omega).  Cell index floor(x), capped at
// n-2 (the right/top cell on the last node line).  Derivatives in grid units,
// zero in a clamped coordinate.
template <bool BF16, bool GRAD>
__device__ __forceinline__ float sample(const void *img, int n, int pitch, int c, int r, float vx, float vy,
                                        float *gx, float *gy)
{
    float fx = floorf(vx), fy = floorf(vy);
    int jx = c + (int)fx, jy = r + (int)fy;
    float ax = vx - fx, ay = vy - fy;
    bool clx = false, cly = false;
    if (jx < 0) {
        jx = 0; ax = 0.f; clx = true;
    } else if (jx >= n - 1) {
        clx = (jx > n - 1) || (ax > 0.f);
        jx = n - 2; ax = 1.f;
    }
    if (jy < 0) {
        jy = 0; ay = 0.f; cly = true;
    } else if (jy >= n - 1) {
        cly = (jy > n - 1) || (ay > 0.f);
        jy = n - 2; ay = 1.f;
    }
    int i0 = jy * pitch + jx;
    float t00 = ldimg<BF16>(img, i0), t01 = ldimg<BF16>(img, i0 + 1);
    float t10 = ldimg<BF16>(img, i0 + pitch), t11 = ldimg<BF16>(img, i0 + pitch + 1);
    float v = (1.f - ay) * ((1.f - ax) * t00 + ax * t01) + ay * ((1.f - ax) * t10 + ax * t11);
    if constexpr (GRAD) {
        *gx = clx ? 0.f : (1.f - ay) * (t01 - t00) + ay * (t11 - t10);
        *gy = cly ? 0.f : (1.f - ax) * (t10 - t00) + ax * (t11 - t01);
    }
    return v;
}

// sample() at a compensated displacement (exact cell choice at cell lines).
template <bool BF16, bool GRAD>
__device__ __forceinline__ float sample_df(const void *img, int n, int pitch, int c, int r, float4 u, float *gx,
                                           float *gy)
{
    int ix, iy;
    float ax, ay;
    df_split(u.x, u.z, ix, ax);
    df_split(u.y, u.w, iy, ay);
    int jx = c + ix, jy = r + iy;
    bool clx = false, cly = false;
    if (jx < 0) {
        jx = 0; ax = 0.f; clx = true;
    } else if (jx >= n - 1) {
        clx = (jx > n - 1) || (ax > 0.f);
        jx = n - 2; ax = 1.f;
    }
    if (jy < 0) {
        jy = 0; ay = 0.f; cly = true;
    } else if (jy >= n - 1) {
        cly = (jy > n - 1) || (ay > 0.f);
        jy = n - 2; ay = 1.f;
    }
    int i0 = jy * pitch + jx;
    float t00 = ldimg<BF16>(img, i0), t01 = ldimg<BF16>(img, i0 + 1);
    float t10 = ldimg<BF16>(img, i0 + pitch), t11 = ldimg<BF16>(img, i0 + pitch + 1);
    float v = (1.f - ay) * ((1.f - ax) * t00 + ax * t01) + ay * ((1.f - ax) * t10 + ax * t11);
    if constexpr (GRAD) {
        *gx = clx ? 0.f : (1.f - ay) * (t01 - t00) + ay * (t11 - t10);
        *gy = cly ? 0.f : (1.f - ax) * (t10 - t00) + ax * (t11 - t01);
    }
    return v;
}

// Bilinear interpolant of a float2 field (for composition), clamped.
__device__ __forceinline__ float2 sample2(const float2 *f, int n, int pitch, int c, int r, float vx, float vy)
{
    float fx = floorf(vx), fy = floorf(vy);
    int jx = c + (int)fx, jy = r + (int)fy;
    float ax = vx - fx, ay = vy - fy;
    if (jx < 0) { jx = 0; ax = 0.f; } else if (jx >= n - 1) { jx = n - 2; ax = 1.f; }
    if (jy < 0) { jy = 0; ay = 0.f; } else if (jy >= n - 1) { jy = n - 2; ay = 1.f; }
    int i0 = jy * pitch + jx;
    float2 a = f[i0], b = f[i0 + 1], cc = f[i0 + pitch], d = f[i0 + pitch + 1];
    float2 o;
    o.x = (1.f - ay) * ((1.f - ax) * a.x + ax * b.x) + ay * ((1.f - ax) * cc.x + ax * d.x);
    o.y = (1.f - ay) * ((1.f - ax) * a.y + ax * b.y) + ay * ((1.f - ax) * cc.y + ax * d.y);
    return o;
}

__device__ __forceinline__ int find_entry(const int *pref, int nent, int item)
{
    // largest e with pref[e] <= item
    int lo = 0, hi = nent - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (__ldg(pref + mid) <= item) lo = mid; else hi = mid - 1;
    }
    return lo;
}

}  // namespace

// ---------------------------------------------------------------------------
// Pyramid construction
// ---------------------------------------------------------------------------

// Restriction 1/16 [1 2 1; 2 4 2; 1 2 1] with mirrored boundary.  grid: (x tiles, y
// tiles, images); node (r, c) of a fine image z is fine[z fstride + min(r, lim)
// fpitch + min(c, lim)]: lim < nf - 1 embeds a frame of lim + 1 pixels on the
// vertex grid by repeating its last row and column, without a copy of it.
__global__ void k_restrict_img(const float *__restrict__ fine, int64_t fstride, int64_t fpitch, int nf, int lim,
                               float *__restrict__ coarse, int64_t cstride, int cpitch)
{
    int z = blockIdx.z;
    int nc = (nf + 1) / 2;
    int J = blockIdx.x * blockDim.x + threadIdx.x, I = blockIdx.y * blockDim.y + threadIdx.y;
    if (I >= nc || J >= nc) return;
    const float *F = fine + z * fstride;
    const float w[3] = {0.25f, 0.5f, 0.25f};
    float s = 0.f;
#pragma unroll
    for (int a = -1; a <= 1; a++) {
        int r = 2 * I + a;
        r = min(r < 0 ? -r : (r > nf - 1 ? 2 * (nf - 1) - r : r), lim);
#pragma unroll
        for (int b = -1; b <= 1; b++) {
            int c = 2 * J + b;
            c = min(c < 0 ? -c : (c > nf - 1 ? 2 * (nf - 1) - c : c), lim);
            s += w[a + 1] * w[b + 1] * F[(int64_t)r * fpitch + c];
        }
    }
    coarse[z * cstride + (int64_t)I * cpitch + J] = s;
}

// One raw level of the images under construction, node access as above.
__device__ __forceinline__ const float *level_row(const RawLevel &L, int z, int r)
{
    return L.img + z * L.stride + (int64_t)min(r, L.lim) * L.pitch;
}

// Per image and level: FE mean (w^T F) and FE standard deviation ((F-mean)^T M
// (F-mean))^1/2, two passes over the cells, summed in double.  Each image's cell
// rows are cut into STATS_SPLIT parts, one block each (grid: parts x levels,
// images); the parts' sums go to `part` and are added in order by
// k_image_stats_fin (deterministic).
constexpr int STATS_SPLIT = 32;

__device__ __forceinline__ double block_sum_d(double v, double *red)
{
    v = warp_sum_d(v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) t += red[w];
    __syncthreads();
    return t;
}

// PASS 0: sum of the cell means; PASS 1: sum of the cell mass forms of F - mean.
// Each cell's term in FP32, their sum in FP64 (GB300's FP64 rate is a small
// fraction of its FP32 rate): a thread adds its cells of a row (columns t, t + 256,
// ..) in FP32, then the row's share in FP64.  PASS 1 centres on the FP64 mean
// rounded to FP32: the cell form's linear term in that offset sums to zero (M 1 = w
// and sum w (F - mean) = 0), so only its square, ~1e-14 of the variance, remains.
// A row is loaded once, two columns per cell (its lower edge is the next row's
// upper one), STATS_COLS columns per thread at a time with the next row in flight;
// four loads per cell and one row at a time left the pass at 1.2 TB/s of the images
// (134 us for 40 x 1025^2).
constexpr int STATS_COLS = 4;  // 4 x 256 columns: sides up to 1024 in one sweep
template <int PASS>
__global__ void __launch_bounds__(256) k_image_stats_part(const RawLevels lv, const double *__restrict__ stats,
                                                          int n_img, double *__restrict__ part)
{
    __shared__ double red[32];
    const int k = blockIdx.x / STATS_SPLIT, sp = blockIdx.x % STATS_SPLIT, z = blockIdx.y;
    const RawLevel L = lv.l[k];
    const int n = L.n, rows = n - 1, per = (rows + STATS_SPLIT - 1) / STATS_SPLIT;
    const int r0 = sp * per, r1 = min(rows, r0 + per);
    const float mf = PASS ? (float)stats[2 * ((int64_t)k * n_img + z)] : 0.f;
    double s = 0.0;
    if (n - 1 <= STATS_COLS * 256) {
        float p0[STATS_COLS], p1[STATS_COLS], q0[STATS_COLS], q1[STATS_COLS];
        auto load = [&](int r, float (&x0)[STATS_COLS], float (&x1)[STATS_COLS]) {
            const float *row = level_row(L, z, r);
#pragma unroll
            for (int j = 0; j < STATS_COLS; j++) {
                const int c = threadIdx.x + 256 * j;
                x0[j] = c < n - 1 ? row[min(c, L.lim)] : 0.f;
                x1[j] = c < n - 1 ? row[min(c + 1, L.lim)] : 0.f;
            }
        };
        auto step = [&](const float (&x0)[STATS_COLS], const float (&x1)[STATS_COLS], const float (&y0)[STATS_COLS],
                        const float (&y1)[STATS_COLS]) {
            float rs = 0.f;
#pragma unroll
            for (int j = 0; j < STATS_COLS; j++)
                if ((int)threadIdx.x + 256 * j < n - 1) {
                    if (!PASS) {
                        rs += 0.25f * ((x0[j] + x1[j]) + (y0[j] + y1[j]));
                    } else {
                        const float a = x0[j] - mf, b = x1[j] - mf, cc = y1[j] - mf, d = y0[j] - mf;  // cyclic
                        rs += 4.f * (a * a + b * b + cc * cc + d * d) + 4.f * (a * b + b * cc + cc * d + d * a) +
                              2.f * (a * cc + b * d);
                    }
                }
            s += (double)rs;
        };
        if (r0 < r1) {
            load(r0, p0, p1);
            load(r0 + 1, q0, q1);
            // the row after the cells' lower edge is loaded while they are summed
            for (int r = r0; r < r1; r++) {
                float t0[STATS_COLS], t1[STATS_COLS];
                load(min(r + 2, n - 1), t0, t1);
                step(p0, p1, q0, q1);
#pragma unroll
                for (int j = 0; j < STATS_COLS; j++) { p0[j] = q0[j]; p1[j] = q1[j]; q0[j] = t0[j]; q1[j] = t1[j]; }
            }
        }
    } else {
        for (int r = r0; r < r1; r++) {
            const float *x = level_row(L, z, r), *y = level_row(L, z, r + 1);
            float rs = 0.f;
            for (int c = threadIdx.x; c < n - 1; c += 256) {
                const int c1 = min(c + 1, L.lim);
                if (!PASS) {
                    rs += 0.25f * ((x[c] + x[c1]) + (y[c] + y[c1]));
                } else {
                    const float a = x[c] - mf, b = x[c1] - mf, cc = y[c1] - mf, d = y[c] - mf;  // cyclic
                    rs += 4.f * (a * a + b * b + cc * cc + d * d) + 4.f * (a * b + b * cc + cc * d + d * a) +
                          2.f * (a * cc + b * d);
                }
            }
            s += (double)rs;
        }
    }
    const double t = block_sum_d(s, red) * (PASS ? 1.0 / 36.0 : 1.0);
    if (threadIdx.x == 0) part[((int64_t)k * n_img + z) * STATS_SPLIT + sp] = t;
}

// One thread per image and level: the parts in order; pass 0 writes the mean, pass 1
// sigma, of the finest level into fstats too.
__global__ void k_image_stats_fin(const RawLevels lv, int n_img, int pass, const double *__restrict__ part,
                                  double *__restrict__ out, double *__restrict__ fstats)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_img * lv.nl) return;
    const int k = i / n_img, z = i % n_img, n = lv.l[k].n;
    double v[STATS_SPLIT];
#pragma unroll
    for (int q = 0; q < STATS_SPLIT; q++) v[q] = part[(int64_t)i * STATS_SPLIT + q];
    double t = 0.0;
#pragma unroll
    for (int q = 0; q < STATS_SPLIT; q++) t += v[q];
    const double h2 = 1.0 / ((double)(n - 1) * (n - 1));
    const double r = pass ? sqrt(t * h2) : t * h2;
    out[2 * i + pass] = r;
    if (k == lv.nl - 1) fstats[2 * z + pass] = r;
}

// doubles of scratch and results for n_img images of nl levels
int image_stats_doubles(int n_img, int nl) { return n_img * nl * (STATS_SPLIT + 2); }

// F~ = (F - mean) / sigma rounded to float, as FP64 arithmetic gives it: the
// quotient as an unevaluated sum of two floats (mean and 1 / sigma each as two), to
// about 2^-45; where that does not settle the rounding (one value in 10^5), in FP64.
// FP64 divisions of every pixel made the normalisation 860 us for 40 x 1025^2.
struct NormScale {
    float mh, ml, ih, il, eps;
    double m, s;
};

__device__ __forceinline__ float normalised(const NormScale &q, float x)
{
    float dh, dl;
    two_sum(x, -q.mh, dh, dl);
    const float e = dl - q.ml, ph = dh * q.ih;
    const float lo = fmaf(dh, q.ih, -ph) + fmaf(dh, q.il, e * q.ih);
    const float tol = fmaf(fabsf(ph), 2.2737368e-13f, q.eps);  // 2^-42
    const float a = ph + (lo - tol), b = ph + (lo + tol);
    if (a == b) return a;
    return (float)(((double)x - q.m) / q.s);
}

// Normalised images (stored as float or bf16) and their M~ R~ images at all levels:
// M~ R~ is the FE mass matrix in units of h^2, M1 (x) M1 with the 1D weights 1/6,
// 4/6, 1/6 (2/6 on the diagonal at the border), applied to the stored image.  The
// weights are taken as the integers 36 M~ and the sum is divided by 36 once, so that
// no rounded weight biases every node the same way.  The gradient and trial passes
// take the NCC terms int R~ phi_i from it.  A block normalises a 32 x 32 node tile
// and one node around it into shared memory and writes both images from there.
// grid (tiles of all levels, images).
template <bool BF16>
__global__ void __launch_bounds__(256) k_norm_mass(const RawLevels lv, const double *__restrict__ stats, int n_img,
                                                   char *__restrict__ out, float *__restrict__ mr, int64_t ostride)
{
    __shared__ float sh[34][35];
    __shared__ NormScale scale;
    const int z = blockIdx.y;
    int k = 0, tile = blockIdx.x;
    while (tile >= lv.tiles[k]) tile -= lv.tiles[k++];
    const RawLevel L = lv.l[k];
    const int n = L.n, tx = (n + 31) / 32, r0 = (tile / tx) * 32, c0 = (tile % tx) * 32;
    if (threadIdx.x == 0) {
        NormScale q;
        const double *st = stats + 2 * ((int64_t)k * n_img + z);
        q.m = st[0];
        q.s = st[1];
        const double inv = 1.0 / q.s;
        q.mh = (float)q.m;
        q.ml = (float)(q.m - (double)q.mh);
        q.ih = (float)inv;
        q.il = (float)(inv - (double)q.ih);
        q.eps = fabsf(q.mh) * q.ih * 2.2737368e-13f;
        scale = q;
    }
    __syncthreads();
    const int tc = threadIdx.x & 31, tr = threadIdx.x >> 5;
    auto value = [&](int r, int c) {
        float v = 0.f;
        if (r >= 0 && r < n && c >= 0 && c < n) v = normalised(scale, level_row(L, z, r)[min(c, L.lim)]);
        if (BF16) v = __bfloat162float(__float2bfloat16_rn(v));
        return v;
    };
#pragma unroll
    for (int q = 0; q < 5; q++) {
        const int lr = tr + 8 * q;
        if (lr < 34) sh[lr][tc + 1] = value(r0 - 1 + lr, c0 + tc);
    }
    if (threadIdx.x < 68) {
        const int lr = threadIdx.x >> 1, side = threadIdx.x & 1;
        sh[lr][side ? 33 : 0] = value(r0 - 1 + lr, side ? c0 + 32 : c0 - 1);
    }
    __syncthreads();
    const int c = c0 + tc;
    if (c >= n) return;
    const int64_t base = z * ostride + L.out;
    const float wc = (c == 0 || c == n - 1) ? 2.f : 4.f;
#pragma unroll
    for (int q = 0; q < 4; q++) {
        const int lr = tr + 8 * q, r = r0 + lr;
        if (r >= n) continue;
        const int64_t o = base + (int64_t)r * L.opitch + c;
        const float v = sh[lr + 1][tc + 1];
        if (BF16) reinterpret_cast<__nv_bfloat16 *>(out)[o] = __float2bfloat16_rn(v);
        else reinterpret_cast<float *>(out)[o] = v;
        // nodes past the grid are zero in the tile
        const float wr = (r == 0 || r == n - 1) ? 2.f : 4.f;
        float acc = 0.f;
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const float row = (sh[lr + a][tc] + wc * sh[lr + a][tc + 1]) + sh[lr + a][tc + 2];
            acc += (a == 1 ? wr : 1.f) * row;
        }
        mr[o] = acc / 36.f;
    }
}

// Statistics, normalised and M~ R~ images of n_img images from their raw levels
// (finest last): out and mr point at the first image's pyramid block, ostride
// elements apart; work: image_stats_doubles(n_img, nl).
void launch_pyramid(const RawLevels &lv, int n_img, int bf16, double *work, double *fstats, void *out, float *mr,
                    int64_t ostride, cudaStream_t st)
{
    double *stats = work, *part = work + 2 * (int64_t)n_img * lv.nl;
    const dim3 grid(STATS_SPLIT * lv.nl, n_img);
    const int nf = (n_img * lv.nl + 63) / 64;
    k_image_stats_part<0><<<grid, 256, 0, st>>>(lv, stats, n_img, part);
    k_image_stats_fin<<<nf, 64, 0, st>>>(lv, n_img, 0, part, stats, fstats);
    k_image_stats_part<1><<<grid, 256, 0, st>>>(lv, stats, n_img, part);
    k_image_stats_fin<<<nf, 64, 0, st>>>(lv, n_img, 1, part, stats, fstats);
    int tiles = 0;
    for (int k = 0; k < lv.nl; k++) tiles += lv.tiles[k];
    if (bf16) k_norm_mass<true><<<dim3(tiles, n_img), 256, 0, st>>>(lv, stats, n_img, (char *)out, mr, ostride);
    else k_norm_mass<false><<<dim3(tiles, n_img), 256, 0, st>>>(lv, stats, n_img, (char *)out, mr, ostride);
}

// ---------------------------------------------------------------------------
// Operator initialisation: composition and restriction of the initial guess
// ---------------------------------------------------------------------------

// init 1: U0 = left; init 2: U0(x) = left(x) + right(x + left(x)) (phi_jk o phi_ij,
// right sampled bilinearly, clamped).  grid: (x tiles, y tiles, ops).
__global__ void k_compose(BatchDev b)
{
    const OpDesc &op = b.ops[blockIdx.z];
    if (op.init == 0) return;
    const LevelDesc &L = op.lv[op.nl - 1];
    int c = blockIdx.x * blockDim.x + threadIdx.x, r = blockIdx.y * blockDim.y + threadIdx.y;
    if (r >= L.n || c >= L.n) return;
    float2 a = op.left[(int64_t)r * op.slot_pitch + c];
    if (op.init == 2) {
        float2 q = sample2(op.right, L.n, op.slot_pitch, c, r, a.x, a.y);
        a.x += q.x;
        a.y += q.y;
    }
    L.V[0][(int64_t)r * L.pitch + c].u = make_float4(a.x, a.y, 0.f, 0.f);
}

// Restrict U0 from level index k+1 to k (grid units halve).  grid (x, y, ops).
__global__ void k_restrict_u(BatchDev b, int step)
{
    const OpDesc &op = b.ops[blockIdx.z];
    int k = op.nl - 1 - step;  // destination level index
    if (op.init == 0 || k < 0) return;
    const LevelDesc &C = op.lv[k], &F = op.lv[k + 1];
    int J = blockIdx.x * blockDim.x + threadIdx.x, I = blockIdx.y * blockDim.y + threadIdx.y;
    if (I >= C.n || J >= C.n) return;
    int nf = F.n;
    const float w[3] = {0.25f, 0.5f, 0.25f};
    float sx = 0.f, sy = 0.f;
#pragma unroll
    for (int a = -1; a <= 1; a++) {
        int r = 2 * I + a;
        r = r < 0 ? -r : (r > nf - 1 ? 2 * (nf - 1) - r : r);
#pragma unroll
        for (int bb = -1; bb <= 1; bb++) {
            int c = 2 * J + bb;
            c = c < 0 ? -c : (c > nf - 1 ? 2 * (nf - 1) - c : c);
            float4 v = F.V[0][(int64_t)r * F.pitch + c].u;
            float ww = w[a + 1] * w[bb + 1];
            sx += ww * v.x;
            sy += ww * v.y;
        }
    }
    C.V[0][(int64_t)I * C.pitch + J].u = make_float4(0.5f * sx, 0.5f * sy, 0.f, 0.f);
}

// Identity initial guess: zero U0 on the coarsest level.  grid (x, y, ops).
__global__ void k_zero_u(BatchDev b)
{
    const OpDesc &op = b.ops[blockIdx.z];
    if (op.init != 0) return;
    const LevelDesc &C = op.lv[0];
    int c = blockIdx.x * blockDim.x + threadIdx.x, r = blockIdx.y * blockDim.y + threadIdx.y;
    if (r >= C.n || c >= C.n) return;
    C.V[0][(int64_t)r * C.pitch + c].u = make_float4(0.f, 0.f, 0.f, 0.f);
}

__global__ void k_init_state(BatchDev b, int n_ops)
{
    int o = blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= n_ops) return;
    OpState s;
    memset(&s, 0, sizeof(s));
    s.phase = PH_START;
    s.lvl = 0;
    s.cur = 0;
    s.src = 0;
    s.tau = b.tau_init;
    s.status = OPST_CONVERGED;
    b.st[o] = s;
}

// ---------------------------------------------------------------------------
// Work planning: compacted per-family op lists and tile prefix sums
// ---------------------------------------------------------------------------

constexpr int PLAN_WARP = 32;  // batches up to this wide are planned by every warp itself

// The next step of an operator, from its state: the tile counts and the
// description that the gradient and trial passes read.
__device__ __forceinline__ void set_step(OpState &s, const OpDesc &op)
{
    const LevelDesc &L = op.lv[s.lvl];
    s.tG = s.phase == PH_GRAD ? L.tg : 0;
    s.tT = s.phase == PH_DONE ? 0 : L.tt;
    StepDesc &d = s.step;
    d.T = L.T;
    d.MR = L.MR;
    d.Vs = s.phase == PH_PROLONG ? L.V[s.cur] : L.V[s.src];
    d.Vc = L.V[s.cur];
    const LevelDesc &C = op.lv[s.phase == PH_PROLONG ? s.lvl - 1 : s.lvl];
    d.VC = C.V[s.src];
    d.cpitch = C.pitch;
    d.phase = s.phase;
    d.n = L.n;
    d.pitch = L.pitch;
    d.hg = L.hg;
    d.ht = L.ht;
    d.ntr = s.ntr;
    d.part0 = op.part0;
    d.ih2 = 1.f / L.h2;
    d.isig = s.cur_ev.isig;
    d.c36 = s.cur_ev.c36;
    d.cT = s.cur_ev.cT;
}

// A warp's view of the step's work items (tiles of one family).  Batches of up to
// PLAN_WARP operators: lane l holds operator l's tile range, from one load and a
// warp scan.  Wider ones: the compacted lists (cnt = -1, incl = their length).
struct WorkPlan {
    int items, incl, cnt;
};

template <bool GRAD>
__device__ __forceinline__ WorkPlan work_plan(const BatchDev &b, int lane)
{
    WorkPlan w;
    const int2 p = b.plan[lane];  // (at least PLAN_WARP entries exist)
    const int n_ops = b.ctr[0];
    if (n_ops <= PLAN_WARP) {
        w.cnt = lane < n_ops ? (GRAD ? p.x : p.y) : 0;
        w.incl = w.cnt;
#pragma unroll
        for (int k = 1; k < 32; k <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, w.incl, k);
            if (lane >= k) w.incl += y;
        }
        w.items = __shfl_sync(0xffffffffu, w.incl, 31);
    } else {
        w.cnt = -1;
        w.incl = b.ctr[GRAD ? 2 : 3];
        w.items = b.ctr[GRAD ? 5 : 6];
    }
    return w;
}

// Operator of a work item and the item's tile index in it (warp-uniform).
template <bool GRAD>
__device__ __forceinline__ int find_item(const BatchDev &b, const WorkPlan &w, int item, int &tile)
{
    if (w.cnt >= 0) {
        const int o = __ffs(__ballot_sync(0xffffffffu, w.incl > item)) - 1;
        tile = item - __shfl_sync(0xffffffffu, w.incl - w.cnt, o);
        return o;
    }
    const int *pref = GRAD ? b.prefG : b.prefT;
    const int e = find_entry(pref, w.incl, item);
    tile = item - pref[e];
    return (GRAD ? b.listG : b.listT)[e];
}

// The lists and tile prefixes of the next step from the operators' plan entries,
// by one block of REG_CTL_THREADS threads: one scan of {entries, gradient tiles,
// trial tiles} per REG_CTL_THREADS operators.  (An operator with gradient tiles
// always has trial tiles.)
__device__ void plan_lists(const BatchDev &b)
{
    __shared__ int4 wsum[REG_CTL_THREADS / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int n_ops = b.ctr[0];
    int offG = 0, offT = 0, itG = 0, itT = 0;  // entries and tiles of the operators before this chunk
    for (int base = 0; base < n_ops; base += REG_CTL_THREADS) {
        const int o = base + threadIdx.x;
        // other blocks wrote the entries in this launch: past L1
        const int2 p = o < n_ops ? __ldcg(b.plan + o) : make_int2(0, 0);
        // entries of both lists in one word (at most REG_CTL_THREADS each)
        const int inc = (p.x > 0 ? 1 : 0) | (p.y > 0 ? 1 << 16 : 0);
        int e = inc, g = p.x, t = p.y;
#pragma unroll
        for (int k = 1; k < 32; k <<= 1) {
            const int ye = __shfl_up_sync(0xffffffffu, e, k), yg = __shfl_up_sync(0xffffffffu, g, k),
                      yt = __shfl_up_sync(0xffffffffu, t, k);
            if (lane >= k) { e += ye; g += yg; t += yt; }
        }
        if (lane == 31) wsum[wid] = make_int4(e, g, t, 0);
        __syncthreads();
        int4 before = make_int4(0, 0, 0, 0), all = before;
#pragma unroll
        for (int w = 0; w < REG_CTL_THREADS / 32; w++) {
            const int4 x = wsum[w];
            if (w < wid) { before.x += x.x; before.y += x.y; before.z += x.z; }
            all.x += x.x; all.y += x.y; all.z += x.z;
        }
        const int ex = e - inc + before.x;
        if (p.x > 0) {
            b.listG[offG + (ex & 0xffff)] = o;
            b.prefG[offG + (ex & 0xffff)] = itG + g - p.x + before.y;
        }
        if (p.y > 0) {
            b.listT[offT + (ex >> 16)] = o;
            b.prefT[offT + (ex >> 16)] = itT + t - p.y + before.z;
        }
        offG += all.x & 0xffff;
        offT += all.x >> 16;
        itG += all.y;
        itT += all.z;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        b.prefG[offG] = itG;
        b.prefT[offT] = itT;
        b.ctr[2] = offG;
        b.ctr[3] = offT;
        b.ctr[5] = itG;
        b.ctr[6] = itT;
    }
}

// Plan of a batch's first step from the operators' states (the control kernel
// plans the others).
__global__ void __launch_bounds__(REG_CTL_THREADS) k_plan(BatchDev b)
{
    const int n_ops = b.ctr[0];
    for (int o = threadIdx.x; o < n_ops; o += REG_CTL_THREADS) {
        set_step(b.st[o], b.ops[o]);
        b.plan[o] = make_int2(b.st[o].tG, b.st[o].tT);
    }
    __threadfence();
    __syncthreads();
    if (n_ops > PLAN_WARP) plan_lists(b);
    if (threadIdx.x == 0) b.ctr[7] = n_ops;
}

// ---------------------------------------------------------------------------
// Prolongation to the next level of the multilevel flow, and the result.
// ---------------------------------------------------------------------------
namespace {

// u + tau d of the coarser level at node (r, c) of the next one: 2 x bilinear
// prolongation (coarse grid unit = 2 fine units); the weights 2, 1, 1/2 are
// exact, the sum is compensated.
__device__ __forceinline__ float4 prolong_node(const NodeRec *V, int cpitch, float tau, int r, int c)
{
    const int I = r >> 1, J = c >> 1, oi = r & 1, oj = c & 1;
    const float w2 = (oi ? 0.5f : 1.f) * (oj ? 0.5f : 1.f) * 2.f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int a = 0; a <= 1; a++)
#pragma unroll
        for (int bb = 0; bb <= 1; bb++) {
            if ((a && !oi) || (bb && !oj)) continue;
            const int64_t idx = (int64_t)(I + a) * cpitch + (J + bb);
            float4 u = V[idx].u;
            if (tau != 0.f) {
                float2 d = V[idx].d;
                u = df_add2(u, tau * d.x, tau * d.y);
            }
            df_add(acc.x, acc.z, w2 * u.x);
            df_add(acc.x, acc.z, w2 * u.z);
            df_add(acc.y, acc.w, w2 * u.y);
            df_add(acc.y, acc.w, w2 * u.w);
        }
    return acc;
}

}  // namespace

// The finest level's u with its pending step into the destination slots, once
// all operators of the batch are done (their workspaces are their own, so the
// records wait there).  grid (x tiles, y tiles, ops), block (32, 8).
__global__ void __launch_bounds__(256) k_final(BatchDev b)
{
    const OpDesc &op = b.ops[blockIdx.z];
    const LevelDesc &Lv = op.lv[op.nl - 1];
    const int n = Lv.n;
    if ((int)(blockIdx.x * 32) >= n || (int)(blockIdx.y * 8) >= n) return;  // block-uniform
    const int c = blockIdx.x * 32 + threadIdx.x, r = blockIdx.y * 8 + threadIdx.y;
    const OpState &s = b.st[blockIdx.z];
    float corr = 0.f;  // judged ops: |final - learned start|
    if (r < n && c < n) {
        const float tau = (float)s.tau_acc;
        const NodeRec &v = Lv.V[s.src][(int64_t)r * Lv.pitch + c];
        float4 u = v.u;
        if (tau != 0.f) {
            float2 d = v.d;
            u = df_add2(u, tau * d.x, tau * d.y);
        }
        const float2 res = make_float2(u.x + u.z, u.y + u.w);
        float2 &dst = op.out[(int64_t)r * op.slot_pitch + c];
        if (op.judge) {
            const float2 g0 = dst;
            corr = fabsf(res.x - g0.x) + fabsf(res.y - g0.y);
        }
        dst = res;
    }
    if (op.judge) {  // block-uniform
        const float w = warp_sum(corr);
        if (threadIdx.x == 0) atomicAdd(&b.st[blockIdx.z].corr, (double)w);
    }
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0 && threadIdx.y == 0)
        atomicAdd(&b.work[KW_PFIN], (unsigned long long)n * n);
}

// ---------------------------------------------------------------------------
// G: accept the pending step (u <- u + tau d) and compute the L2 gradient-flow
// direction at the new u:
//   dNCC/dThat_i = h^2 [ (M~ R~)_i / sigma_T - NCC (M~ (That - T_bar))_i / sigma_T^2 ]
//   psi_{i,c}    = -[...] dT_c(i) + lambda (K u_c)_i            (dE/du~ = h^2 psi)
//   d_{i,c}      = -psi_{i,c} / (h^2 omega_i)                  (d = -g / w, w = h^2 omega)
//   slope        = g^T d = -sum psi^2 / omega
//   Qud          = u^T K d = sum_i d_i . (K u)_i
// with M~ = M1 (x) M1 and K = K1 (x) M1 + M1 (x) K1 (1D mass M1 = [1 4 1] / 6,
// 2/6 on the diagonal at the border; 1D stiffness K1 = [-1 2 -1], 1 on the
// diagonal at the border), applied as separable stencils with the integer
// weights 6 M1 and 6 K1: along the column in registers, along the row by
// shuffles; the scale 1/36 or 1/6 is folded into per-tile coefficients, so that
// no rounded weight biases every node alike.  M~ R~ comes with the pyramid;
// 36 M~ That is stored for the trial passes of the search.  Strip tile: 30
// owned node columns by Lv.hg owned rows, one halo node around them.
// ---------------------------------------------------------------------------
// FEW false (many tiles): one tile per warp, whose walk down 32 rows amortises the
// halo rows.  FEW true: a block shares a tile, each warp a quarter of its rows, since
// the length of the walk, a record -> template latency per row, is then the pass's
// length; the rows' terms of the two sums go through shared memory and are added
// in row order, so that both forms give the same sums.  Per launch of a single 1024^2
// operator 14.5 -> 8 us, of 7 operators of 64^2 8.2 -> 4.9, of a 21 x 512^2 scan 20 ->
// 14; of a 33 x 1024^2 scan 67 us as it was (57 now), 83 us with tiles shared.
constexpr int GRAD_WARPS = REG_STRIP_THREADS / 32;
template <bool BF16, bool FEW>
__global__ void __launch_bounds__(REG_STRIP_THREADS, FEW ? 6 : 8) k_grad(BatchDev b)
{
    __shared__ float2 rows[FEW ? 64 : 1][32];
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int nwarps = gridDim.x * (FEW ? 1 : GRAD_WARPS);
    for (int item = FEW ? blockIdx.x : blockIdx.x * GRAD_WARPS + (threadIdx.x >> 5);; item += nwarps) {
        // read again for every tile: held in registers over the row walk it spills
        const WorkPlan wp = work_plan<true>(b, lane);
        if (item >= wp.items) break;
        int t;
        const StepDesc &s = b.st[find_item<true>(b, wp, item, t)].step;
        const int n = s.n, pitch = s.pitch, ntx = (n + REG_GW - 1) / REG_GW, h = s.hg;
        const int part = s.part0 + t;
        const int tile0 = (t / ntx) * h, c = (t % ntx) * REG_GW - 1 + lane;
        // (h is 4, 8, .. 64.  The wide form's own expressions: through the shared functions
        // a batch of 16 x 1024^2 took 24.0 instead of 20.3 ms of it, at the same registers)
        int r0 = tile0, rLast = min(tile0 + h - 1, n - 1);
        if constexpr (FEW) {
            const GradRows g = grad_rows(tile0, h, n, threadIdx.x >> 5, GRAD_WARPS);
            r0 = g.r0;
            rLast = g.rLast;
        }
        const bool colIn = c >= 0 && c < n;
        const bool own = colIn && lane >= 1 && lane <= REG_GW;
        const bool cEdge = (c == 0 || c == n - 1);
        const float cx6 = cEdge ? 2.f : 4.f;  // 6 M1 on the diagonal
        const float wx = cEdge ? 0.5f : 1.f, iwx = cEdge ? 2.f : 1.f;
        const float tau = s.tau_acc;
        // the stencils run on the integer weights 6 M1 and 6 K1 (36 M~, 6 K); their
        // scale is in the operator's coefficients, each rounded once by the control
        // kernel: 1 / sigma, NCC / sigma^2 / 36, NCC / sigma^2 T_bar.  They and the
        // record pointers are read from the descriptor (one line, in L1) in every row:
        // kept in registers they had the row's own values spilled (48 bytes a row and
        // 67 us per launch of a 33 x 1024^2 scan, now 8 bytes and 57 us)
        // rows r-2 (suffix A) and r-1 (suffix M) of this column; row r is read
        // in the iteration and row r-1 is completed by it
        float tA = 0.f, tM = 0.f, kxAx = 0.f, kxAy = 0.f, kxMx = 0.f, kxMy = 0.f;
        float dyMx = 0.f, dyMy = 0.f, gxM = 0.f, gyM = 0.f, mrM = 0.f;
        float4 uM = make_float4(0.f, 0.f, 0.f, 0.f);
        float slope = 0.f, qud = 0.f;
        // the record and M~R~ of the next row are loaded while a row is worked on
        float4 nu = make_float4(0.f, 0.f, 0.f, 0.f);
        float2 nd = make_float2(0.f, 0.f);
        float nmr = 0.f;
        if (colIn && (FEW ? grad_loads_first(r0, n) : r0 - 1 >= 0)) {
            const int idx = (r0 - 1) * pitch + c;
            const float4 *rec = reinterpret_cast<const float4 *>(s.Vs + idx);
            nu = rec[0];
            nd = *reinterpret_cast<const float2 *>(rec + 1);
            nmr = s.MR[idx];
        }
        for (int r = r0 - 1; r <= rLast + 1; r++) {
            const bool in = colIn && r >= 0 && r < n;
            float4 u = nu;
            const float2 dp = make_float2(nd.x, nd.y);
            const float mr = nmr;
            if (colIn && r + 1 < n && r + 1 <= rLast + 1) {
                const int idx = (r + 1) * pitch + c;
                const float4 *rec = reinterpret_cast<const float4 *>(s.Vs + idx);
                nu = rec[0];
                nd = *reinterpret_cast<const float2 *>(rec + 1);
                nmr = s.MR[idx];
            }
            float tv = 0.f, gx = 0.f, gy = 0.f;
            if (in) {
                if (tau != 0.f) u = df_add2(u, tau * dp.x, tau * dp.y);
                tv = sample_df<BF16, true>(s.T, n, pitch, c, r, u, &gx, &gy);
            } else {
                u = make_float4(0.f, 0.f, 0.f, 0.f);
            }
            // u(r, c+1) - u(r, c) and u(r, c) - u(r-1, c), each from the hi and
            // lo parts (the stiffness terms are small differences of values of
            // several grid units); 0 where a node is missing
            float4 uR;
            uR.x = __shfl_down_sync(FULL, u.x, 1);
            uR.y = __shfl_down_sync(FULL, u.y, 1);
            uR.z = __shfl_down_sync(FULL, u.z, 1);
            uR.w = __shfl_down_sync(FULL, u.w, 1);
            const bool hasR = in && c + 1 < n, hasU = in && r >= 1 && r >= r0;
            const float dxx = hasR ? (uR.x - u.x) + (uR.z - u.z) : 0.f;
            const float dxy = hasR ? (uR.y - u.y) + (uR.w - u.w) : 0.f;
            const float dyx = hasU ? (u.x - uM.x) + (u.z - uM.z) : 0.f;
            const float dyy = hasU ? (u.y - uM.y) + (u.w - uM.w) : 0.f;
            // K1 along the row: [u(c) - u(c-1)] - [u(c+1) - u(c)]
            const float kxx = __shfl_up_sync(FULL, dxx, 1) - dxx;
            const float kxy = __shfl_up_sync(FULL, dxy, 1) - dxy;
            const int m = r - 1;
            if (m >= r0) {
                const bool mEdge = (m == 0 || m == n - 1);
                const float cy6 = mEdge ? 2.f : 4.f;
                // 36 M~ That at (m, c): 6 M1 down the column, then along the row
                const float vt = (tA + tv) + cy6 * tM;
                const float mt36 = (__shfl_up_sync(FULL, vt, 1) + __shfl_down_sync(FULL, vt, 1)) + cx6 * vt;
                // K1 along the column at m: [u(m) - u(m-1)] - [u(m+1) - u(m)]
                const float kyx = dyMx - dyx, kyy = dyMy - dyy;
                const float KYx = (__shfl_up_sync(FULL, kyx, 1) + __shfl_down_sync(FULL, kyx, 1)) + cx6 * kyx;
                const float KYy = (__shfl_up_sync(FULL, kyy, 1) + __shfl_down_sync(FULL, kyy, 1)) + cx6 * kyy;
                if (own) {
                    // 6 (K u)
                    const float kux = (kxAx + kxx) + cy6 * kxMx + KYx;
                    const float kuy = (kxAy + kxy) + cy6 * kxMy + KYy;
                    const float om = wx * (mEdge ? 0.5f : 1.f), iom = iwx * (mEdge ? 2.f : 1.f);
                    // dNCC/dThat / h^2 = (M~R~) / sigma - NCC (M~That - T_bar omega) / sigma^2
                    const float A = mrM * s.isig - s.c36 * mt36 + s.cT * om;
                    const float psx = -A * gxM + b.lam6 * kux, psy = -A * gyM + b.lam6 * kuy;
                    const float sc = s.ih2 * iom;
                    const float dnx = -psx * sc, dny = -psy * sc;
                    const int idx = m * pitch + c;
                    float4 *rec = reinterpret_cast<float4 *>(s.Vc + idx);
                    rec[0] = uM;
                    rec[1] = make_float4(dnx, dny, mt36, mrM);
                    if constexpr (FEW) {
                        rows[m - tile0][lane] = make_float2(psx * psx + psy * psy, dnx * kux + dny * kuy);
                    } else {
                        slope -= (psx * psx + psy * psy) * iom;
                        qud += dnx * kux + dny * kuy;
                    }
                }
            }
            tA = tM; tM = tv;
            kxAx = kxMx; kxAy = kxMy; kxMx = kxx; kxMy = kxy;
            dyMx = dyx; dyMy = dyy;
            gxM = gx; gyM = gy; mrM = mr; uM = u;
        }
        if constexpr (FEW) {
            __syncthreads();
            if (threadIdx.x < 32 && own) {
                const int end = min(tile0 + h, n);
#pragma unroll 4
                for (int m = tile0; m < end; m++) {
                    const float iom = iwx * ((m == 0 || m == n - 1) ? 2.f : 1.f);
                    const float2 q = rows[m - tile0][lane];
                    slope -= q.x * iom;
                    qud += q.y;
                }
            }
            __syncthreads();
            if (threadIdx.x >= 32) continue;
        }
        slope = warp_sum(slope);
        qud = warp_sum(qud / 6.f);
        if (lane < PG_STRIDE) b.partG[(int64_t)part * PG_STRIDE + lane] = lane == 0 ? slope : qud;
    }
}

// ---------------------------------------------------------------------------
// S: the H1-type smoother (Section "Gradient flow": d = -A^{-1} E'[phi], A
// selected to smooth).  A = M_s (x) M_s, the tensor-product Gram matrix of
// M_s = M1 + (s^2/2) K1 with s a number of grid spacings; in grid units of
// the level the direction is d = (T (x) T)^{-1} (omega d_L2), T = M_s / h the
// dimensionless tridiagonal matrix (off-diagonal 1/6 - s^2/2, diagonal
// 2/3 + s^2, 1/3 + s^2/2 at the ends) and d_L2 = -psi / (h^2 omega) the lumped
// direction of the gradient pass.  The Kronecker inverse is one tridiagonal
// solve along every row, then one along every column (Thomas elimination
// with the level's precomputed pivots).  The previous iterate's node records
// (not read again before the next gradient pass overwrites them) hold the
// intermediate fields: the row solutions in u.x, u.y, 6 K u in d, the columns'
// elimination in mt, mr.
//
// The sweeps are serial chains of two or three FP32 operations per element.  With
// their loads in the chain (each element read from global memory when its turn
// came) a row took 145 us and a column 192 us at 257^2; here the elements come
// from shared memory, filled ahead by whole-warp copies: 236 -> 42 us for the
// gradient pass and both smoother passes of a step (5 operators of 257^2 and
// coarser levels), 263 -> 63 ms for a 6 x 256^2 scan.
// ---------------------------------------------------------------------------
namespace {

__device__ __forceinline__ float2 *sm_x(NodeRec *V, int64_t idx) { return reinterpret_cast<float2 *>(&V[idx].u); }
__device__ __forceinline__ float2 *sm_y(NodeRec *V, int64_t idx) { return reinterpret_cast<float2 *>(&V[idx].mt); }

constexpr int SM_BATCH = 8;     // elements of a sweep held in registers at a time
constexpr int SM_RING = 32;     // rows of the column sweeps' ring, filled SM_GROUP at a time
constexpr int SM_GROUP = 8;

// Rows per block of the row pass: 16 (one warp sweeps 16 rows x 2 components) up to
// 1025 nodes per side, where they and the pivots take 139 KB of shared memory; fewer
// beyond, 164 KB at 4097.
__host__ __device__ __forceinline__ int smooth_row_chunk(int n) { return n <= 1025 ? 16 : (n <= 2049 ? 8 : 4); }

__device__ __forceinline__ void copy_async8(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src));
}
__device__ __forceinline__ void copy_async16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src));
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;"); }
template <int N>
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N)); }

}  // namespace

// Rows: a block holds smooth_row_chunk(n) rows of one operator in shared memory.
// Warp 0 sweeps them (lane = row and component: with n = 2^l + 1 the 32 lanes hit
// 32 banks) while the other warps form 6 K u of the same rows for the column
// pass (strips of 30 columns and a halo, by the gradient pass's integer
// stencils, hi and lo parts of u differenced separately).
__global__ void __launch_bounds__(256) k_smooth_rows(BatchDev b)
{
    extern __shared__ __align__(16) float2 smem_rows[];
    const unsigned FULL = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int n_ops = b.ctr[0];
    const float a = b.sm_a;
    for (int it = blockIdx.x; it < n_ops * b.rch; it += gridDim.x) {
        const int o = it / b.rch, ch = it % b.rch;
        const StepDesc &s = b.st[o].step;
        if (s.phase != PH_GRAD) continue;
        const int n = s.n, pitch = s.pitch, R = smooth_row_chunk(n), r0 = ch * R;
        if (r0 >= n) continue;
        const int nr = min(R, n - r0);
        const NodeRec *Vc = s.Vc;
        NodeRec *Vs = const_cast<NodeRec *>(s.Vs);
        const float2 *gtab = b.ops[o].lv[b.st[o].lvl].sm_tab;
        float2 *tab = smem_rows, *ys = smem_rows + n;  // ys[row n + c]
        for (int c = tid; c < n; c += 256) tab[c] = gtab[c];
        for (int q = wid; q < nr; q += 8) {
            const int r = r0 + q;
            const float omr = (r == 0 || r == n - 1) ? 0.5f : 1.f;
            const NodeRec *row = Vc + (int64_t)r * pitch;
#pragma unroll 8
            for (int c = lane; c < n; c += 32) {
                const float2 d = row[c].d;
                const float om = omr * ((c == 0 || c == n - 1) ? 0.5f : 1.f);
                ys[q * n + c] = make_float2(om * d.x, om * d.y);
            }
        }
        __syncthreads();
        if (wid == 0) {
            if ((lane >> 1) < nr) {
                float *p = reinterpret_cast<float *>(ys + (lane >> 1) * n) + (lane & 1);
                float v[SM_BATCH], m[SM_BATCH], nv[SM_BATCH], nm[SM_BATCH];
                // elimination, then substitution: the next batch is read while a
                // batch is worked on
                float y = 0.f;
#pragma unroll
                for (int k = 0; k < SM_BATCH; k++) { nv[k] = p[2 * min(k, n - 1)]; nm[k] = tab[min(k, n - 1)].y; }
                for (int c = 0; c < n; c += SM_BATCH) {
#pragma unroll
                    for (int k = 0; k < SM_BATCH; k++) { v[k] = nv[k]; m[k] = nm[k]; }
#pragma unroll
                    for (int k = 0; k < SM_BATCH; k++) {
                        const int cc = min(c + SM_BATCH + k, n - 1);
                        nv[k] = p[2 * cc];
                        nm[k] = tab[cc].y;
                    }
#pragma unroll
                    for (int k = 0; k < SM_BATCH; k++)
                        if (c + k < n) {
                            y = __fsub_rn(v[k], __fmul_rn(a, y)) * m[k];  // (a y rounded first)
                            p[2 * (c + k)] = y;
                        }
                }
                float x = 0.f;
#pragma unroll
                for (int k = 0; k < SM_BATCH; k++) { const int cc = max(n - 1 - k, 0); nv[k] = p[2 * cc]; nm[k] = tab[cc].x; }
                for (int c = n - 1; c >= 0; c -= SM_BATCH) {
#pragma unroll
                    for (int k = 0; k < SM_BATCH; k++) { v[k] = nv[k]; m[k] = nm[k]; }
#pragma unroll
                    for (int k = 0; k < SM_BATCH; k++) {
                        const int cc = max(c - SM_BATCH - k, 0);
                        nv[k] = p[2 * cc];
                        nm[k] = tab[cc].x;
                    }
#pragma unroll
                    for (int k = 0; k < SM_BATCH; k++)
                        if (c - k >= 0) {
                            const float cp = c - k < n - 1 ? m[k] : 0.f;
                            x = v[k] - cp * x;
                            p[2 * (c - k)] = x;
                        }
                }
            }
        } else {
            const int nst = (n + REG_GW - 1) / REG_GW;
            for (int st = wid - 1; st < nst; st += 7) {
                const int c = st * REG_GW - 1 + lane;
                const bool colIn = c >= 0 && c < n, own = colIn && lane >= 1 && lane <= REG_GW;
                const float cx6 = (c == 0 || c == n - 1) ? 2.f : 4.f;
                // rolling rows r+1 (P), r (C), r-1 (N) of u and of K1 along the row
                auto ldu = [&](int r) {
                    return (colIn && r >= 0 && r < n) ? reinterpret_cast<const float4 *>(Vc + (int64_t)r * pitch + c)[0]
                                                      : make_float4(0.f, 0.f, 0.f, 0.f);
                };
                auto kx_of = [&](const float4 &u, int r) {
                    // [u(c) - u(c-1)] - [u(c+1) - u(c)] along the row (0 past the grid)
                    float4 uR;
                    uR.x = __shfl_down_sync(FULL, u.x, 1);
                    uR.y = __shfl_down_sync(FULL, u.y, 1);
                    uR.z = __shfl_down_sync(FULL, u.z, 1);
                    uR.w = __shfl_down_sync(FULL, u.w, 1);
                    const bool rowIn = r >= 0 && r < n, hasR = colIn && rowIn && c + 1 < n;
                    const float dxx = hasR ? (uR.x - u.x) + (uR.z - u.z) : 0.f;
                    const float dxy = hasR ? (uR.y - u.y) + (uR.w - u.w) : 0.f;
                    return make_float2(__shfl_up_sync(FULL, dxx, 1) - dxx, __shfl_up_sync(FULL, dxy, 1) - dxy);
                };
                const int rT = r0 + nr - 1;
                float4 uP = ldu(rT + 1), uC = ldu(rT), uNext = ldu(rT - 1);
                float2 kP = kx_of(uP, rT + 1), kC = kx_of(uC, rT);
                for (int r = rT; r >= r0; r--) {
                    const float4 uN = uNext;
                    if (r > r0) uNext = ldu(r - 2);
                    const float2 kN = kx_of(uN, r - 1);
                    // K1 along the column at (r, c): [u(r) - u(r-1)] - [u(r+1) - u(r)]
                    const bool hasU = colIn && r >= 1, hasD = colIn && r + 1 < n;
                    const float kyx = (hasU ? (uC.x - uN.x) + (uC.z - uN.z) : 0.f) - (hasD ? (uP.x - uC.x) + (uP.z - uC.z) : 0.f);
                    const float kyy = (hasU ? (uC.y - uN.y) + (uC.w - uN.w) : 0.f) - (hasD ? (uP.y - uC.y) + (uP.w - uC.w) : 0.f);
                    const float KYx = (__shfl_up_sync(FULL, kyx, 1) + __shfl_down_sync(FULL, kyx, 1)) + cx6 * kyx;
                    const float KYy = (__shfl_up_sync(FULL, kyy, 1) + __shfl_down_sync(FULL, kyy, 1)) + cx6 * kyy;
                    if (own) {
                        const float cy6 = (r == 0 || r == n - 1) ? 2.f : 4.f;
                        const float kux = (kP.x + kN.x) + cy6 * kC.x + KYx;  // 6 (K u)
                        const float kuy = (kP.y + kN.y) + cy6 * kC.y + KYy;
                        Vs[(int64_t)r * pitch + c].d = make_float2(kux, kuy);
                    }
                    uP = uC; uC = uN;
                    kP = kC; kC = kN;
                }
            }
        }
        __syncthreads();
        for (int q = wid; q < nr; q += 8) {
            const int64_t row = (int64_t)(r0 + q) * pitch;
            for (int c = lane; c < n; c += 32) *sm_x(Vs, row + c) = ys[q * n + c];
        }
        __syncthreads();
    }
}

// Columns: a one-warp block holds REG_GW owned columns (lanes 1 .. REG_GW) and
// walks down for the elimination and up for the substitution, its rows arriving in
// a ring in shared memory; on the way up it writes d into the current records
// and sums the new slope g^T d = -h^4 sum omega d_L2 . d and u^T K d.
__global__ void __launch_bounds__(32) k_smooth_cols(BatchDev b)
{
    // ring rows: 16 B (6 K u, elimination) and 8 B (d_L2) per column; going down
    // the first 8 B per column of the same rows hold the row solutions
    __shared__ float4 ringV[SM_RING][32];
    __shared__ float2 ringD[SM_RING][32];
    extern __shared__ __align__(16) float2 tab_cols[];
    const int lane = threadIdx.x & 31;
    const int n_ops = b.ctr[0];
    const float a = b.sm_a;
    for (int it = blockIdx.x; it < n_ops * b.cch; it += gridDim.x) {
        const int o = it / b.cch, ch = it % b.cch;
        const StepDesc &s = b.st[o].step;
        if (s.phase != PH_GRAD) continue;
        const int n = s.n, pitch = s.pitch;
        if (ch * REG_GW >= n) continue;  // warp-uniform
        const int c = ch * REG_GW - 1 + lane;
        const bool own = c < n && lane >= 1 && lane <= REG_GW;
        NodeRec *Vc = s.Vc + c;
        NodeRec *Vs = const_cast<NodeRec *>(s.Vs) + c;
        const float2 *gtab = b.ops[o].lv[b.st[o].lvl].sm_tab;
        __syncwarp();
        for (int r = lane; r < n; r += 32) tab_cols[r] = gtab[r];
        // down: rows r .. r + SM_GROUP - 1 of the row solutions are one copy group
        float2 *ringX = ringD[0];
        auto fill_down = [&](int r0) {
            if (own)
                for (int k = 0; k < SM_GROUP; k++) {
                    const int r = r0 + k;
                    if (r < n) copy_async8(ringX + (r % SM_RING) * 32 + lane, sm_x(Vs, (int64_t)r * pitch));
                }
            copy_commit();
        };
        for (int k = 0; k < SM_RING - SM_GROUP; k += SM_GROUP) fill_down(k);
        float2 y = make_float2(0.f, 0.f);
        for (int r0 = 0; r0 < n; r0 += SM_GROUP) {
            fill_down(r0 + SM_RING - SM_GROUP);
            copy_wait<SM_RING / SM_GROUP - 1>();
            __syncwarp();
            if (own) {
                float2 x[SM_GROUP];
                float m[SM_GROUP];
#pragma unroll
                for (int k = 0; k < SM_GROUP; k++) {
                    x[k] = ringX[((r0 + k) % SM_RING) * 32 + lane];
                    m[k] = tab_cols[min(r0 + k, n - 1)].y;
                }
#pragma unroll
                for (int k = 0; k < SM_GROUP; k++)
                    if (r0 + k < n) {
                        y.x = (x[k].x - a * y.x) * m[k];
                        y.y = (x[k].y - a * y.y) * m[k];
                        *sm_y(Vs, (int64_t)(r0 + k) * pitch) = y;
                    }
            }
            __syncwarp();  // the group's slots are free for the next fill
        }
        copy_wait<0>();
        __threadfence();  // the copies below read what the stores above wrote
        __syncwarp();
        // up: group g holds rows n-1 - g SM_GROUP .. downwards, slot by distance
        auto fill_up = [&](int q0) {
            if (own)
                for (int k = 0; k < SM_GROUP; k++) {
                    const int r = n - 1 - (q0 + k);
                    if (r >= 0) {
                        copy_async16(&ringV[(q0 + k) % SM_RING][lane], &Vs[(int64_t)r * pitch].d);
                        copy_async8(&ringD[(q0 + k) % SM_RING][lane], &Vc[(int64_t)r * pitch].d);
                    }
                }
            copy_commit();
        };
        for (int k = 0; k < SM_RING - SM_GROUP; k += SM_GROUP) fill_up(k);
        const float omc = (c == 0 || c == n - 1) ? 0.5f : 1.f;
        float2 dnext = make_float2(0.f, 0.f);
        float sl = 0.f, qd = 0.f;
        for (int q0 = 0; q0 < n; q0 += SM_GROUP) {
            fill_up(q0 + SM_RING - SM_GROUP);
            copy_wait<SM_RING / SM_GROUP - 1>();
            __syncwarp();
            if (own) {
#pragma unroll
                for (int k = 0; k < SM_GROUP; k++) {
                    const int r = n - 1 - (q0 + k);
                    if (r >= 0) {
                        const float4 v = ringV[(q0 + k) % SM_RING][lane];  // 6 K u, elimination
                        const float2 dl = ringD[(q0 + k) % SM_RING][lane];
                        const float cp = r < n - 1 ? tab_cols[r].x : 0.f;
                        float2 dn;
                        dn.x = v.z - cp * dnext.x;
                        dn.y = v.w - cp * dnext.y;
                        dnext = dn;
                        const float om = omc * ((r == 0 || r == n - 1) ? 0.5f : 1.f);
                        sl += om * (dl.x * dn.x + dl.y * dn.y);
                        qd += dn.x * v.x + dn.y * v.y;
                        Vc[(int64_t)r * pitch].d = dn;
                    }
                }
            }
            __syncwarp();
        }
        copy_wait<0>();
        sl = warp_sum(sl);
        qd = warp_sum(qd / 6.f);
        if (lane == 0) {
            b.partS[((int64_t)o * b.cch + ch) * 2] = sl;
            b.partS[((int64_t)o * b.cch + ch) * 2 + 1] = qd;
        }
    }
}

// Row chunks per operator, and the dynamic shared memory of the two passes, for
// levels of up to n nodes per side.
int smooth_row_chunks(int n) { return (n + smooth_row_chunk(n) - 1) / smooth_row_chunk(n); }
static size_t smooth_rows_smem(int n) { return sizeof(float2) * (size_t)n * (smooth_row_chunk(n) + 1); }

// Room for the largest side (per device; cheap enough to repeat per handle).
int smooth_prepare()
{
    return cudaFuncSetAttribute(k_smooth_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smooth_rows_smem(4097)) ==
                       cudaSuccess &&
                   cudaFuncSetAttribute(k_smooth_cols, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)(sizeof(float2) * 4097)) == cudaSuccess
               ? 0
               : 1;
}

// n: nodes per side of the handle's finest level; ops: operators of the widest
// batch.
void launch_smooth(int nsm, int ops, int n, cudaStream_t st, const BatchDev &b)
{
    const int rows = std::min((int64_t)ops * b.rch, (int64_t)2 * nsm), cols = std::min((int64_t)ops * b.cch, (int64_t)8 * nsm);
    k_smooth_rows<<<rows, 256, smooth_rows_smem(n), st>>>(b);
    k_smooth_cols<<<cols, 32, sizeof(float2) * (size_t)n, st>>>(b);
}

// Bilinear sampling helpers of the trial pass.
namespace {

struct Texel4 {
    int jx, jy;
    float ax, ay;
    bool clx, cly;
    float t00, t01, t10, t11;
};

__device__ __forceinline__ void locate(int n, int c, int r, float vx, float vy, int &jx, int &jy, float &ax,
                                       float &ay, bool &clx, bool &cly)
{
    float fx, fy;
    jx = c + floor_i(vx, fx);
    jy = r + floor_i(vy, fy);
    ax = vx - fx;
    ay = vy - fy;
    clx = cly = false;
    if (jx < 0) { jx = 0; ax = 0.f; clx = true; }
    else if (jx >= n - 1) { clx = (jx > n - 1) || (ax > 0.f); jx = n - 2; ax = 1.f; }
    if (jy < 0) { jy = 0; ay = 0.f; cly = true; }
    else if (jy >= n - 1) { cly = (jy > n - 1) || (ay > 0.f); jy = n - 2; ay = 1.f; }
}

template <bool BF16>
__device__ __forceinline__ void fetch(Texel4 &q, const void *img, int pitch)
{
    int i0 = q.jy * pitch + q.jx;
    q.t00 = ldimg<BF16>(img, i0);
    q.t01 = ldimg<BF16>(img, i0 + 1);
    q.t10 = ldimg<BF16>(img, i0 + pitch);
    q.t11 = ldimg<BF16>(img, i0 + pitch + 1);
}

__device__ __forceinline__ float bil(const Texel4 &q)
{
    return (1.f - q.ay) * ((1.f - q.ax) * q.t00 + q.ax * q.t01) + q.ay * ((1.f - q.ax) * q.t10 + q.ax * q.t11);
}

}  // namespace

// ---------------------------------------------------------------------------
// T: warp + energy as FE sums over a strip tile of 31 x 32 cells.
// Level-start pass (tau = 0), at u:
//   [0] int That / h^2 = sum omega_i That_i      [1] int That^2 / h^2 = That^T M~ That
//   [2] int That R~ / h^2 = sum (M~ R~)_i That_i   [3 MAXT] Quu, the Dirichlet form of u
// Trial pass: for every step size tau_j the change against the current u,
// delta_j = That(u + tau_j d) - That(u) per node:
//   [3j] sum omega delta   [3j+1] 2 sum (M~ That) delta + delta^T M~ delta
//   [3j+2] sum (M~ R~) delta
// and in the first pass of a search [3 MAXT + 2] Qdd, the Dirichlet form of d
// (the Dirichlet form of u + tau d is Quu + 2 tau Qud + tau^2 Qdd).
// When u and u + tau d lie in the same bilinear cell, delta is formed from the
// cell's four texels as
//   tau d_x [(1-a_y') (t01-t00) + a_y' (t11-t10)] + tau d_y [(1-a_x) (t10-t00) + a_x (t11-t01)],
// so that its float rounding is relative to delta itself (the quantity the
// Armijo test compares), not to That; a tiny move across a cell line is split
// into exact segments, and a move of 2^-10 grid units or more takes a fresh
// sample.
// Sums over nodes use per-node weights (omega and the stored M~ That, M~ R~);
// the quadratic forms are summed per cell.  With the cyclic corner order the
// element mass matrix is (1/36) [4 2 1 2; 2 4 2 1; 1 2 4 2; 2 1 2 4], and
//   36 v^T M~_e v = 4 P(top) + 4 P(bottom) + 2 top . [2 1; 1 2] bottom,
//   P(x0, x1) = x0 (x0 + x1) + x1^2,
// so each row's P is formed once for the two cells that share the row.  The
// cell's Dirichlet form is (P(p, q) + P(r, s)) / 3 per component, p, q the x
// differences of its top and bottom rows and r, s the y differences of its
// left and right columns.  Lane l holds node column c0 + l; lanes 0..30 own
// the cells to their right, lane 31 supplies the right corners.
// ---------------------------------------------------------------------------
namespace {

__device__ __forceinline__ float pform(float x0, float x1) { return x0 * (x0 + x1) + x1 * x1; }

struct StripGeom {
    int n, pitch, h, r0, rEnd, c;
    bool colIn, cellCol, nodeCol;
    float wx;
};

__device__ __forceinline__ StripGeom strip_geom(const StepDesc &Lv, int t, int lane)
{
    StripGeom g;
    g.n = Lv.n;
    g.pitch = Lv.pitch;
    const int ntx = (g.n - 1 + REG_CW - 1) / REG_CW;
    g.h = Lv.ht;
    g.r0 = (t / ntx) * g.h;
    g.c = (t % ntx) * REG_CW + lane;
    g.rEnd = min(g.r0 + g.h, g.n - 1);
    g.colIn = g.c < g.n;
    g.cellCol = lane < REG_CW && g.c < g.n - 1;
    g.nodeCol = g.colIn && (lane < REG_CW || g.c == g.n - 1);
    g.wx = (g.c == 0 || g.c == g.n - 1) ? 0.5f : 1.f;
    return g;
}

// The 3 x 3 texel patch around the base cell of a node, extended towards the
// direction of its move, and the per-node terms of the exact change of the
// interpolant for moves of less than one cell (patch_delta).
struct Patch {
    float ax, ay;    // fractions of the base point in its cell (clamped coordinates: 0 or 1)
    float lx, ly;    // signed distance to the next cell line in the move direction
    float s0x, s1x;  // slope along x at a_y of the base cell and of its neighbour in the move direction
    float v0[3], v1[3];  // t(row + 1) - t(row) in the base row band and in the neighbour band,
                         // columns: base left, base right, neighbour outer
    bool nbx, nby;   // the neighbour cell exists (else the interpolant is flat beyond the border)
    bool posx, posy; // move direction
    int clx, cly;    // 0: inside; otherwise the raw cell index of the clamped base point (never 0)
    float rax, ray;  // raw fraction of a clamped base point
    float t0;        // the interpolant at the base point
};

template <bool BF16>
__device__ __forceinline__ void make_patch(Patch &P, const void *T, int n, int pitch, int c, int r, float4 u, float dx,
                                           float dy)
{
    int ix, iy;
    float fx, fy;
    df_split(u.x, u.z, ix, fx);
    df_split(u.y, u.w, iy, fy);
    int jx = c + ix, jy = r + iy;
    P.rax = fx;
    P.ray = fy;
    P.clx = P.cly = 0;
    float ax = fx, ay = fy;
    if (jx < 0) { P.clx = jx; jx = 0; ax = 0.f; }
    else if (jx >= n - 1) { if (jx > n - 1 || fx > 0.f) P.clx = jx; jx = n - 2; ax = 1.f; }
    if (jy < 0) { P.cly = jy; jy = 0; ay = 0.f; }
    else if (jy >= n - 1) { if (jy > n - 1 || fy > 0.f) P.cly = jy; jy = n - 2; ay = 1.f; }
    P.ax = ax;
    P.ay = ay;
    P.posx = dx >= 0.f;
    P.posy = dy >= 0.f;
    P.nbx = P.posx ? (jx + 1 <= n - 2) : (jx >= 1);
    P.nby = P.posy ? (jy + 1 <= n - 2) : (jy >= 1);
    const int cx2 = P.posx ? min(jx + 2, n - 1) : max(jx - 1, 0);
    const int ry2 = P.posy ? min(jy + 2, n - 1) : max(jy - 1, 0);
    const int rows[3] = {jy, jy + 1, ry2}, cols[3] = {jx, jx + 1, cx2};
    float t[3][3];
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
        for (int b = 0; b < 3; b++) t[a][b] = ldimg<BF16>(T, rows[a] * pitch + cols[b]);
    P.t0 = (1.f - ay) * ((1.f - ax) * t[0][0] + ax * t[0][1]) + ay * ((1.f - ax) * t[1][0] + ax * t[1][1]);
    P.lx = P.posx ? 1.f - ax : -ax;
    P.ly = P.posy ? 1.f - ay : -ay;
    P.s0x = (1.f - ay) * (t[0][1] - t[0][0]) + ay * (t[1][1] - t[1][0]);
    // neighbour cell along x: columns (1, 2) when moving right, (2, 0) when moving left
    const float nl0 = P.posx ? t[0][1] : t[0][2], nr0 = P.posx ? t[0][2] : t[0][0];
    const float nl1 = P.posx ? t[1][1] : t[1][2], nr1 = P.posx ? t[1][2] : t[1][0];
    P.s1x = P.nbx ? (1.f - ay) * (nr0 - nl0) + ay * (nr1 - nl1) : 0.f;
#pragma unroll
    for (int b = 0; b < 3; b++) {
        P.v0[b] = t[1][b] - t[0][b];
        P.v1[b] = P.posy ? t[2][b] - t[1][b] : t[0][b] - t[2][b];
    }
}

// Change of the interpolant for the move (ex, ey) from the base point of P,
// split into a move along x in the base row band and a move along y at the new
// column; each part is a sum of segment lengths times the slope of the cell
// the segment lies in, so that its rounding is relative to the change itself
// (a single float fraction could not resolve a move far below its ulp across a
// cell line).  Past the grid border the interpolant is flat; a base point
// outside the grid contributes only the part of the move back inside.
// Returns false (and no value) for a move of a cell or more.
__device__ __forceinline__ bool patch_delta(const Patch &P, int n, float ex, float ey, float &del)
{
    bool ok = true;
    // x part
    float xpart, f;
    bool nbcol = false;  // the y part runs in the neighbour column cell
    if (P.clx) {
        ok = fabsf(ex) < 1.f;
        // length of the move inside the grid: from the left border (raw cell
        // -1) or back from the right border (raw cell n-1); 0 further out
        const float in = (P.clx == -1) ? fmaxf(P.rax + ex - 1.f, 0.f)
                                        : ((P.clx == n - 1) ? fminf(P.rax + ex, 0.f) : 0.f);
        xpart = in * P.s0x;
        f = P.ax + in;
    } else {
        const float ax1 = P.ax + ex;
        if (ax1 >= 0.f && ax1 < 1.f) {
            xpart = ex * P.s0x;
            f = ax1;
        } else {
            const float rest = ex - P.lx;  // length beyond the cell line
            ok = fabsf(rest) < 1.f;
            xpart = P.lx * P.s0x + rest * P.s1x;
            f = P.nbx ? (P.posx ? rest : 1.f + rest) : (P.posx ? 1.f : 0.f);
            nbcol = P.nbx;
        }
    }
    // y part at the new column: slopes of the base and neighbour row bands
    const float vl0 = nbcol ? (P.posx ? P.v0[1] : P.v0[2]) : P.v0[0];
    const float vr0 = nbcol ? (P.posx ? P.v0[2] : P.v0[0]) : P.v0[1];
    const float sy0 = (1.f - f) * vl0 + f * vr0;
    float ypart;
    if (P.cly) {
        ok = ok && fabsf(ey) < 1.f;
        const float in = (P.cly == -1) ? fmaxf(P.ray + ey - 1.f, 0.f)
                                        : ((P.cly == n - 1) ? fminf(P.ray + ey, 0.f) : 0.f);
        ypart = in * sy0;
    } else {
        const float ay1 = P.ay + ey;
        if (ay1 >= 0.f && ay1 < 1.f) {
            ypart = ey * sy0;
        } else {
            const float rest = ey - P.ly;
            ok = ok && fabsf(rest) < 1.f;
            const float vl1 = nbcol ? (P.posx ? P.v1[1] : P.v1[2]) : P.v1[0];
            const float vr1 = nbcol ? (P.posx ? P.v1[2] : P.v1[0]) : P.v1[1];
            const float sy1 = P.nby ? (1.f - f) * vl1 + f * vr1 : 0.f;
            ypart = P.ly * sy0 + rest * sy1;
        }
    }
    del = xpart + ypart;
    return ok;
}

// Shared memory of one block of the trial pass (one tile).
constexpr int TRIAL_WARPS = REG_STRIP_THREADS / 32;
constexpr int TRIAL_BLOCKS = 7;   // resident blocks per SM
constexpr int TWR = REG_TRIAL_ROWS;  // most cell rows of a tile
template <int JM>
struct TrialTile {
    // per node: A, B, 36 M~That, M~R~ of a node whose moves stay in its cell, else its
    // changes delta_j (four step sizes per plane)
    float4 node[(JM + 3) / 4][TWR + 1][32];
    float qt[TWR + 1][32];                 // Dirichlet form of d over the cells above a row
    unsigned slow[TWR + 1];                // nodes on the exact path, per row
    unsigned short qn[(TWR + 1) * 32];     // queued nodes: row << 5 | lane, in row order
    unsigned short qc[TWR * 32];           // cells with such a corner (between rows row - 1 and row)
    float mom[9][32];                      // per-lane moments
    double start[TRIAL_WARPS][4];          // level-start pass: the warps' sums
};

// The order of the exact sums.  A lane adds the exact changes of every 32nd queued
// node and cell of a window of rows; a window ends after TW rows, or when more than
// TQ - 32 nodes (with those of the row above it) or TC - 32 cells are queued.  (The
// windows are those of a pass that walks the rows with queues of TQ and TC entries;
// keeping its order of additions keeps every sum, and through the gradient's
// coefficients every iterate, bit for bit what it was.)
constexpr int TW = 12, TQ = 96, TC = 192;

// A sum of floats held without rounding beyond 2^-72 of it, as three floats: the
// FP64 pipe of this chip takes 16 cycles of an SM for a warp's addition and as
// many for the conversion, which made the level-start pass of 16 x 1025^2 nodes
// 720 us long; two exact FP32 additions take less than one cycle each.
struct Sum3 {
    float a = 0.f, b = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float x)
    {
        float e, e2;
        two_sum(a, x, a, e);
        two_sum(b, e, b, e2);
        c += e2;
    }
    __device__ __forceinline__ double value() const { return (double)a + ((double)b + (double)c); }
};

// Level-start sums of node rows ra .. rb-1 of one strip tile at u (and the cells
// between them; rows ra > r0 of a tile take the row above for their cells), at
// least in double precision: they seed every search of the level (the trial passes
// only add changes to them), and the pass runs once per level.  After a level
// change (PH_PROLONG) the pass forms u itself from the coarser level's records
// and stores the nodes it owns: the prolongation is needed here only, once per
// level and operator, and as a kernel of its own it cost every step an (almost
// always empty) launch of 3 us.
template <bool BF16>
__device__ __forceinline__ void start_rows(const StepDesc &s, const StripGeom &g, int ra, int rb, double *v)
{
    const unsigned FULL = 0xffffffffu;
    const bool prol = s.phase == PH_PROLONG;
    NodeRec *V = s.Vc;
    const NodeRec *VC = s.VC;
    const float ptau = s.tau_acc;
    Sum3 s1, s3, q2, quu;
    float tP = 0.f, tPR = 0.f, pux = 0.f, puy = 0.f;
    float4 uP = make_float4(0.f, 0.f, 0.f, 0.f);
    const int first = ra > g.r0 ? ra - 1 : ra;  // the row above the first one, for the cells between
    for (int r = first; r < rb; r++) {
        float4 u = make_float4(0.f, 0.f, 0.f, 0.f);
        float t0 = 0.f, mr = 0.f;
        const bool own = g.nodeCol && r >= ra && (r < g.r0 + g.h || r == g.n - 1);
        if (g.colIn) {
            const int64_t idx = (int64_t)r * g.pitch + g.c;
            if (prol) {
                u = prolong_node(VC, s.cpitch, ptau, r, g.c);
                if (own) V[idx].u = u;
            } else {
                u = V[idx].u;
            }
            mr = s.MR[idx];
            t0 = sample_df<BF16, false>(s.T, g.n, g.pitch, g.c, r, u, nullptr, nullptr);
        }
        if (own) {
            const float w = g.wx * ((r == 0 || r == g.n - 1) ? 0.5f : 1.f);
            s1.add(w * t0);
            s3.add(mr * t0);
        }
        const float tR = __shfl_down_sync(FULL, t0, 1);
        float4 uR;
        uR.x = __shfl_down_sync(FULL, u.x, 1);
        uR.y = __shfl_down_sync(FULL, u.y, 1);
        uR.z = __shfl_down_sync(FULL, u.z, 1);
        uR.w = __shfl_down_sync(FULL, u.w, 1);
        const float qx = (uR.x - u.x) + (uR.z - u.z), qy = (uR.y - u.y) + (uR.w - u.w);
        const float rx = (u.x - uP.x) + (u.z - uP.z), ry = (u.y - uP.y) + (u.w - uP.w);
        const float sx = __shfl_down_sync(FULL, rx, 1), sy = __shfl_down_sync(FULL, ry, 1);
        if (g.cellCol && r > first) {
            // the cell between rows r-1 and r: each row's form twice, the cross terms
            q2.add(2.f * pform(t0, tR));
            q2.add(2.f * pform(tP, tPR));
            q2.add(tP * (2.f * t0 + tR) + tPR * (t0 + 2.f * tR));
            quu.add(pform(pux, qx) + pform(rx, sx) + pform(puy, qy) + pform(ry, sy));
        }
        tP = t0; tPR = tR;
        pux = qx; puy = qy; uP = u;
    }
    v[0] = s1.value();
    v[1] = q2.value() * (1.0 / 18.0);
    v[2] = s3.value();
    v[3] = quu.value() * (1.0 / 3.0);
}

// Exact change of the interpolant at one node for every step size, for a
// node whose largest move leaves its cell (or whose base point lies outside
// the grid): the moves that stay in the cell take the polynomial of the base
// cell, the others the texel patch, or a fresh sample for moves of a cell or
// more (whose rounding, ~1e-7 of That, is small against such a change).
template <bool BF16, int JM>
__device__ __forceinline__ void node_deltas_exact(const void *T, int n, int pitch, const float *tau, int J, int c,
                                                  int r, float4 u, float4 dm, float *delta)
{
    Patch P;
    make_patch<BF16>(P, T, n, pitch, c, r, u, dm.x, dm.y);
    const bool cl = P.clx || P.cly;
    // dThat/dx at a_y, dThat/dy at a_x and the mixed derivative of the base cell
    const float sy = P.v0[0] + P.ax * (P.v0[1] - P.v0[0]);
    const float A = dm.x * P.s0x + dm.y * sy;
    const float B = dm.x * dm.y * (P.v0[1] - P.v0[0]);
#pragma unroll
    for (int j = 0; j < JM; j++) {
        delta[j] = 0.f;
        if (j < J) {
            const float ex = tau[j] * dm.x, ey = tau[j] * dm.y;
            const float ax1 = P.ax + ex, ay1 = P.ay + ey;
            float del;
            if (!cl && ax1 >= 0.f && ax1 < 1.f && ay1 >= 0.f && ay1 < 1.f) {
                del = tau[j] * (A + tau[j] * B);
            } else if (!patch_delta(P, n, ex, ey, del)) {
                Texel4 t;
                locate(n, c, r, (u.x + u.z) + ex, (u.y + u.w) + ey, t.jx, t.jy, t.ax, t.ay, t.clx, t.cly);
                fetch<BF16>(t, T, pitch);
                del = bil(t) - P.t0;
            }
            delta[j] = del;
        }
    }
}

// pform and the rest of a cell's form (below) for two values at a time, rounded as the
// scalar expressions are.
__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 pform2(float2 x0, float2 x1)
{
    return __ffma2_rn(x1, x1, __fmul2_rn(x0, __fadd2_rn(x0, x1)));
}
// 2 (P(top) + P(bottom)) + top . [2 1; 1 2] bottom, the rows' forms given
__device__ __forceinline__ float2 cell2(float2 pt, float2 pb, float2 tl, float2 tr, float2 bl, float2 br)
{
    const float2 two = f2(2.f, 2.f);
    return __ffma2_rn(tr, __ffma2_rn(two, br, bl),
                      __ffma2_rn(tl, __ffma2_rn(two, bl, br), __fmul2_rn(two, __fadd2_rn(pt, pb))));
}

// Row counts of the exact path's queues, one row per lane (row 32 apart): the mask
// of the row's nodes, and inclusive prefixes of the queued nodes and cells.
struct RowQueues {
    unsigned s, cells;   // nodes on the exact path; mixed cells between this row and the one above
    int pn, pc;          // inclusive prefixes over rows 0 .. lane
    unsigned s32, cells32;
    int tn, tc;          // totals
};

template <int JM>
__device__ __forceinline__ RowQueues row_queues(const TrialTile<JM> &sh, int nr, unsigned cellmask, int lane)
{
    RowQueues q;
    q.s = lane < nr ? sh.slow[lane] : 0u;
    const unsigned up = __shfl_up_sync(0xffffffffu, q.s, 1);
    // a cell's corners: columns l and l + 1 of both rows
    q.cells = lane > 0 && lane < nr ? (up | up >> 1 | q.s | q.s >> 1) & cellmask : 0u;
    q.pn = __popc(q.s);
    q.pc = __popc(q.cells);
#pragma unroll
    for (int k = 1; k < 32; k <<= 1) {
        const int a = __shfl_up_sync(0xffffffffu, q.pn, k), b = __shfl_up_sync(0xffffffffu, q.pc, k);
        if (lane >= k) { q.pn += a; q.pc += b; }
    }
    const unsigned s31 = __shfl_sync(0xffffffffu, q.s, 31);
    q.s32 = nr > 32 ? sh.slow[32] : 0u;
    q.cells32 = nr > 32 ? (s31 | s31 >> 1 | q.s32 | q.s32 >> 1) & cellmask : 0u;
    q.tn = __shfl_sync(0xffffffffu, q.pn, 31) + __popc(q.s32);
    q.tc = __shfl_sync(0xffffffffu, q.pc, 31) + __popc(q.cells32);
    return q;
}

// Trial sums of one strip tile for the step sizes tau_0..tau_{J-1}, by one block.
// All step sizes move a node along the same ray u + tau d, and while the moved
// point stays in the base cell the change of the bilinear interpolant is exactly
//   delta(tau) = tau A + tau^2 B,  A = d . grad That (at the base point),
//   B = d_x d_y (t00 - t01 - t10 + t11),
// so the sums over such nodes are polynomials in tau of per-node moments (sum omega
// A, sum omega B, ...) and of per-cell ones (18 A^T M~ A, 18 A^T M~ B, 18 B^T M~ B),
// gathered once for all step sizes.  A node whose largest move leaves the cell, and
// every cell touching one, is summed exactly for each step size.  Phases, the tile's
// nodes in shared memory between them:
//   1. every warp walks some rows without a branch, a row's texel loads and the next
//      row's records in flight together: A, B, and which nodes take the exact path;
//   2. lists of those nodes and of the cells that touch one;
//   3. exact changes, one node per thread; beside them the moments, one kind per
//      warp, each down the rows;
//   4. per two step sizes (one warp) the exact nodes and cells.
// One warp per tile doing all of this row by row held 128 registers (16 warps on an
// SM) and waited for the record -> template gather of every row: per launch of a 33 x
// 1024^2 scan 122 -> 104 us, of a 21 x 512^2 one 37 -> 23, of a single 1024^2 operator
// 24 -> 15, of 7 operators of 64^2 12.6 -> 8.  It pays where tiles are few: with the 200
// operators of a 400 x 1024^2 scan's batches a launch is bound by its instructions and
// takes what it took (0.96 ms, 0.95 before, the prolongation now among it).  Seven blocks per SM at one row in flight
// (72 registers) beat six (80) at one or two rows, 104 against 112 and 109 us.
template <bool BF16, int JM>
__device__ __forceinline__ void trial_tile(const BatchDev &b, const StepDesc &s, const StripGeom &g, TrialTile<JM> &sh,
                                           int part, int wid, int lane)
{
    const unsigned FULL = 0xffffffffu;
    const unsigned lt = (1u << lane) - 1u;
    const int J = min(s.ntr, JM), n = g.n, pitch = g.pitch;
    const bool withQ = (s.phase == PH_GRAD);
    const float4 *V = reinterpret_cast<const float4 *>(s.Vc);
    const void *T = s.T;
    // node rows r0 .. r0 + nr - 1, this warp's i0 .. i1 - 1
    const int w0 = g.r0, cells = g.rEnd - w0, nr = cells + 1;
    const int rw = (cells + TRIAL_WARPS - 1) / TRIAL_WARPS;
    const int i0 = min(wid * rw, nr), i1 = wid == TRIAL_WARPS - 1 ? nr : min(i0 + rw, nr);
    {
        float tmax = 0.f;
#pragma unroll
        for (int j = 0; j < JM; j++) tmax = fmaxf(tmax, j < J ? s.tau[j] : 0.f);
        // lanes past the grid work on its last column and count nothing
        const int cc = min(g.c, n - 1);
        const float4 *Vcol = V + 2 * cc;  // (a level's records: below 2^27 words)
        float dPx = 0.f, dPy = 0.f, pdx = 0.f, pdy = 0.f;
        if (withQ && i0 > 0 && i0 < i1) {
            const float4 dm = Vcol[2 * (w0 + i0 - 1) * pitch + 1];
            dPx = dm.x;
            dPy = dm.y;
            pdx = __shfl_down_sync(FULL, dPx, 1) - dPx;
            pdy = __shfl_down_sync(FULL, dPy, 1) - dPy;
        }
        float4 nu = Vcol[2 * (w0 + min(i0, cells)) * pitch], nd = Vcol[2 * (w0 + min(i0, cells)) * pitch + 1];
        for (int i = i0; i < i1; i++) {
            const int r = w0 + i;
            const float4 dm = nd;  // d, 36 M~That, M~R~
            Texel4 q;
            int ix, iy;
            df_split(nu.x, nu.z, ix, q.ax);
            df_split(nu.y, nu.w, iy, q.ay);
            const int jx = cc + ix, jy = r + iy;
            // a base point outside the grid, or a largest move that leaves the
            // cell (then every smaller one along the ray stays inside)
            const float ax1 = q.ax + tmax * dm.x, ay1 = q.ay + tmax * dm.y;
            const bool slw = (unsigned)jx > (unsigned)(n - 2) || (unsigned)jy > (unsigned)(n - 2) ||
                             !(ax1 >= 0.f && ax1 < 1.f) || !(ay1 >= 0.f && ay1 < 1.f);
            q.jx = min(max(jx, 0), n - 2);
            q.jy = min(max(jy, 0), n - 2);
            fetch<BF16>(q, T, pitch);
            const int o = 2 * (w0 + min(i + 1, cells)) * pitch;
            nu = Vcol[o];
            nd = Vcol[o + 1];
            const float dtx = q.t01 - q.t00, dtx1 = q.t11 - q.t10;
            const float sx = dtx + q.ay * (dtx1 - dtx);                            // dThat/dx
            const float sy = (q.t10 - q.t00) + q.ax * ((q.t11 - q.t01) - (q.t10 - q.t00));  // dThat/dy
            const float A = dm.x * sx + dm.y * sy;
            const float B = dm.x * dm.y * (dtx1 - dtx);
            const unsigned ms = __ballot_sync(FULL, slw && g.colIn);
            if (lane == 0) sh.slow[i] = ms;
            sh.node[0][i][lane] = make_float4(A, B, dm.z, dm.w);
            if (withQ) {
                // Dirichlet form of d over the cells between rows r-1 and r
                const float dRx = __shfl_down_sync(FULL, dm.x, 1), dRy = __shfl_down_sync(FULL, dm.y, 1);
                const float qx = dRx - dm.x, qy = dRy - dm.y;
                const float rx = dm.x - dPx, ry = dm.y - dPy;
                const float sx = __shfl_down_sync(FULL, rx, 1), sy = __shfl_down_sync(FULL, ry, 1);
                sh.qt[i][lane] = pform(pdx, qx) + pform(rx, sx) + pform(pdy, qy) + pform(ry, sy);
                pdx = qx; pdy = qy; dPx = dm.x; dPy = dm.y;
            }
        }
    }
    __syncthreads();
    // lists, each warp its rows'
    const unsigned cellmask = __ballot_sync(FULL, g.cellCol);
    const RowQueues rq = row_queues(sh, nr, cellmask, lane);
    if (rq.tn > 0)
        for (int i = i0; i < i1; i++) {
            const int src = i & 31;
            const unsigned ms = i < 32 ? __shfl_sync(FULL, rq.s, src) : rq.s32;
            const unsigned mc = i < 32 ? __shfl_sync(FULL, rq.cells, src) : rq.cells32;
            const int en = i < 32 ? __shfl_sync(FULL, rq.pn, src) : rq.tn, ec = i < 32 ? __shfl_sync(FULL, rq.pc, src) : rq.tc;
            if (ms >> lane & 1) sh.qn[en - __popc(ms) + __popc(ms & lt)] = (unsigned short)((i << 5) | lane);
            if (mc >> lane & 1) sh.qc[ec - __popc(mc) + __popc(mc & lt)] = (unsigned short)((i << 5) | lane);
        }
    __syncthreads();
    // exact changes in place of the queued nodes' entries (the moments below skip them)
    if (rq.tn > 0) {
        float tau[JM];
#pragma unroll
        for (int j = 0; j < JM; j++) tau[j] = j < J ? s.tau[j] : 0.f;
        for (int k = wid * 32 + lane; k < rq.tn; k += REG_STRIP_THREADS) {
            const int e = sh.qn[k], i = e >> 5, ln = e & 31;
            const int r = w0 + i, c = g.c - lane + ln;
            const int idx = 2 * (r * pitch + c);
            const float4 u = V[idx], dm = V[idx + 1];
            float del[(JM + 3) / 4 * 4];
#pragma unroll
            for (int j = JM; j < (JM + 3) / 4 * 4; j++) del[j] = 0.f;
            node_deltas_exact<BF16, JM>(T, n, pitch, tau, J, c, r, u, dm, del);
#pragma unroll
            for (int m = 0; m < (JM + 3) / 4; m++)
                sh.node[m][i][ln] = make_float4(del[4 * m], del[4 * m + 1], del[4 * m + 2], del[4 * m + 3]);
        }
    }
    if (wid == 0) {
        // node moments (owned nodes that stay in their cell)
        float mWA = 0.f, mWB = 0.f, mTA = 0.f, mTB = 0.f, mRA = 0.f, mRB = 0.f;
#pragma unroll 4
        for (int i = 0; i < nr; i++) {
            const int r = w0 + i;
            const float4 q = sh.node[0][i][lane];
            const bool own = g.nodeCol && (r < g.r0 + g.h || r == n - 1);
            const float w = g.wx * ((r == 0 || r == n - 1) ? 0.5f : 1.f);
            if (own && !(sh.slow[i] >> lane & 1)) {
                mWA += w * q.x; mWB += w * q.y;
                mTA += q.z * q.x; mTB += q.z * q.y;
                mRA += q.w * q.x; mRB += q.w * q.y;
            }
        }
        sh.mom[0][lane] = mWA; sh.mom[1][lane] = mWB;
        sh.mom[2][lane] = mTA; sh.mom[3][lane] = mTB;
        sh.mom[4][lane] = mRA; sh.mom[5][lane] = mRB;
    } else if (wid == 1) {
        // cell moments of A and of B (cells whose four corners stay in their cells)
        float2 q = f2(0.f, 0.f), Pv = q, ab0 = q, abR0 = q;
        unsigned mP = 0u;
        const int rn = min(lane + 1, 31);
#pragma unroll 4
        for (int i = 0; i < nr; i++) {
            const float2 ab = *reinterpret_cast<const float2 *>(&sh.node[0][i][lane]);
            const float2 abR = *reinterpret_cast<const float2 *>(&sh.node[0][i][rn]);
            const unsigned m = sh.slow[i];
            const float2 P = pform2(ab, abR);
            if (g.cellCol && i > 0 && !((mP | m) >> lane & 3u)) q = __fadd2_rn(q, cell2(Pv, P, ab0, abR0, ab, abR));
            Pv = P;
            ab0 = ab;
            abR0 = abR;
            mP = m;
        }
        sh.mom[6][lane] = q.x;
        sh.mom[8][lane] = q.y;
    } else if (wid == 2) {
        // their mixed moments
        float qab = 0.f, Ap = 0.f, ApR = 0.f, Bp = 0.f, BpR = 0.f, PabP = 0.f;
        unsigned mP = 0u;
        const int rn = min(lane + 1, 31);
#pragma unroll 4
        for (int i = 0; i < nr; i++) {
            const float2 q = *reinterpret_cast<const float2 *>(&sh.node[0][i][lane]);
            const float2 qr = *reinterpret_cast<const float2 *>(&sh.node[0][i][rn]);
            const float A = q.x, B = q.y, AR = qr.x, BR = qr.y;
            const unsigned m = sh.slow[i];
            const float Pab = A * B + AR * BR + 0.5f * (A * BR + AR * B);
            if (g.cellCol && i > 0 && !((mP | m) >> lane & 3u)) {
                const float ha = 2.f * A + AR, haR = A + 2.f * AR, hb = 2.f * B + BR, hbR = B + 2.f * BR;
                qab += 2.f * (PabP + Pab) + 0.5f * (Ap * hb + ApR * hbR + Bp * ha + BpR * haR);
            }
            PabP = Pab;
            Ap = A; ApR = AR; Bp = B; BpR = BR;
            mP = m;
        }
        sh.mom[7][lane] = qab;
    } else {
        float qdd = 0.f;
        if (withQ) {
#pragma unroll 8
            for (int i = 1; i < nr; i++)
                if (g.cellCol) qdd += sh.qt[i][lane];
        }
        const float tot = warp_sum(qdd / 3.f);
        if (lane == 0) {
            b.partT[(int64_t)part * PT_STRIDE + 3 * REG_MAX_TRIALS + 2] = tot;
            if (rq.tn) atomicAdd(&b.work[KW_TEXACT], (unsigned long long)rq.tn);
        }
    }
    __syncthreads();
    // two step sizes per warp: the exact nodes and cells, window by window, then the
    // sums
    for (int j = 2 * wid; j < J; j += 2 * TRIAL_WARPS) {
        const float2 t = f2(s.tau[j], j + 1 < J ? s.tau[j + 1] : 0.f);
        float2 sn0 = f2(0.f, 0.f), sn1 = sn0, sn2 = sn0, sq = sn0;
        // a node's two changes: at word 2 (j / 2 mod 2) of its entry in plane j / 4, or
        // from A and B in the first words of its entry
        const float2 *plane = reinterpret_cast<const float2 *>(&sh.node[0][0][0]);
        const int dofs = (j >> 2) * (TWR + 1) * 64 + ((j >> 1) & 1);
        if (rq.tn > 0) {
            int a = 0, carry = 0, pna = 0, pca = 0;
            for (;;) {
                const bool trig = lane >= a && lane < nr &&
                                  (lane - a == TW - 1 || carry + rq.pn - pna > TQ - 32 || rq.pc - pca > TC - 32 ||
                                   lane == nr - 1);
                const unsigned bt = __ballot_sync(FULL, trig);
                const int e = bt ? __ffs(bt) - 1 : 32;  // the window's last row
                const int pne = e < 32 ? __shfl_sync(FULL, rq.pn, e) : rq.tn;
                const int pce = e < 32 ? __shfl_sync(FULL, rq.pc, e) : rq.tc;
                for (int k = pna + lane; k < pne; k += 32) {
                    const int en = sh.qn[k], i = en >> 5, ln = en & 31;
                    const int r = w0 + i, c = g.c - lane + ln;
                    if ((ln < REG_CW || c == n - 1) && (r < g.r0 + g.h || r == n - 1)) {
                        const float2 zw = reinterpret_cast<const float2 *>(V + 2 * (r * pitch + c) + 1)[1];
                        const float w = ((c == 0 || c == n - 1) ? 0.5f : 1.f) * ((r == 0 || r == n - 1) ? 0.5f : 1.f);
                        const float2 d = plane[2 * en + dofs];
                        sn0 = __ffma2_rn(f2(w, w), d, sn0);
                        sn1 = __ffma2_rn(f2(zw.x, zw.x), d, sn1);
                        sn2 = __ffma2_rn(f2(zw.y, zw.y), d, sn2);
                    }
                }
                for (int k = pca + lane; k < pce; k += 32) {
                    const int en = sh.qc[k], i = en >> 5, ln = en & 31;
                    const unsigned mt = sh.slow[i - 1] >> ln, mb = sh.slow[i] >> ln;
                    auto corner = [&](unsigned slow, int node) {
                        const float2 q = plane[2 * node + ((slow & 1) ? dofs : 0)];
                        const float2 pl = __fmul2_rn(t, __ffma2_rn(t, f2(q.y, q.y), f2(q.x, q.x)));
                        return (slow & 1) ? q : pl;
                    };
                    const float2 tl = corner(mt, en - 32), tr = corner(mt >> 1, en - 31);
                    const float2 bl = corner(mb, en), br = corner(mb >> 1, en + 1);
                    sq = __fadd2_rn(sq, cell2(pform2(tl, tr), pform2(bl, br), tl, tr, bl, br));
                }
                if (e >= nr - 1) break;
                carry = __popc(__shfl_sync(FULL, rq.s, e));
                a = e + 1;
                pna = pne;
                pca = pce;
            }
        }
        const float mWA = sh.mom[0][lane], mWB = sh.mom[1][lane], mTA = sh.mom[2][lane], mTB = sh.mom[3][lane];
        const float mRA = sh.mom[4][lane], mRB = sh.mom[5][lane];
        const float qaa = sh.mom[6][lane], qab = sh.mom[7][lane], qbb = sh.mom[8][lane];
        auto sums = [&](int jj, float t, float sn0, float sn1, float sn2, float sq) {
            const float v0 = t * (mWA + t * mWB) + sn0;
            const float v1 = (t * (mTA + t * mTB) + t * t * (qaa + t * (2.f * qab + t * qbb)) + sn1 +
                              sq) / 18.f;
            const float v2 = t * (mRA + t * mRB) + sn2;
            const float t0 = warp_sum(v0), t1 = warp_sum(v1), t2 = warp_sum(v2);
            if (lane < 3) b.partT[(int64_t)part * PT_STRIDE + 3 * jj + lane] = lane == 0 ? t0 : (lane == 1 ? t1 : t2);
        };
        sums(j, t.x, sn0.x, sn1.x, sn2.x, sq.x);
        if (j + 1 < J) sums(j + 1, t.y, sn0.y, sn1.y, sn2.y, sq.y);
    }
}

}  // namespace

template <bool BF16, int JM>
__global__ void __launch_bounds__(REG_STRIP_THREADS, TRIAL_BLOCKS) k_trial(BatchDev b)
{
    __shared__ TrialTile<JM> sh;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int item = blockIdx.x;; item += gridDim.x) {
        const WorkPlan wp = work_plan<false>(b, lane);
        if (item >= wp.items) break;
        int tile;
        const StepDesc &s = b.st[find_item<false>(b, wp, item, tile)].step;
        const StripGeom g = strip_geom(s, tile, lane);
        const int part = s.part0 + tile;
        if (s.phase == PH_START || s.phase == PH_PROLONG) {
            // sums in double, reduced in double: [0..2] and the Dirichlet form of u
            double v[4];
            const int rows = g.rEnd - g.r0 + 1, per = (rows + TRIAL_WARPS - 1) / TRIAL_WARPS;
            const int ra = g.r0 + min(wid * per, rows);
            start_rows<BF16>(s, g, ra, min(ra + per, g.rEnd + 1), v);
#pragma unroll
            for (int k = 0; k < 4; k++) {
                const double tot = warp_sum_d(v[k]);
                if (lane == 0) sh.start[wid][k] = tot;
            }
            __syncthreads();
            if (threadIdx.x < 4) {
                double t = 0.0;
#pragma unroll
                for (int w = 0; w < TRIAL_WARPS; w++) t += sh.start[w][threadIdx.x];
                b.partU[4 * (int64_t)part + threadIdx.x] = t;
            }
        } else {
            trial_tile<BF16, JM>(b, s, g, sh, part, wid, lane);
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// C: per-operator sums, the Armijo state machine, and the plan of the next step
// ---------------------------------------------------------------------------
namespace {

// (The rare paths are calls: the code of a step's common path runs once per launch, and
// its length in instruction fetches counts.)
__device__ __noinline__ void eval_rare(EvalAt &v, double var)
{
    const double sig = var > 0.0 ? sqrt(var) : 0.0;
    v.ncc = v.S3 / sig;
    v.isig = (float)(1.0 / sig);
    v.c36 = (float)(v.ncc / (sig * sig) / 36.0);
    v.cT = (float)(v.ncc / (sig * sig) * v.S1);
}

// NCC and the gradient pass's coefficients from the FE sums.  The square root and
// division of double precision take 600 cycles each here, the chain of rsqrt_step and
// times nine dependent operations of 62.
__device__ __forceinline__ void eval_at(EvalAt &v, double S1, double S2, double S3)
{
    const double var = S2 - S1 * S1;
    v.S1 = S1;
    v.S2 = S2;
    v.S3 = S3;
    if (var > 1e-30 && var < 1e30) {
        const RootInv r = rsqrt_step(var, rsqrtf((float)var));
        v.ncc = times(S3, r);
        v.isig = (float)r.r;
        const double q = v.ncc * (r.r * r.r);
        v.c36 = (float)(q * (1.0 / 36.0));
        v.cT = (float)(q * S1);
    } else {  // (almost) no variance, or not finite
        EvalAt w = v;
        eval_rare(w, var);
        v = w;
    }
}

// Positive doubles compare like their bits, and doubling one adds to its
// exponent field: the step sizes of the search stay off the slow FP64 pipe.
// (Numbers near the ends of the exponent range take the multiplication.)
__device__ __noinline__ double pow2_rare(double x, int e) { return scalbn(x, e); }
__device__ __forceinline__ double pow2_scale(double x, int e)
{
    const long long w = __double_as_longlong(x);
    const int ex = (int)(w >> 52);
    return ex > 8 && ex < 0x7f0 ? __longlong_as_double(w + ((long long)e << 52)) : pow2_rare(x, e);
}
__device__ __forceinline__ double twice(double x) { return pow2_scale(x, 1); }
__device__ __forceinline__ double half_of(double x) { return pow2_scale(x, -1); }
__device__ __forceinline__ bool pos_le(double a, double b) { return __double_as_longlong(a) <= __double_as_longlong(b); }
__device__ __forceinline__ bool pos_eq(double a, double b) { return __double_as_longlong(a) == __double_as_longlong(b); }

__device__ __forceinline__ void trace_trial(const BatchDev &b, int o, int n, int iter, double want, double slope,
                                            const EvalAt &v)
{
    unsigned long long k = atomicAdd(b.trace_len, 1ull);
    if ((long long)k < b.trace_cap) {
        double *rec = b.trace + 7 * k;
        rec[0] = o; rec[1] = n; rec[2] = iter - 1; rec[3] = want;
        rec[4] = v.dE; rec[5] = b.sigma * want * slope; rec[6] = v.acc;
    }
}

// The Armijo state machine of one operator after a step, by one warp (s and op in
// shared memory, s written by this warp only).  Lane j holds trial j (lane 0 a
// level's start, its energy in dE); the decisions are uniform, taken from ballots
// over the lanes.
__device__ __forceinline__ void control_op(const BatchDev &b, OpState &s, const OpDesc &op, int o, int n, int lane,
                                           const EvalAt &ev, double mytau, double slope)
{
    const unsigned FULL = 0xffffffffu;
    const int ph = s.phase, ntr = s.ntr;
    int iter = s.iter, status = -1;  // status >= 0: the level ends
    bool go = false;                 // next: a gradient pass at the level
    double pending = 0.0, tau = s.tau;
    const unsigned long long nn = (unsigned long long)n * n;
    int evals = ph == PH_START || ph == PH_PROLONG ? 1 : ntr, seq = 0;
    if (ph == PH_START || ph == PH_PROLONG) {
        if (lane == 0) {
            s.cur_ev = ev;
            s.E = ev.dE;
        }
        iter = 0;
        tau = b.tau_init;
        const bool fin = __shfl_sync(FULL, (int)isfinite(ev.dE), 0);
        if (!fin) status = OPST_NONFINITE;
        else if (op.lock_tau && op.lock_off[s.lvl + 1] == op.lock_off[s.lvl]) status = OPST_MAXITER;
        else go = true;
    } else {
        bool search_on = true;
        if (ph == PH_GRAD) {
            iter++;
            if (!(slope < 0.0)) {
                status = slope == 0.0 ? OPST_ZERO_GRAD : OPST_NONFINITE;
                search_on = false;
                evals = 0;
            }
        }
        const unsigned accs = __ballot_sync(FULL, lane < ntr && ev.acc);
        if (search_on && op.lock_tau) {
            // lockstep replay: take the given step whatever the test says (the
            // trace records the test), end the level after the last given step
            seq = 1;
            if (lane == 0) {
                if (b.trace) trace_trial(b, o, n, iter, mytau, slope, ev);
                s.E += ev.dE;
                s.cur_ev = ev;
            }
            tau = pending = s.trial_tau[0];
            if (iter >= op.lock_off[s.lvl + 1] - op.lock_off[s.lvl]) status = OPST_MAXITER;
            else go = true;
        } else if (search_on) {
            // walk the sequential Armijo search over the step sizes evaluated this pass
            int search = s.search, best = -1;  // best: the last trial accepted in this pass
            double btau = s.btau, sh_tau = s.sh_tau;
            bool finish = false, more = false;
            int guard = 0;
#pragma unroll 1
            for (; guard < 4 * REG_MAX_TRIALS + 8 && !finish && status < 0; guard++) {
                const double want =
                    search == SEARCH_INIT ? tau : (search == SEARCH_WIDEN ? twice(btau) : half_of(sh_tau));
                if (search == SEARCH_WIDEN && !pos_le(want, b.tau_max)) { finish = true; break; }
                if (search == SEARCH_SHRINK && !pos_le(b.tau_min, want)) { status = OPST_STALLED; break; }
                const unsigned at = __ballot_sync(FULL, lane < ntr && pos_eq(mytau, want));
                if (!at) {
                    // continue the search in another pass
                    int k = 0;
                    double t = want;
                    while (k < b.J && (search == SEARCH_WIDEN ? pos_le(t, b.tau_max) : pos_le(b.tau_min, t))) {
                        if (lane == k) {
                            s.trial_tau[k] = t;
                            s.step.tau[k] = (float)t;
                        }
                        t = search == SEARCH_WIDEN ? twice(t) : half_of(t);
                        k++;
                    }
                    if (lane == 0) {
                        s.ntr = k;
                        s.phase = PH_TRIAL;
                    }
                    more = true;
                    break;
                }
                const int j = __ffs(at) - 1;
                seq++;
                if (b.trace && lane == j) trace_trial(b, o, n, iter, want, slope, ev);
                const bool acc = accs >> j & 1;
                if (acc) best = j;
                if (search == SEARCH_SHRINK) {
                    if (acc) { btau = want; finish = true; }
                    else sh_tau = want;
                } else if (acc) {
                    search = SEARCH_WIDEN;
                    btau = want;
                } else if (search == SEARCH_INIT) {
                    search = SEARCH_SHRINK;
                    sh_tau = want;
                } else {
                    finish = true;
                }
            }
            if (finish) {
                const bool conv = best >= 0 ? __shfl_sync(FULL, ev.conv, best) != 0 : s.best_ev.conv != 0;
                __syncwarp();
                if (best >= 0) {
                    if (lane == best) {
                        s.cur_ev = ev;
                        s.E += ev.dE;
                    }
                } else if (lane == 0) {
                    s.cur_ev = s.best_ev;
                    s.E += s.best_ev.dE;
                }
                tau = pending = btau;
                if (conv) status = OPST_CONVERGED;
                else if (iter >= b.iter_max) status = OPST_MAXITER;
                else go = true;
            } else if (more) {
                if (lane == max(best, 0) && best >= 0) s.best_ev = ev;
                if (lane == 0) {
                    s.search = search;
                    s.btau = btau;
                    s.sh_tau = sh_tau;
                }
            } else if (status < 0) {  // the search did not terminate: internal error
                if (lane == 0) {
                    atomicExch(&b.ctr[8], 1);
                    s.phase = PH_DONE;
                }
            }
        }
    }
    __syncwarp();
    if (status >= 0) {
        const int lvl = s.lvl, cur = s.cur, last = op.nl - 1;
        __syncwarp();
        if (lane == 0) {
            if (status == OPST_NONFINITE) s.nonfinite_seen = 1;
            s.status = status;
            s.tau_acc = pending;
            s.step.tau_acc = (float)pending;
            s.src = cur;
            if (lvl < last) {
                s.phase = PH_PROLONG;
                s.lvl = lvl + 1;
                s.cur = 0;
            } else {
                s.phase = PH_DONE;
            }
        }
    } else if (go) {
        if (lane == 0) {
            s.phase = PH_GRAD;
            s.tau_acc = pending;
            s.step.tau_acc = (float)pending;
            s.src = s.cur;
            s.cur = 1 - s.cur;
            s.search = SEARCH_INIT;
        }
        // step sizes in the sequential Armijo order: tau, then 2 tau (if accepted), else
        // tau / 2; the pass covers the most likely continuations of both branches
        const int J = b.J;
        if (op.lock_tau) {
            // replay: the one step size the reference sequence accepted here
            if (lane == 0) {
                const double t = op.lock_tau[op.lock_off[s.lvl] + iter];
                s.trial_tau[0] = t;
                s.step.tau[0] = (float)t;
                s.ntr = 1;
            }
        } else if (pos_le(pow2_scale(tau, J / 2), b.tau_max) && pos_le(b.tau_min, pow2_scale(tau, -((J - 1) / 2)))) {
            if (lane < J) {
                const double t = pow2_scale(tau, (lane & 1) ? (lane + 1) / 2 : -(lane / 2));
                s.trial_tau[lane] = t;
                s.step.tau[lane] = (float)t;
            }
            if (lane == 0) s.ntr = J;
        } else if (lane == 0) {  // at the ends of the admitted range
            int k = 0;
            double up = tau, dn = tau;
            auto put = [&](double t) {
                s.trial_tau[k] = t;
                s.step.tau[k++] = (float)t;
            };
            put(up);
            while (k < J) {
                const double u2 = twice(up), d2 = half_of(dn);
                const bool canUp = pos_le(u2, b.tau_max), canDn = pos_le(b.tau_min, d2);
                if (!canUp && !canDn) break;
                if (canUp) { up = u2; put(up); }
                if (k < J && canDn) { dn = d2; put(dn); }
            }
            s.ntr = k;
        }
    }
    if (lane == 0) {
        s.tau = tau;
        s.iter = iter;
        if (ph == PH_GRAD) {
            s.iters_total += 1;
            s.slope = slope;
        }
        s.evals += evals;
        s.trials_seq += seq;
        if (seq) atomicAdd(&b.work[KW_TSEQ], nn * seq);
    }
    __syncwarp();
}

// Adds over the 32 lanes (the sum in every lane, not split alike).
__device__ __forceinline__ void warp_sum3(Sum3 &v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float a = __shfl_xor_sync(0xffffffffu, v.a, o), c = __shfl_xor_sync(0xffffffffu, v.b, o),
                    d = __shfl_xor_sync(0xffffffffu, v.c, o);
        v.add(a);
        v.add(c);
        v.add(d);
    }
}

}  // namespace

// One block per operator (grid stride): the block sums the operator's tile
// partials, the lanes of a warp evaluate all trials side by side and run the state
// machine on copies of the state and the descriptor in shared memory.  Batches of
// more than PLAN_WARP operators: the last block to finish makes the lists of the next
// step (narrower ones need none).  Latency bound at every size.
//
// The FP64 pipe takes 16 cycles for a warp's operation and 62 until its result: sums
// and reductions of the tiles' floats in FP64 were 6000 of 15000 cycles at 65^2 nodes
// and 18000 of 28000 at 1025^2, a chain of square roots and divisions 2900, the state
// machine as one thread's loads and stores 3000 to 4700.  The sums run in float
// triples now (exact to 2^-72, more than FP64 keeps): thread (g, kk) adds entry kk of
// every ng-th record (kk fastest, so a warp reads neighbouring floats), only the
// entries that the pass wrote, 3 per step size and one Dirichlet form (at most 13
// for up to four step sizes: 32 groups; else 16 groups), and the gradient pass's two
// sums as two more entries; then one warp per entry adds the groups.
__global__ void __launch_bounds__(REG_CTL_THREADS) k_control(BatchDev b)
{
    constexpr int NW = REG_CTL_THREADS / 32;
    constexpr int NS = sizeof(OpState) / 8, ND = sizeof(OpDesc) / 8;
    static_assert(sizeof(OpState) % 8 == 0 && sizeof(OpDesc) % 8 == 0 && NS + ND <= REG_CTL_THREADS,
                  "state and descriptor copied in one pass");
    __shared__ __align__(16) double sbuf[NS], dbuf[ND];
    __shared__ float red[3][REG_CTL_THREADS + 32];
    __shared__ float sums[3][32];
    __shared__ double startS[4];
    __shared__ int last;
    OpState &s = *reinterpret_cast<OpState *>(sbuf);
    const OpDesc &op = *reinterpret_cast<const OpDesc *>(dbuf);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int lg = b.J <= 4 ? 4 : 5, ng = REG_CTL_THREADS >> lg;
    int n_ops = 0;
    // (the first operator's state is read beside the operator count: a grid never has
    // more blocks than there is room for operators)
    for (int o = blockIdx.x; o == (int)blockIdx.x || o < n_ops; o += gridDim.x) {
        if (tid < NS) sbuf[tid] = reinterpret_cast<const double *>(b.st + o)[tid];
        else if (tid < NS + ND) dbuf[tid - NS] = reinterpret_cast<const double *>(b.ops + o)[tid - NS];
        n_ops = b.ctr[0];
        if (o >= n_ops) return;
        __syncthreads();
        const int ph = s.phase;
        if (ph != PH_DONE) {
            const int n = s.step.n, ntr = s.ntr, nt = s.tT;
            const double h2 = op.lv[s.lvl].h2d;
            const bool start = ph == PH_START || ph == PH_PROLONG;
            if (tid == REG_CTL_THREADS - 1) {
                // algorithmic work of this step (nodes of the level each kernel swept)
                const unsigned long long nn = (unsigned long long)n * n;
                if (ph == PH_PROLONG) atomicAdd(&b.work[KW_PPROL], nn);
                if (start) atomicAdd(&b.work[KW_TSTART], nn);
                if (ph == PH_GRAD) atomicAdd(&b.work[KW_G], nn);
                if (!start) {
                    atomicAdd(&b.work[KW_T], nn);
                    atomicAdd(&b.work[KW_TSAMPLES], nn * (unsigned long long)ntr);
                }
            }
            // entries 0 .. 3 ntr - 1 and the Dirichlet form of d; the last two of a group
            // are the gradient pass's (or the smoother's)
            const int ne = 3 * ntr + 1, e0 = (1 << lg) - 2;
            if (start) {
                // doubles: three sums and the Dirichlet form of u
                if (wid < 4) {
                    double v = 0.0;
                    for (int it = lane; it < nt; it += 32) v += b.partU[4 * ((int64_t)op.part0 + it) + wid];
                    v = warp_sum_d(v);
                    if (lane == 0) startS[wid] = v;
                }
                __syncthreads();
            } else {
                const int kk = tid & ((1 << lg) - 1), g = tid >> lg;
                const float *rec = nullptr;
                int stride = PT_STRIDE, cnt = 0;
                if (kk < ne) {
                    rec = b.partT + (int64_t)op.part0 * PT_STRIDE + (kk < ne - 1 ? kk : 3 * REG_MAX_TRIALS + 2);
                    cnt = nt;
                } else if (kk >= e0 && ph == PH_GRAD) {
                    // gradient tiles, or the smoother's column chunks
                    rec = (b.smooth ? b.partS + (int64_t)o * b.cch * 2 : b.partG + (int64_t)op.part0 * PG_STRIDE) + (kk - e0);
                    stride = PG_STRIDE;
                    cnt = b.smooth ? (n + REG_GW - 1) / REG_GW : s.tG;
                }
                Sum3 v;
                int it = g;
                // eight loads in flight
                for (; it < cnt; it += 8 * ng) {
                    float x[8];
#pragma unroll
                    for (int q = 0; q < 8; q++) x[q] = it + q * ng < cnt ? rec[(it + q * ng) * stride] : 0.f;
#pragma unroll
                    for (int q = 0; q < 8; q++)
                        if (it + q * ng < cnt) v.add(x[q]);
                }
                const int at = kk * (ng + 1) + g;
                red[0][at] = v.a;
                red[1][at] = v.b;
                red[2][at] = v.c;
                __syncthreads();
                for (int k = wid; k < (1 << lg); k += NW) {
                    if (k >= ne && k < e0) continue;
                    Sum3 w;
                    if (lane < ng) {
                        const int i = k * (ng + 1) + lane;
                        w.a = red[0][i];
                        w.b = red[1][i];
                        w.c = red[2][i];
                    }
                    warp_sum3(w);
                    if (lane == 0) {  // (one lane's triple: the lanes split the sum differently)
                        sums[0][k] = w.a;
                        sums[1][k] = w.b;
                        sums[2][k] = w.c;
                    }
                }
                __syncthreads();
            }
            if (wid == 0) {
                const unsigned FULL = 0xffffffffu;
                EvalAt v;
                v.dE = 0.0;
                v.acc = v.conv = 0;
                double slope = s.slope, mytau = 0.0;
                if (start) {
                    eval_at(v, h2 * startS[0], h2 * startS[1], h2 * startS[2]);
                    v.dE = -v.ncc + 0.5 * b.lambda * h2 * startS[3];
                } else {
                    // lane k: entry k's sum
                    const double e = (double)sums[0][lane] + ((double)sums[1][lane] + (double)sums[2][lane]);
                    double Qud = s.Qud, Qdd = s.Qdd;
                    const double eq = __shfl_sync(FULL, e, ne - 1), es = __shfl_sync(FULL, e, e0),
                                 eu = __shfl_sync(FULL, e, e0 + 1);
                    if (ph == PH_GRAD) {
                        // the Dirichlet forms of the search: u^T K d from the gradient pass
                        // (or the smoother), d^T K d from its first trial pass
                        slope = b.smooth ? -h2 * h2 * es : es;
                        Qud = eu;
                        Qdd = eq;
                    }
                    const int j3 = 3 * min(lane, ntr - 1);
                    const double d1 = __shfl_sync(FULL, e, j3), d2 = __shfl_sync(FULL, e, j3 + 1),
                                 d3 = __shfl_sync(FULL, e, j3 + 2);
                    mytau = s.trial_tau[min(lane, REG_MAX_TRIALS - 1)];
                    const double E = s.E, hl = 0.5 * b.lambda * h2;
                    const double reg = hl * (mytau * fma(mytau, Qdd, 2.0 * Qud));
                    const double bound = b.sigma * mytau * slope, stop = b.eps * (fabs(E) > 1.0 ? fabs(E) : 1.0);
                    eval_at(v, s.cur_ev.S1 + h2 * d1, s.cur_ev.S2 + h2 * d2, s.cur_ev.S3 + h2 * d3);
                    // energy change E(u + tau d) - E(u) from the accumulated sums at u
                    v.dE = -(v.ncc - s.cur_ev.ncc) + reg;
                    v.acc = v.dE <= bound;
                    v.conv = -v.dE < stop;
                    __syncwarp();
                    if (lane == 0 && ph == PH_GRAD) {
                        s.Qud = Qud;
                        s.Qdd = Qdd;
                    }
                }
                __syncwarp();
                control_op(b, s, op, o, n, lane, v, mytau, slope);
                if (lane == 0) {
                    set_step(s, op);
                    b.plan[o] = make_int2(s.tG, s.tT);
                    if (s.phase == PH_DONE) atomicAdd(&b.ctr[7], -1);
                }
            }
            __syncthreads();
            if (tid < NS) reinterpret_cast<double *>(b.st + o)[tid] = sbuf[tid];
        }
        __syncthreads();
    }
    if (n_ops <= PLAN_WARP) return;
    // the last block makes the lists: its reads of the other blocks' entries follow
    // their fences
    if (tid == 0) {
        __threadfence();
        last = atomicAdd(&b.ctr[9], 1) == min((int)gridDim.x, n_ops) - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    plan_lists(b);
    if (tid == 0) b.ctr[9] = 0;
}

// ---------------------------------------------------------------------------
// Series averaging (Section "Introduction": the frames f_i o phi_{0,i} of a
// registered series are averaged into one frame)
// ---------------------------------------------------------------------------

// Node (r, c) of the finest level: 1/m sum_k F_k(x + u_k(x)), F_k frame k's
// stored finest level with its normalisation undone (F = F~ sigma_k + mean_k),
// sampled bilinearly and clamped to the grid; u_k from fields[k] (float2 grid
// units of the finest level; null = the identity), as sums in double give it.
// Three FP64 operations per sample and the division (16 cycles of an SM each for a
// warp) took 345 of the 415 us for 64 frames of 1025^2, so the products, their sum
// and its product with 1/m run in float pairs (PairSum, whose bound grows with the
// number of frames; the means' sum and 1/m are two constants of the block); a node
// whose rounding that does not settle, one in 10^4 at 64 frames, is summed again in
// FP64 by its warp.  A call for 64 frames takes 258 us (443 with FP64 sums, 308 with the
// end of a node in FP64: two divisions); bound by issue and the latency of field ->
// texel chains.
constexpr int AVG_FRAMES = 128;  // frames staged in shared memory at a time
constexpr int AVG_BATCH = 2;     // frames whose fields, then texels, a thread has in flight
template <bool BF16>
__global__ void __launch_bounds__(256) k_average(const void *__restrict__ pyr, int64_t frame_block, int64_t img_off,
                                                 int n, int pitch, const double *__restrict__ fstats,
                                                 const float2 *const *__restrict__ fields, int slot_pitch, int m,
                                                 float *__restrict__ out, int opitch)
{
    __shared__ const float2 *fld[AVG_FRAMES];
    __shared__ const void *img[AVG_FRAMES];
    __shared__ float2 sig[AVG_FRAMES];  // sigma_k as two floats
    __shared__ float2 mean_sum, inv_m;  // as two floats
    const int c = blockIdx.x * 32 + threadIdx.x, r = blockIdx.y * 8 + threadIdx.y;
    const int tid = threadIdx.y * 32 + threadIdx.x;
    const bool in = r < n && c < n;
    const int node = r * slot_pitch + c;
    auto image = [&](int k) {
        return BF16 ? (const void *)(reinterpret_cast<const __nv_bfloat16 *>(pyr) + k * frame_block + img_off)
                    : (const void *)(reinterpret_cast<const float *>(pyr) + k * frame_block + img_off);
    };
    if (tid < 32) {
        double s = 0.0;
        for (int k = tid; k < m; k += 32) s += fstats[2 * k];
        s = warp_sum_d(s);
        if (tid == 0) mean_sum = make_float2((float)s, (float)(s - (double)(float)s));
    } else if (tid == 32) {
        const double s = 1.0 / m;
        inv_m = make_float2((float)s, (float)(s - (double)(float)s));
    }
    PairSum sum;
    for (int k0 = 0; k0 < m; k0 += AVG_FRAMES) {
        const int mk = min(AVG_FRAMES, m - k0);
        __syncthreads();
        for (int k = tid; k < mk; k += 256) {
            fld[k] = fields[k0 + k];
            img[k] = image(k0 + k);
            const double s = fstats[2 * (k0 + k) + 1];
            const float sh = (float)s;
            sig[k] = make_float2(sh, (float)(s - (double)sh));
        }
        __syncthreads();
        if (in) {
            static_assert(AVG_BATCH <= 2, "folded after at most two products");
            auto add = [&](int k, float v) { sum.add(v, sig[k].x, sig[k].y); };
            for (int k = 0; k < mk; k += AVG_BATCH) {
                float2 u[AVG_BATCH];
                float far = 0.f;
#pragma unroll
                for (int q = 0; q < AVG_BATCH; q++) {
                    const float2 *f = fld[min(k + q, mk - 1)];
                    u[q] = f ? f[node] : make_float2(0.f, 0.f);
                }
#pragma unroll
                for (int q = 0; q < AVG_BATCH; q++) far += fabsf(u[q].x) + fabsf(u[q].y);
                if (far < 2097152.f) {
                    Texel4 t[AVG_BATCH];
#pragma unroll
                    for (int q = 0; q < AVG_BATCH; q++) {
                        locate(n, c, r, u[q].x, u[q].y, t[q].jx, t[q].jy, t[q].ax, t[q].ay, t[q].clx, t[q].cly);
                        fetch<BF16>(t[q], img[min(k + q, mk - 1)], pitch);
                    }
#pragma unroll
                    for (int q = 0; q < AVG_BATCH; q++)
                        if (k + q < mk) add(k + q, bil(t[q]));
                } else {  // beyond floor_i's range, or NaN
                    for (int q = 0; q < AVG_BATCH && k + q < mk; q++)
                        add(k + q, sample<BF16, false>(img[k + q], n, pitch, c, r, u[q].x, u[q].y, nullptr, nullptr));
                }
                sum.fold();
            }
        }
    }
    float p, pl;
    sum.scaled(mean_sum.x, mean_sum.y, inv_m.x, inv_m.y, p, pl);
    const float size = (sum.mag + fabsf(mean_sum.x)) * inv_m.x, tol = sum.tolerance(m, mean_sum.x, inv_m.x);
    const float a = p + (pl - tol), b = p + (pl + tol);
    float res = a;
    // Open nodes (the low parts of tiny values underflow: open too) in FP64, the frames
    // over the lanes of the node's warp: one thread's chain of m gathers was 20 us for
    // 64 frames, as long as it takes at the end of the launch.
    unsigned open = __ballot_sync(0xffffffffu, in && (!(a == b) || !(size > 1e-25f)));
    while (open) {
        const int src = __ffs(open) - 1, cs = blockIdx.x * 32 + src;
        open &= open - 1;
        double acc = 0.0;
        for (int k = threadIdx.x; k < m; k += 32) {
            const float2 *f = fields[k];
            const float2 u = f ? f[(int64_t)r * slot_pitch + cs] : make_float2(0.f, 0.f);
            const float v = sample<BF16, false>(image(k), n, pitch, cs, r, u.x, u.y, nullptr, nullptr);
            acc += (double)v * fstats[2 * k + 1] + fstats[2 * k];
        }
        acc = warp_sum_d(acc);
        if ((int)threadIdx.x == src) res = (float)(acc / m);
    }
    if (in) out[(int64_t)r * opitch + c] = res;
}

void launch_average(int bf16, cudaStream_t st, const void *pyr, int64_t frame_block, int64_t img_off, int n,
                    int pitch, const double *fstats, const float2 *const *fields, int slot_pitch, int m, float *out,
                    int opitch)
{
    dim3 blk(32, 8), grid(cdiv(n, 32), cdiv(n, 8));
    if (bf16) k_average<true><<<grid, blk, 0, st>>>(pyr, frame_block, img_off, n, pitch, fstats, fields, slot_pitch, m, out, opitch);
    else k_average<false><<<grid, blk, 0, st>>>(pyr, frame_block, img_off, n, pitch, fstats, fields, slot_pitch, m, out, opitch);
}

// ---------------------------------------------------------------------------
// Rigid variant (Definition "Rigid transformation": phi(x) = R(alpha) x + t;
// Section "Gradient flow": no smoother in the rigid case)
// ---------------------------------------------------------------------------

// Rigid displacement of node (c, r) in grid units of a level of n nodes:
// u = (R(alpha) - I) x + t with a = cos(alpha) - 1, b = sin(alpha) and the
// translation (tx, ty) in grid units.
__device__ __forceinline__ float2 rigid_u(const RigidReq &q, int c, int r)
{
    return make_float2(fmaf(q.a, (float)c, fmaf(-q.b, (float)r, q.tx)), fmaf(q.b, (float)c, fmaf(q.a, (float)r, q.ty)));
}

// One block per 32 x 32 node tile, operator and requested parameter set (grid:
// tiles, ops, sets; one block for all sets of a tile left small batches waiting on
// four serial passes).  For parameter set j < q.n_e: the FE sums of the warped template
// That = T(x + u) over the tile (nodes and cells it owns): sum omega That,
// sum of the Q1 element mass forms of That, sum That M~R~ (multiplied by h^2
// on the host).  With q.grad: the data part of dE/dtheta at parameter set 0,
//   -sum_i dNCC/dThat_i (dT_0 du_0/dtheta + dT_1 du_1/dtheta),
//   dNCC/dThat_i = h^2 [ M~R~_i / sigma_T - NCC ((M~ That)_i - T_bar omega_i) / sigma_T^2 ],
// derivatives in Omega units.  That of the tile and a one-node halo is kept in
// shared memory for the cell forms and M~ That.
template <bool BF16>
__global__ void __launch_bounds__(256) k_rigid_eval(const RigidLevel *__restrict__ lv, const RigidReq *__restrict__ req,
                                                    double *__restrict__ part)
{
    constexpr int TS = 32, HS = TS + 2;
    __shared__ float sh[HS][HS + 1];
    __shared__ float red[8][RIGID_SUMS];
    const int o = blockIdx.y;
    const RigidLevel L = lv[o];
    const int n = L.n;
    const int tx = (n + TS - 1) / TS;
    const int tile = blockIdx.x;
    if (tile >= tx * tx) return;
    const int c0 = (tile % tx) * TS, r0 = (tile / tx) * TS;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    double *out = part + ((int64_t)o * gridDim.x + tile) * RIGID_SUMS;
    const RigidReq *qs = req + (int64_t)o * REG_MAX_TRIALS;
    auto omega = [n](int i) { return (i == 0 || i == n - 1) ? 0.5f : 1.f; };
    auto w6 = [n](int i, int a) { return a == 0 ? ((i == 0 || i == n - 1) ? 2.f : 4.f) : 1.f; };
    const int j = blockIdx.z;
    if (j >= qs[0].n_e) return;
    {
        const RigidReq q = qs[j];
        const bool grad = (j == 0) && q.grad;
        // That on the tile plus a one-node halo (nodes outside the grid: 0)
        for (int k = threadIdx.x; k < HS * HS; k += blockDim.x) {
            const int rr = r0 - 1 + k / HS, cc = c0 - 1 + k % HS;
            float v = 0.f;
            if (rr >= 0 && rr < n && cc >= 0 && cc < n) {
                const float2 u = rigid_u(q, cc, rr);
                v = sample<BF16, false>(L.T, n, L.pitch, cc, rr, u.x, u.y, nullptr, nullptr);
            }
            sh[k / HS][k % HS] = v;
        }
        __syncthreads();
        float s1 = 0.f, s2 = 0.f, s3 = 0.f, g0 = 0.f, g1 = 0.f, g2 = 0.f;
        for (int k = threadIdx.x; k < TS * TS; k += blockDim.x) {
            const int lr = k / TS, lc = k % TS, r = r0 + lr, c = c0 + lc;
            if (r >= n || c >= n) continue;
            const float t = sh[lr + 1][lc + 1];
            const float om = omega(r) * omega(c);
            const float mr = L.MR[(int64_t)r * L.pitch + c];
            s1 += om * t;
            s3 += t * mr;
            if (r < n - 1 && c < n - 1) {
                // cell (r, c): corners a=(r,c) b=(r,c+1) cc=(r+1,c+1) d=(r+1,c), element mass (1/36)[4 2 1 2; ...]
                const float A = t, B = sh[lr + 1][lc + 2], C = sh[lr + 2][lc + 2], D = sh[lr + 2][lc + 1];
                s2 += (4.f * (A * A + B * B + C * C + D * D) + 4.f * (A * B + B * C + C * D + D * A) +
                       2.f * (A * C + B * D)) * (1.f / 36.f);
            }
            if (grad) {
                // (36 M~ That)_i: integer weights, boundary rows/cols halved
                float mt = 0.f;
                for (int a = -1; a <= 1; a++) {
                    if (r + a < 0 || r + a >= n) continue;
                    float row = 0.f;
                    for (int b = -1; b <= 1; b++) {
                        if (c + b < 0 || c + b >= n) continue;
                        row += w6(c, b) * sh[lr + 1 + a][lc + 1 + b];
                    }
                    mt += w6(r, a) * row;
                }
                const float2 u = rigid_u(q, c, r);
                float dx, dy;
                sample<BF16, true>(L.T, n, L.pitch, c, r, u.x, u.y, &dx, &dy);
                // dNCC/dThat_i / h^2, times (n - 1) for derivatives in Omega units
                const float dn = (mr * q.inv_sig - q.ncc_over_var * (mt * (1.f / 36.f) - q.tbar * om)) * q.nm1;
                const float x0 = (float)c * q.h, x1 = (float)r * q.h;
                g0 -= dn * (dx * (-q.sa * x0 - q.ca * x1) + dy * (q.ca * x0 - q.sa * x1));
                g1 -= dn * dx;
                g2 -= dn * dy;
            }
        }
        float v[6] = {s1, s2, s3, g0, g1, g2};
        const int nv = grad ? 6 : 3;
        for (int m = 0; m < nv; m++) {
            float w = warp_sum(v[m]);
            if (lane == 0) red[wid][m] = w;
        }
        __syncthreads();
        if (threadIdx.x < nv) {
            double acc = 0.0;
            for (int w = 0; w < 8; w++) acc += red[w][threadIdx.x];
            out[(threadIdx.x < 3 ? 3 * j : 3 * REG_MAX_TRIALS - 3) + threadIdx.x] = acc;
        }
    }
}

// Per operator: the tiles' partial sums in a fixed order (one block per op): warp by
// warp of 32 tiles, then the warps' sums in order, up to 256 tiles; beyond, a lane
// first adds every 256th.  Each warp takes (sum, group of 32 tiles) pairs of the sums
// the request asks for; one sum after the other through the whole block took 21 us.
__global__ void __launch_bounds__(1024) k_rigid_reduce(const double *__restrict__ part, int tiles_stride,
                                                       const RigidLevel *__restrict__ lv,
                                                       const RigidReq *__restrict__ req, double *__restrict__ sums)
{
    const int o = blockIdx.x;
    const int n = lv[o].n, tx = (n + 31) / 32, tiles = tx * tx;
    const RigidReq &q = req[(int64_t)o * REG_MAX_TRIALS];
    __shared__ double red[RIGID_SUMS][8];
    const int lane = threadIdx.x & 31, groups = min(8, (tiles + 31) / 32);
    const int ne = q.n_e > 0 ? 3 * q.n_e + (q.grad ? 3 : 0) : 0;
    for (int p = threadIdx.x >> 5; p < ne * groups; p += 32) {
        const int k = p / groups, g = p % groups;
        const int m = k < 3 * q.n_e ? k : 3 * REG_MAX_TRIALS + (k - 3 * q.n_e);
        double acc = 0.0;
        for (int t = g * 32 + lane; t < tiles; t += 256) acc += part[((int64_t)o * tiles_stride + t) * RIGID_SUMS + m];
        acc = warp_sum_d(acc);
        if (lane == 0) red[m][g] = acc;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < ne; k += 1024) {
        const int m = k < 3 * q.n_e ? k : 3 * REG_MAX_TRIALS + (k - 3 * q.n_e);
        double acc = 0.0;
        for (int w = 0; w < groups; w++) acc += red[m][w];
        sums[(int64_t)o * RIGID_SUMS + m] = acc;
    }
}

// The finest-level field of rigid parameters, in pixels (= grid units of the
// finest level), into a slot: u = (R(alpha) - I) x + t.
__global__ void k_rigid_fill(RigidReq q, int n, float2 *__restrict__ slot, int pitch)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x, r = blockIdx.y * blockDim.y + threadIdx.y;
    if (r >= n || c >= n) return;
    slot[(int64_t)r * pitch + c] = rigid_u(q, c, r);
}

void launch_rigid(int bf16, int tiles, int n_ops, int sets, cudaStream_t st, const RigidLevel *lv, const RigidReq *req,
                  double *part, double *sums)
{
    dim3 grid(tiles, n_ops, sets);
    if (bf16) k_rigid_eval<true><<<grid, 256, 0, st>>>(lv, req, part);
    else k_rigid_eval<false><<<grid, 256, 0, st>>>(lv, req, part);
    k_rigid_reduce<<<n_ops, 1024, 0, st>>>(part, tiles, lv, req, sums);
}

void launch_rigid_fill(const RigidReq &q, int n, float2 *slot, int pitch, cudaStream_t st)
{
    k_rigid_fill<<<dim3(cdiv(n, 32), cdiv(n, 8)), dim3(32, 8), 0, st>>>(q, n, slot, pitch);
}

// ---------------------------------------------------------------------------
// Slot conversion helpers
// ---------------------------------------------------------------------------

// slot (float2, (side+1)^2 grid) -> planes (2 x side x side) for output
__global__ void k_slot_to_planes(const float2 *__restrict__ slot, int pitch, int side, float *__restrict__ out)
{
    int c = blockIdx.x * blockDim.x + threadIdx.x, r = blockIdx.y * blockDim.y + threadIdx.y;
    if (r >= side || c >= side) return;
    float2 v = slot ? slot[(int64_t)r * pitch + c] : make_float2(0.f, 0.f);
    out[(int64_t)r * side + c] = v.x;
    out[(int64_t)side * side + (int64_t)r * side + c] = v.y;
}

// Frames k0 .. k0 + gridDim.z - 1 of a series' deformations, planes (2 x side
// x side each) from their slots: frame k > 0 from slot k - 1 (slots slot_elems
// apart), frame 0 from slot0 (null: the identity, zero displacement).
__global__ void k_slots_to_planes(const float2 *__restrict__ slots, int64_t slot_elems, int k0,
                                  const float2 *__restrict__ slot0, int pitch, int side, float *__restrict__ out)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x, r = blockIdx.y * blockDim.y + threadIdx.y;
    if (r >= side || c >= side) return;
    const int k = k0 + blockIdx.z;
    const float2 *slot = k == 0 ? slot0 : slots + (int64_t)(k - 1) * slot_elems;
    const float2 v = slot ? slot[(int64_t)r * pitch + c] : make_float2(0.f, 0.f);
    float *o = out + (int64_t)blockIdx.z * 2 * side * side;
    o[(int64_t)r * side + c] = v.x;
    o[(int64_t)side * side + (int64_t)r * side + c] = v.y;
}

// planes (2 x n x n) -> slot grid (n x n float2 with pitch)
__global__ void k_planes_to_slot(const float *__restrict__ in, int n, float2 *__restrict__ slot, int pitch)
{
    int c = blockIdx.x * blockDim.x + threadIdx.x, r = blockIdx.y * blockDim.y + threadIdx.y;
    if (r >= n || c >= n) return;
    slot[(int64_t)r * pitch + c] = make_float2(in[(int64_t)r * n + c], in[(int64_t)n * n + (int64_t)r * n + c]);
}

// Host launch wrappers for the templated kernels.
// few: the form for few tiles.
void launch_grad(int bf16, bool few, int grid, cudaStream_t st, const BatchDev &b)
{
    if (few) {
        if (bf16) k_grad<true, true><<<grid, REG_STRIP_THREADS, 0, st>>>(b);
        else k_grad<false, true><<<grid, REG_STRIP_THREADS, 0, st>>>(b);
    } else {
        if (bf16) k_grad<true, false><<<grid, REG_STRIP_THREADS, 0, st>>>(b);
        else k_grad<false, false><<<grid, REG_STRIP_THREADS, 0, st>>>(b);
    }
}

template <int JM>
static void launch_trial_j(int bf16, int grid, cudaStream_t st, const BatchDev &b)
{
    if (bf16) k_trial<true, JM><<<grid, REG_STRIP_THREADS, 0, st>>>(b);
    else k_trial<false, JM><<<grid, REG_STRIP_THREADS, 0, st>>>(b);
}

// J = trials per pass; the kernel instance holds room for the next power of two.
void launch_trial(int bf16, int J, int grid, cudaStream_t st, const BatchDev &b)
{
    if (J <= 1) launch_trial_j<1>(bf16, grid, st, b);
    else if (J <= 2) launch_trial_j<2>(bf16, grid, st, b);
    else if (J <= 4) launch_trial_j<4>(bf16, grid, st, b);
    else launch_trial_j<8>(bf16, grid, st, b);
}

// Resident blocks per SM of the step kernels.  Each asks for the smallest
// shared-memory carveout that still holds its register-limited number of
// blocks, which leaves the rest of the on-chip memory to L1 (the template
// gathers).
template <class K>
static int occupancy(K kernel, int threads, int carveout)
{
    int occ = 0;
    if (carveout < 0) {
        cudaFuncAttributes fa;
        int dev = 0, max_smem = 0, regs_sm = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
        cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev);
        cudaFuncGetAttributes(&fa, kernel);
        const int by_regs = fa.numRegs > 0 ? regs_sm / (fa.numRegs * threads) : 1;
        const size_t need = (size_t)by_regs * (fa.sharedSizeBytes + 1024);  // 1 KB reserved per block
        carveout = max_smem > 0 ? (int)std::min<size_t>(100, (need * 100 + max_smem - 1) / max_smem) : 100;
    }
    cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, carveout);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, threads, 0);
    return occ;
}

int step_blocks_per_sm(int which, int J)
{
    int occ = 0;
    if (which == 1) {
        occupancy(k_grad<true, false>, REG_STRIP_THREADS, 0);
        occ = occupancy(k_grad<false, false>, REG_STRIP_THREADS, 0);
    } else if (which == 0) {
        occupancy(k_grad<true, true>, REG_STRIP_THREADS, -1);
        occ = occupancy(k_grad<false, true>, REG_STRIP_THREADS, -1);
    } else {
        if (J <= 1) { occupancy(k_trial<true, 1>, REG_STRIP_THREADS, -1); occ = occupancy(k_trial<false, 1>, REG_STRIP_THREADS, -1); }
        else if (J <= 2) { occupancy(k_trial<true, 2>, REG_STRIP_THREADS, -1); occ = occupancy(k_trial<false, 2>, REG_STRIP_THREADS, -1); }
        else if (J <= 4) { occupancy(k_trial<true, 4>, REG_STRIP_THREADS, -1); occ = occupancy(k_trial<false, 4>, REG_STRIP_THREADS, -1); }
        else { occupancy(k_trial<true, 8>, REG_STRIP_THREADS, -1); occ = occupancy(k_trial<false, 8>, REG_STRIP_THREADS, -1); }
    }
    cudaGetLastError();
    return occ;
}
