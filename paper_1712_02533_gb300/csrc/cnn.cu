// The learned initialiser: a small convolutional network that predicts a coarse
// initial displacement for a frame pair, trained on the GPU on displacements
// that the plain method computes (its forward, backward and update kernels).
//
// Network: input 2 x S x S (reference, template; normalised), six 3x3
// convolutions with zero padding 1 -- 2->32 stride 2, 32->32 stride 2, three
// 32->32 stride 1, 32->2 stride 1 -- with a ReLU after every layer but the
// last; output 2 x S/4 x S/4, the displacement in input pixels at input pixels
// (4i, 4j).  Loss: mean squared difference to a target displacement.
// Parameters: one flat float vector, layer by layer W (O x C x 3 x 3) then b.
//
// Layout: the FP32 path keeps activations NCHW in float, one buffer per layer,
// on the CUDA cores.  The tensor-core path runs with BF16 operands and FP32
// accumulation: the forward of all six layers and the data and weight
// gradients of the four 32 -> 32 layers on tcgen05 with TMEM accumulators;
// the outputs of layers 0..4 are then BF16 in a channel-group planar layout
// [b][c / 8][y][x][c % 8], the operand layout of those kernels.  The remaining
// gradients (the first and last layers' weights, whose few channels make them
// bandwidth work, and the last layer's data) run on the CUDA cores in FP32.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>

#include "../../include/reg.h"
#include "cnn_internal.h"

namespace {

constexpr int NL = 6;
struct LayerShape {
    int C, O, S;
};
constexpr LayerShape LAYERS[NL] = {{2, 32, 2}, {32, 32, 2}, {32, 32, 1}, {32, 32, 1}, {32, 32, 1}, {32, 2, 1}};

constexpr int64_t layer_params(int k) { return (int64_t)LAYERS[k].O * LAYERS[k].C * 9 + LAYERS[k].O; }
int64_t param_offset(int k)
{
    int64_t o = 0;
    for (int j = 0; j < k; j++) o += layer_params(j);
    return o;
}
int64_t total_params() { return param_offset(NL); }


// ---------------------------------------------------------------------------
// Last layer (32 -> 2, stride 1, no ReLU), forward: one thread per output pixel
// (b, y, x) computes both channels.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(128) k_conv_last(const float *__restrict__ in, int H, const float *__restrict__ theta,
                                                   float *__restrict__ out, int total)
{
    __shared__ float2 w[32 * 9];  // [c][tap], both output channels
    for (int i = threadIdx.x; i < 32 * 9; i += blockDim.x) w[i] = make_float2(theta[i], theta[32 * 9 + i]);
    const float b0 = theta[2 * 32 * 9], b1 = theta[2 * 32 * 9 + 1];
    __syncthreads();
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= total) return;
    const int x = p % H, y = (p / H) % H, b = p / (H * H);
    float acc0 = b0, acc1 = b1;
    for (int c = 0; c < 32; c++) {
        const float *src = in + ((int64_t)b * 32 + c) * H * H;
        float v[9];
#pragma unroll
        for (int dy = 0; dy < 3; dy++)
#pragma unroll
            for (int dx = 0; dx < 3; dx++) {
                const int iy = y + dy - 1, ix = x + dx - 1;
                v[dy * 3 + dx] = (iy >= 0 && iy < H && ix >= 0 && ix < H) ? src[iy * H + ix] : 0.f;
            }
        // per output channel the products are added in the order (c, tap)
#pragma unroll
        for (int k = 0; k < 9; k++) {
            const float2 wv = w[c * 9 + k];
            acc0 = fmaf(wv.x, v[k], acc0);
            acc1 = fmaf(wv.y, v[k], acc1);
        }
    }
    out[(((int64_t)b * 2) * H + y) * H + x] = acc0;
    out[(((int64_t)b * 2 + 1) * H + y) * H + x] = acc1;
}

// ---------------------------------------------------------------------------
// Last layer, data gradient: gx[b, c, iy, ix] = sum over (o, dy, dx) of W[o, c, dy, dx]
// gz[b, o, iy + 1 - dy, ix + 1 - dx], times the ReLU mask of the layer below (its
// output a > 0).  One thread per pixel, all 32 channels.
// MASK_PLANAR: a_below is BF16 in the planar layout of the tensor-core layers instead of
// FP32 NCHW.
// ---------------------------------------------------------------------------
template <bool MASK_PLANAR>
__global__ void __launch_bounds__(128) k_bwd_data_last(const float *__restrict__ gz, const float *__restrict__ theta,
                                                       const void *__restrict__ a_below, float *__restrict__ gx,
                                                       int H, int total)
{
    // weights as [o][tap][c], so that one vector load brings the weights of
    // several input channels for an output gradient value
    __shared__ __align__(16) float w[2 * 9 * 32];
    for (int i = threadIdx.x; i < 2 * 9 * 32; i += blockDim.x) {
        const int o = i / (32 * 9), r = i - o * (32 * 9), c = r / 9, k = r - c * 9;
        w[(o * 9 + k) * 32 + c] = theta[i];
    }
    __syncthreads();
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= total) return;
    const int ix = p % H, iy = (p / H) % H, b = p / (H * H);
    float acc[32];
#pragma unroll
    for (int c = 0; c < 32; c++) acc[c] = 0.f;
#pragma unroll
    for (int dy = 0; dy < 3; dy++) {
        const int oy = iy + 1 - dy;
        if (oy < 0 || oy >= H) continue;
#pragma unroll
        for (int dx = 0; dx < 3; dx++) {
            const int ox = ix + 1 - dx;
            if (ox < 0 || ox >= H) continue;
            for (int o = 0; o < 2; o++) {
                const float g = gz[(((int64_t)b * 2 + o) * H + oy) * H + ox];
                const float4 *wk = reinterpret_cast<const float4 *>(w + (o * 9 + dy * 3 + dx) * 32);
#pragma unroll
                for (int q = 0; q < 8; q++) {
                    const float4 wv = wk[q];
                    acc[4 * q] = fmaf(wv.x, g, acc[4 * q]);
                    acc[4 * q + 1] = fmaf(wv.y, g, acc[4 * q + 1]);
                    acc[4 * q + 2] = fmaf(wv.z, g, acc[4 * q + 2]);
                    acc[4 * q + 3] = fmaf(wv.w, g, acc[4 * q + 3]);
                }
            }
        }
    }
#pragma unroll
    for (int c = 0; c < 32; c++) {
        const int64_t i = (((int64_t)b * 32 + c) * H + iy) * H + ix;
        bool pos;
        if (MASK_PLANAR) {
            const uint16_t v = reinterpret_cast<const uint16_t *>(
                a_below)[(((int64_t)(4 * b + c / 8) * H + iy) * H + ix) * 8 + (c & 7)];
            pos = v != 0 && !(v & 0x8000u);
        } else {
            pos = reinterpret_cast<const float *>(a_below)[i] > 0.f;
        }
        gx[i] = pos ? acc[c] : 0.f;
    }
}

// ---------------------------------------------------------------------------
// The FP32 path's convolutions with 32 output channels, their data and weight
// gradients.  All are FP32 work of 288 multiply-adds per value moved, so what
// counts is how many multiply-adds follow a shared-memory load: with one pixel
// per thread and all 32 channels each 16-byte weight load fed four of them and
// the loads bounded the kernel (128 us per forward layer of 32 pairs, 64^2
// outputs; 136 us per data gradient).  Here a thread holds four pixels (one
// column of four rows: lanes stay on adjacent columns) by 16 channels, so that a
// weight load feeds 16 (packed in pairs).  Each output's products are added in
// the order they always were, so the results are bit for bit the same.  Forward
// layer 128 -> 74 us, data gradient 136 -> 92 us (stride 2: 222 -> 111 us).
// ---------------------------------------------------------------------------
constexpr int PX = 4, OC = 16;  // pixels and channels per thread

__device__ __forceinline__ void fma_group(float2 (&acc)[PX][OC / 2], const float *w, const float (&v)[PX])
{
#pragma unroll
    for (int q = 0; q < OC / 4; q++) {
        const float4 wv = reinterpret_cast<const float4 *>(w)[q];
        const float2 w0 = make_float2(wv.x, wv.y), w1 = make_float2(wv.z, wv.w);
#pragma unroll
        for (int p = 0; p < PX; p++) {
            const float2 vv = make_float2(v[p], v[p]);
            acc[p][2 * q] = __ffma2_rn(w0, vv, acc[p][2 * q]);
            acc[p][2 * q + 1] = __ffma2_rn(w1, vv, acc[p][2 * q + 1]);
        }
    }
}

// Forward, 32 outputs with ReLU: out[b][o][y][x], rows y = 4 yg .. 4 yg + 3.  grid
// (column-and-row-group blocks, channel halves).  Sum order (c, tap), as k_conv_last.
template <int C, int S>
__global__ void __launch_bounds__(128, 4) k_conv_fwd32(const float *__restrict__ in, int H,
                                                       const float *__restrict__ theta, float *__restrict__ out,
                                                       int Ho, int nyg, int total)
{
    constexpr int NR = S * (PX - 1) + 3;  // input rows of the four output rows
    __shared__ __align__(16) float w[C * 9 * OC];
    __shared__ float bias[OC];
    const int o0 = blockIdx.y * OC;
    for (int i = threadIdx.x; i < C * 9 * OC; i += blockDim.x) {
        const int o = i / (C * 9), ck = i - o * (C * 9);
        w[ck * OC + o] = theta[(o0 + o) * C * 9 + ck];
    }
    if (threadIdx.x < OC) bias[threadIdx.x] = theta[32 * C * 9 + o0 + threadIdx.x];
    __syncthreads();
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= total) return;
    const int x = p % Ho, yg = (p / Ho) % nyg, b = p / (Ho * nyg), y0 = yg * PX;
    float2 acc[PX][OC / 2];
#pragma unroll
    for (int k = 0; k < PX; k++)
#pragma unroll
        for (int o = 0; o < OC / 2; o++) acc[k][o] = make_float2(bias[2 * o], bias[2 * o + 1]);
    const float *src = in + (int64_t)b * C * H * H;
    const int ix0 = S * x - 1, iy0 = S * y0 - 1;
#pragma unroll 1
    for (int c = 0; c < C; c++, src += (int64_t)H * H) {
        float v[NR][3];
#pragma unroll
        for (int r = 0; r < NR; r++)
#pragma unroll
            for (int dx = 0; dx < 3; dx++) {
                const int iy = iy0 + r, ix = ix0 + dx;
                v[r][dx] = (iy >= 0 && iy < H && ix >= 0 && ix < H) ? src[iy * H + ix] : 0.f;
            }
#pragma unroll
        for (int k = 0; k < 9; k++) {
            float q[PX];
#pragma unroll
            for (int j = 0; j < PX; j++) q[j] = v[S * j + k / 3][k % 3];
            fma_group(acc, w + (c * 9 + k) * OC, q);
        }
    }
#pragma unroll
    for (int j = 0; j < PX; j++)
        if (y0 + j < Ho) {
#pragma unroll
            for (int o = 0; o < OC; o++) {
                const float a = (o & 1) ? acc[j][o / 2].y : acc[j][o / 2].x;
                out[(((int64_t)b * 32 + o0 + o) * Ho + y0 + j) * Ho + x] = fmaxf(a, 0.f);
            }
        }
}

// Data gradient of the 32 -> 32 layers with the ReLU mask of the layer below (its
// FP32 output > 0).  Stride 2: an input pixel takes the taps dy with iy + 1 - dy
// even, likewise along x, so the pixels of one parity class (blockIdx.z = 2 py +
// px) share their taps; a thread's rows and the lanes' columns are two apart.  Sum
// order (dy, dx, o), as k_bwd_data_last.
template <int S>
__global__ void __launch_bounds__(128, 4) k_conv_bwd_data32(const float *__restrict__ gz, int Ho,
                                                            const float *__restrict__ theta,
                                                            const float *__restrict__ a_below, float *__restrict__ gx,
                                                            int H, int nyg, int total)
{
    __shared__ __align__(16) float w[32 * 9 * OC];  // [o][tap][c of this half]
    const int c0 = blockIdx.y * OC, py = S == 2 ? blockIdx.z >> 1 : 0, px = S == 2 ? blockIdx.z & 1 : 0;
    for (int i = threadIdx.x; i < 32 * 9 * OC; i += blockDim.x) {
        const int o = i / (9 * OC), r = i - o * (9 * OC), c = r / 9, k = r - c * 9;
        w[(o * 9 + k) * OC + c] = theta[(o * 32 + c0 + c) * 9 + k];
    }
    __syncthreads();
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= total) return;
    const int nx = H / S;
    const int xi = p % nx, yg = (p / nx) % nyg, b = p / (nx * nyg), y0 = yg * PX;  // in class rows and columns
    const int ix = S * xi + px;
    float2 acc[PX][OC / 2];
#pragma unroll
    for (int k = 0; k < PX; k++)
#pragma unroll
        for (int o = 0; o < OC / 2; o++) acc[k][o] = make_float2(0.f, 0.f);
    const int64_t plane = (int64_t)Ho * Ho;
    const float *gb = gz + (int64_t)b * 32 * plane;
#pragma unroll 1
    for (int dy = 0; dy < 3; dy++) {
        if (S == 2 && ((py + 1 - dy) & 1)) continue;  // block-uniform
        int off[PX];
        bool okr[PX];
#pragma unroll
        for (int j = 0; j < PX; j++) {
            const int ty = S * (y0 + j) + py + 1 - dy, oy = S == 2 ? ty >> 1 : ty;
            okr[j] = ty >= 0 && oy < Ho && y0 + j < nx;
            off[j] = oy * Ho;
        }
#pragma unroll 1
        for (int dx = 0; dx < 3; dx++) {
            if (S == 2 && ((px + 1 - dx) & 1)) continue;  // block-uniform
            const int tx = ix + 1 - dx, ox = S == 2 ? tx >> 1 : tx;
            const bool okc = tx >= 0 && ox < Ho;
            const float *g0 = gb + ox;
            const float *wk = w + (dy * 3 + dx) * OC;
#pragma unroll 4
            for (int o = 0; o < 32; o++) {
                float g[PX];
#pragma unroll
                for (int j = 0; j < PX; j++) g[j] = okc && okr[j] ? g0[o * plane + off[j]] : 0.f;
                fma_group(acc, wk + o * 9 * OC, g);
            }
        }
    }
#pragma unroll
    for (int j = 0; j < PX; j++) {
        const int iy = S * (y0 + j) + py;
        if (y0 + j < nx) {
#pragma unroll
            for (int c = 0; c < OC; c++) {
                const int64_t i = (((int64_t)b * 32 + c0 + c) * H + iy) * H + ix;
                const float a = (c & 1) ? acc[j][c / 2].y : acc[j][c / 2].x;
                gx[i] = a_below[i] > 0.f ? a : 0.f;
            }
        }
    }
}

// Weight and bias gradients of the 32 -> 32 layers: gW[o][c][tap] = sum gz[b][o][y][x]
// in[b][c][S y + dy - 1][S x + dx - 1].  A block stages a tile of output pixels
// (the gradient as [pixel][o], the input window as [c][row][column]) and its
// threads (warp = 4 output channels, lane = input channel) sum 4 x 9 products per
// pixel over a window sliding along the row: one broadcast 16-byte load and 3 S
// conflict-free loads per 36 multiply-adds.  The products are added in runs of WG32_RUN
// pixels and the runs' sums then: in one chain over a tile's pixels the error of a
// weight of one pair of 256^2 was 1.6 times that of 256 strided sums and a tree, in
// runs it is 0.83 times that.  With a block per (o, c) pair, which
// read input and gradient 32 times over from L2, a layer took 1155 us (32 pairs);
// now 69 us (66 in one chain) and 4 us for the records' sum.
// Blocks take tiles block, block + grid, ..; each writes one record.
constexpr int WG32_RUN = 16;
template <int S>
struct Wg32 {
    static constexpr int TR = 4, TC = S == 1 ? 32 : 16, NP = TR * TC;
    static constexpr int IR = S * (TR - 1) + 3, IC = S * (TC - 1) + 3;
    static constexpr int CS = (IR * IC) | 1;  // odd channel stride: no bank conflicts across channels
    static constexpr int GS = 36;             // gradient row: 32 channels, 16-byte aligned
};
constexpr int WG32_REC = 32 * 32 * 9 + 32;
constexpr int WG32_BLOCKS = 2;  // per SM

template <int S>
__global__ void __launch_bounds__(256, WG32_BLOCKS) k_wgrad32(const float *__restrict__ in, int H,
                                                              const float *__restrict__ gz, int Ho, int B,
                                                              float *__restrict__ part)
{
    using G = Wg32<S>;
    __shared__ __align__(16) float gs[G::NP * G::GS];
    __shared__ float is[32 * G::CS];
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    float2 tot[2][9];
    float gb[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
        for (int j = 0; j < 9; j++) tot[i][j] = make_float2(0.f, 0.f);
    static_assert(G::TC % WG32_RUN == 0, "whole runs");
    const int tx_n = (Ho + G::TC - 1) / G::TC, ty_n = (Ho + G::TR - 1) / G::TR, nt = B * tx_n * ty_n;
    for (int tile = blockIdx.x; tile < nt; tile += gridDim.x) {
        const int b = tile / (tx_n * ty_n), rr = tile % (tx_n * ty_n);
        const int y0 = (rr / tx_n) * G::TR, x0 = (rr % tx_n) * G::TC;
        __syncthreads();  // the previous tile's reads are done
        // gradient: warp w its own channels 4 w .. 4 w + 3 (bias sums from the registers)
        float gv[4][G::NP / 32];
#pragma unroll
        for (int q = 0; q < 4; q++)
#pragma unroll
            for (int j = 0; j < G::NP / 32; j++) {
                const int p = 32 * j + lane, y = y0 + p / G::TC, x = x0 + p % G::TC;
                gv[q][j] = (y < Ho && x < Ho) ? gz[(((int64_t)b * 32 + 4 * wid + q) * Ho + y) * Ho + x] : 0.f;
            }
        // input window: warp w channels w, w + 8, ..
        constexpr int NI = (G::IR * G::IC + 31) / 32;
#pragma unroll 1
        for (int k = 0; k < 4; k++) {
            const int c = wid + 8 * k;
            const float *src = in + ((int64_t)b * 32 + c) * H * H;
            float iv[NI];
#pragma unroll
            for (int j = 0; j < NI; j++) {
                const int i = 32 * j + lane, iy = S * y0 - 1 + i / G::IC, ix = S * x0 - 1 + i % G::IC;
                iv[j] = (i < G::IR * G::IC && iy >= 0 && iy < H && ix >= 0 && ix < H) ? src[iy * H + ix] : 0.f;
            }
#pragma unroll
            for (int j = 0; j < NI; j++)
                if (32 * j + lane < G::IR * G::IC) is[c * G::CS + 32 * j + lane] = iv[j];
        }
#pragma unroll
        for (int j = 0; j < G::NP / 32; j++) {
            *reinterpret_cast<float4 *>(gs + (32 * j + lane) * G::GS + 4 * wid) =
                make_float4(gv[0][j], gv[1][j], gv[2][j], gv[3][j]);
#pragma unroll
            for (int q = 0; q < 4; q++) gb[q] += gv[q][j];
        }
        __syncthreads();
        const float *ic = is + lane * G::CS;
#pragma unroll 1
        for (int r = 0; r < G::TR; r++) {
            float win[3][3];
#pragma unroll
            for (int dy = 0; dy < 3; dy++)
#pragma unroll
                for (int dx = 0; dx < 3 - S; dx++) win[dy][S + dx] = ic[(S * r + dy) * G::IC + dx];
#pragma unroll 1
            for (int xr = 0; xr < G::TC; xr += WG32_RUN) {
                float2 acc[2][9];
#pragma unroll
                for (int i = 0; i < 2; i++)
#pragma unroll
                    for (int j = 0; j < 9; j++) acc[i][j] = make_float2(0.f, 0.f);
#pragma unroll 4
                for (int x = xr; x < xr + WG32_RUN; x++) {
#pragma unroll
                    for (int dy = 0; dy < 3; dy++) {
#pragma unroll
                        for (int dx = 0; dx < 3 - S; dx++) win[dy][dx] = win[dy][S + dx];
#pragma unroll
                        for (int dx = 3 - S; dx < 3; dx++) win[dy][dx] = ic[(S * r + dy) * G::IC + S * x + dx];
                    }
                    const float4 g = *reinterpret_cast<const float4 *>(gs + (r * G::TC + x) * G::GS + 4 * wid);
                    const float2 g0 = make_float2(g.x, g.y), g1 = make_float2(g.z, g.w);
#pragma unroll
                    for (int j = 0; j < 9; j++) {
                        const float2 v = make_float2(win[j / 3][j % 3], win[j / 3][j % 3]);
                        acc[0][j] = __ffma2_rn(g0, v, acc[0][j]);
                        acc[1][j] = __ffma2_rn(g1, v, acc[1][j]);
                    }
                }
#pragma unroll
                for (int i = 0; i < 2; i++)
#pragma unroll
                    for (int j = 0; j < 9; j++) tot[i][j] = __fadd2_rn(tot[i][j], acc[i][j]);
            }
        }
    }
    float *rec = part + (int64_t)blockIdx.x * WG32_REC;
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
        for (int j = 0; j < 9; j++) {
            rec[((4 * wid + 2 * i) * 32 + lane) * 9 + j] = tot[i][j].x;
            rec[((4 * wid + 2 * i + 1) * 32 + lane) * 9 + j] = tot[i][j].y;
        }
#pragma unroll
    for (int q = 0; q < 4; q++) {
        float v = gb[q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) rec[32 * 32 * 9 + 4 * wid + q] = v;
    }
}

// ---------------------------------------------------------------------------
// Weight gradients of the 2 -> 32 (stride 2) and 32 -> 2 layers.  Their
// arithmetic intensity is a few FLOPs per byte (two input channels, or two
// output channels), so they stay on the CUDA cores in FP32, but each input
// element is read from global memory once: a block stages a tile of the output
// gradient and the input window the tile needs, and its threads form all the
// layer's weight and bias sums from shared memory.  Each block works through a
// fixed sequence of tiles (tile = block + k grid) and writes one partial
// record; cnn_sum_records adds the records in a fixed order, so the result is
// deterministic for a given grid.
// ---------------------------------------------------------------------------
// Asynchronous copies to shared memory, zeros where !in (src then any valid address).
__device__ __forceinline__ void cp_async16(float *dst, const float *src, bool in)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(in ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_async4(float *dst, const float *src, bool in)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(in ? 4 : 0)
                 : "memory");
}

constexpr int WF_TR = 2, WF_TW = 64, WF_NP = WF_TR * WF_TW;  // first layer: 2 output rows x 64 columns
constexpr int WF_XR = 2 * WF_TR + 1, WF_XC = 2 * WF_TW + 1;  // its input window: 5 x 129
constexpr int WF_XS = WF_XC + 1;                              // row stride of the staged window (pixels)
constexpr int WF_GS = WF_NP + 4;                              // row stride of the staged gradient: 16-byte
                                                              // reads of 8 lanes' rows touch 32 banks
constexpr int WF_REC = 32 * 2 * 9 + 32;                       // weights (o, c, tap), then biases

// First layer: gW[o][c][dy][dx] = sum gz[b][o][y][x] x[b][c][2 y + dy - 1][2 x + dx - 1],
// gb[o] = sum gz[b][o][y][x]; x FP32 NCHW (B x 2 x H x H), gz FP32 NCHW (B x
// 32 x Ho x Ho).  Lane o of warp w sums output channel o over 16 pixels of tile
// row w / 4, from column 16 (w % 4): the gradient of four pixels in one shared
// read, the window's pixels as (channel 0, channel 1) pairs broadcast to the warp,
// so that a pixel is nine packed products and four shared reads; even and odd
// pixels go to two sets of sums, added to the totals tile by tile (one chain over a
// block's tiles had 1.1 times the error of the shorter chains before it at 32 pairs, now
// 0.7).  The next tile's copies (cp.async, the gradient;
// registers, the window) run under this tile's sums.
// It reads each byte once (84 MB at 32 x 256^2, 12.4 us at the copy rate).  With
// threads over (4 output channels, pixel), the channels' 19 scalar reads a pixel
// and the copies waited for before each tile's sums it took 51.3 us; now 28.9 us (27.6
// without the totals).
__global__ void __launch_bounds__(256, 2) k_wgrad_first(const float *__restrict__ x, int H,
                                                     const float *__restrict__ gz, int Ho, int B,
                                                     float *__restrict__ part)
{
    // [o][pixel] per buffer; after the last tile the warps' sums
    __shared__ __align__(16) float gs[2][32 * WF_GS];
    // window column c at index c + 1: the columns 2 px + 1, 2 px + 2 of a pixel in one read
    __shared__ __align__(16) float2 xs[WF_XR][WF_XS];
    constexpr int NX = (WF_XR * WF_XC + 255) / 256, NJ = 19;
    static_assert(2 * 32 * WF_GS >= 8 * 32 * NJ, "the warps' sums take the gradient's place");
    const int t = threadIdx.x, lane = t & 31, w = t >> 5, py = w >> 2, px0 = 16 * (w & 3);
    const int tx_n = (Ho + WF_TW - 1) / WF_TW, ty_n = (Ho + WF_TR - 1) / WF_TR, nt = B * tx_n * ty_n;
    const bool vec = Ho % 4 == 0;  // rows 16-byte aligned (gz itself is an allocation)
    float2 xv[NX];
    auto load = [&](int tile, int buf) {
        const int b = tile / (tx_n * ty_n), r = tile % (tx_n * ty_n);
        const int y0 = (r / tx_n) * WF_TR, x0 = (r % tx_n) * WF_TW;
        const float *g0 = gz + (int64_t)b * 32 * Ho * Ho;
        if (vec) {
#pragma unroll
            for (int k = 0; k < 32 * WF_NP / 4 / 256; k++) {
                const int i = t + 256 * k, o = i / (WF_NP / 4), p = 4 * (i % (WF_NP / 4));
                const int y = y0 + p / WF_TW, xx = x0 + p % WF_TW;
                const bool in = y < Ho && xx < Ho;
                cp_async16(&gs[buf][o * WF_GS + p], g0 + (in ? ((int64_t)o * Ho + y) * Ho + xx : 0), in);
            }
        } else {
#pragma unroll 4
            for (int k = 0; k < 32 * WF_NP / 256; k++) {
                const int i = t + 256 * k, o = i / WF_NP, p = i % WF_NP;
                const int y = y0 + p / WF_TW, xx = x0 + p % WF_TW;
                const bool in = y < Ho && xx < Ho;
                cp_async4(&gs[buf][o * WF_GS + p], g0 + (in ? ((int64_t)o * Ho + y) * Ho + xx : 0), in);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        const float *x0p = x + (int64_t)b * 2 * H * H;
#pragma unroll
        for (int k = 0; k < NX; k++) {
            const int i = t + 256 * k, iy = 2 * y0 - 1 + i / WF_XC, ix = 2 * x0 - 1 + i % WF_XC;
            const bool in = i < WF_XR * WF_XC && iy >= 0 && iy < H && ix >= 0 && ix < H;
            const float *p = x0p + (int64_t)iy * H + ix;
            xv[k] = in ? make_float2(p[0], p[(int64_t)H * H]) : make_float2(0.f, 0.f);
        }
    };
    float2 tot[9];
    float gbt = 0.f;
#pragma unroll
    for (int j = 0; j < 9; j++) tot[j] = make_float2(0.f, 0.f);
    int buf = 0;
    if ((int)blockIdx.x < nt) load(blockIdx.x, 0);
    for (int tile = blockIdx.x; tile < nt; tile += gridDim.x, buf ^= 1) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();  // the previous tile's reads are done, this tile's gradient is there
#pragma unroll
        for (int k = 0; k < NX; k++) {
            const int i = t + 256 * k;
            if (i < WF_XR * WF_XC) xs[i / WF_XC][i % WF_XC + 1] = xv[k];
        }
        __syncthreads();
        if (tile + (int)gridDim.x < nt) load(tile + gridDim.x, buf ^ 1);
        float2 acc[2][9];  // this tile's
        float gb[2] = {0.f, 0.f};
#pragma unroll
        for (int i = 0; i < 2; i++)
#pragma unroll
            for (int j = 0; j < 9; j++) acc[i][j] = make_float2(0.f, 0.f);
        float2 win[3];  // the window column left of the next two
#pragma unroll
        for (int dy = 0; dy < 3; dy++) win[dy] = xs[2 * py + dy][2 * px0 + 1];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const float4 g4 = *reinterpret_cast<const float4 *>(&gs[buf][lane * WF_GS + py * WF_TW + px0 + 4 * q]);
            const float g[4] = {g4.x, g4.y, g4.z, g4.w};
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const float2 gg = make_float2(g[i], g[i]);
                gb[i & 1] += g[i];
#pragma unroll
                for (int dy = 0; dy < 3; dy++) {
                    const float4 n = *reinterpret_cast<const float4 *>(&xs[2 * py + dy][2 * (px0 + 4 * q + i) + 2]);
                    const float2 n1 = make_float2(n.x, n.y), n2 = make_float2(n.z, n.w);
                    acc[i & 1][dy * 3] = __ffma2_rn(gg, win[dy], acc[i & 1][dy * 3]);
                    acc[i & 1][dy * 3 + 1] = __ffma2_rn(gg, n1, acc[i & 1][dy * 3 + 1]);
                    acc[i & 1][dy * 3 + 2] = __ffma2_rn(gg, n2, acc[i & 1][dy * 3 + 2]);
                    win[dy] = n2;
                }
            }
        }
#pragma unroll
        for (int j = 0; j < 9; j++) tot[j] = __fadd2_rn(tot[j], __fadd2_rn(acc[0][j], acc[1][j]));
        gbt += gb[0] + gb[1];
    }
    __syncthreads();
    float *red = &gs[0][0] + (w * 32 + lane) * NJ;
#pragma unroll
    for (int j = 0; j < 9; j++) {
        red[j] = tot[j].x;
        red[9 + j] = tot[j].y;
    }
    red[18] = gbt;
    __syncthreads();
    for (int e = t; e < WF_REC; e += 256) {
        // weights (o, c, tap) at (2 o + c) 9 + tap, then the biases
        const int o = e < 576 ? e / 18 : e - 576, j = e < 576 ? e % 18 : 18;
        float sum = 0.f;
        for (int w2 = 0; w2 < 8; w2++) sum += gs[0][(w2 * 32 + o) * NJ + j];
        part[(int64_t)blockIdx.x * WF_REC + e] = sum;
    }
}

constexpr int WL_TR = 4, WL_TW = 32, WL_NP = WL_TR * WL_TW;  // last layer: 4 output rows x 32 columns
constexpr int WL_AR = WL_TR + 2, WL_AC = WL_TW + 2;          // its input window: 6 x 34
constexpr int WL_CS = WL_AR * WL_AC + 1;                     // channel stride (odd: no bank conflicts)
constexpr int WL_REC = 2 * 32 * 9 + 2;

// Last layer: gW[o][c][dy][dx] = sum gz[b][o][y][x] a[b][c][y + dy - 1][x + dx - 1],
// gb[o] = sum gz[b][o][y][x]; a the input (B x 32 x H x H), BF16 in the planar
// layout or FP32 NCHW, gz FP32 NCHW (B x 2 x H x H).  Thread (c, seg) = (t % 32, t / 32) walks 16 pixels of
// tile row seg / 2 with a sliding 3 x 3 window of channel c; a tile's sums are added to
// the totals (one chain over a block's tiles: 1.1 times the error of the strided sums and
// trees of the FP32 pass before it at 128 pairs, now 0.6).
template <bool PLANAR>
__global__ void __launch_bounds__(256) k_wgrad_last(const void *__restrict__ act, int H, const float *__restrict__ gz,
                                                    int B, float *__restrict__ part)
{
    const uint4 *a = reinterpret_cast<const uint4 *>(act);
    __shared__ float as[32 * WL_CS];
    __shared__ float gs[2][WL_NP];
    __shared__ float red[8][32][18];
    __shared__ float redb[8][2];
    const int t = threadIdx.x, c = t & 31, seg = t >> 5, r = seg >> 1, xs0 = (seg & 1) * 16;
    float tot[18], gt0 = 0.f, gt1 = 0.f;
#pragma unroll
    for (int j = 0; j < 18; j++) tot[j] = 0.f;
    const int tx_n = (H + WL_TW - 1) / WL_TW, ty_n = (H + WL_TR - 1) / WL_TR, nt = B * tx_n * ty_n;
    for (int tile = blockIdx.x; tile < nt; tile += gridDim.x) {
        const int b = tile / (tx_n * ty_n), rr0 = tile % (tx_n * ty_n);
        const int y0 = (rr0 / tx_n) * WL_TR, x0 = (rr0 % tx_n) * WL_TW;
        __syncthreads();
        // all of a thread's loads are issued before its stores
        constexpr int NA = (4 * WL_AR * WL_AC + 255) / 256;
        float g;
        uint4 qa[PLANAR ? NA : 1];
        {
            static_assert(2 * WL_NP == 256, "one gradient value per thread");
            const int o = t / WL_NP, p = t % WL_NP, y = y0 + p / WL_TW, xx = x0 + p % WL_TW;
            g = (y < H && xx < H) ? gz[(((int64_t)b * 2 + o) * H + y) * H + xx] : 0.f;
        }
        if constexpr (PLANAR) {
#pragma unroll
            for (int k = 0; k < NA; k++) {
                const int i = t + 256 * k, cg = i / (WL_AR * WL_AC), rr = (i / WL_AC) % WL_AR, cc = i % WL_AC;
                const int iy = y0 - 1 + rr, ix = x0 - 1 + cc;
                qa[k] = make_uint4(0u, 0u, 0u, 0u);
                if (i < 4 * WL_AR * WL_AC && iy >= 0 && iy < H && ix >= 0 && ix < H)
                    qa[k] = a[((int64_t)(4 * b + cg) * H + iy) * H + ix];
            }
        } else {
            // warp w channels w, w + 8, ..: lanes on adjacent columns
            constexpr int NW = (WL_AR * WL_AC + 31) / 32;
#pragma unroll
            for (int k = 0; k < 4; k++) {
                const int ch = (t >> 5) + 8 * k;
                const float *src = reinterpret_cast<const float *>(act) + ((int64_t)b * 32 + ch) * H * H;
                float v[NW];
#pragma unroll
                for (int j = 0; j < NW; j++) {
                    const int i = 32 * j + (t & 31), iy = y0 - 1 + i / WL_AC, ix = x0 - 1 + i % WL_AC;
                    v[j] = (i < WL_AR * WL_AC && iy >= 0 && iy < H && ix >= 0 && ix < H) ? src[iy * H + ix] : 0.f;
                }
#pragma unroll
                for (int j = 0; j < NW; j++)
                    if (32 * j + (t & 31) < WL_AR * WL_AC) as[ch * WL_CS + 32 * j + (t & 31)] = v[j];
            }
        }
        (&gs[0][0])[t] = g;
#pragma unroll
        for (int k = 0; k < (PLANAR ? NA : 0); k++) {
            const int i = t + 256 * k, cg = i / (WL_AR * WL_AC), rr = (i / WL_AC) % WL_AR, cc = i % WL_AC;
            if (i >= 4 * WL_AR * WL_AC) continue;
            const uint32_t wv[4] = {qa[k].x, qa[k].y, qa[k].z, qa[k].w};
            float *dst = as + (8 * cg) * WL_CS + rr * WL_AC + cc;
#pragma unroll
            for (int j = 0; j < 4; j++) {
                dst[(2 * j) * WL_CS] = __uint_as_float(wv[j] << 16);
                dst[(2 * j + 1) * WL_CS] = __uint_as_float(wv[j] & 0xFFFF0000u);
            }
        }
        __syncthreads();
        float acc[18], gb0 = 0.f, gb1 = 0.f;  // this tile's
#pragma unroll
        for (int j = 0; j < 18; j++) acc[j] = 0.f;
        const float *ac = as + c * WL_CS + r * WL_AC + xs0;
        float win[3][3];
#pragma unroll
        for (int dy = 0; dy < 3; dy++) {
            win[dy][0] = ac[dy * WL_AC];
            win[dy][1] = ac[dy * WL_AC + 1];
        }
#pragma unroll 4
        for (int px = 0; px < 16; px++) {
#pragma unroll
            for (int dy = 0; dy < 3; dy++) win[dy][2] = ac[dy * WL_AC + px + 2];
            const int p = r * WL_TW + xs0 + px;
            const float g0 = gs[0][p], g1 = gs[1][p];
#pragma unroll
            for (int dy = 0; dy < 3; dy++)
#pragma unroll
                for (int dx = 0; dx < 3; dx++) {
                    acc[dy * 3 + dx] = fmaf(g0, win[dy][dx], acc[dy * 3 + dx]);
                    acc[9 + dy * 3 + dx] = fmaf(g1, win[dy][dx], acc[9 + dy * 3 + dx]);
                }
            gb0 += g0;
            gb1 += g1;
#pragma unroll
            for (int dy = 0; dy < 3; dy++) {
                win[dy][0] = win[dy][1];
                win[dy][1] = win[dy][2];
            }
        }
#pragma unroll
        for (int j = 0; j < 18; j++) tot[j] += acc[j];
        gt0 += gb0;
        gt1 += gb1;
    }
#pragma unroll
    for (int j = 0; j < 18; j++) red[seg][c][j] = tot[j];
    if (c == 0) {
        redb[seg][0] = gt0;
        redb[seg][1] = gt1;
    }
    __syncthreads();
    for (int e = t; e < WL_REC; e += 256) {
        // weights (o, c, tap) at (32 o + c) 9 + tap, then the biases
        float sum = 0.f;
        if (e < 576) {
            const int o = e / 288, cc = (e % 288) / 9, tap = e % 9;
            for (int w2 = 0; w2 < 8; w2++) sum += red[w2][cc][o * 9 + tap];
        } else {
            for (int w2 = 0; w2 < 8; w2++) sum += redb[w2][e - 576];
        }
        part[(int64_t)blockIdx.x * WL_REC + e] = sum;
    }
}

// Grid of the weight gradient kernels: two blocks per SM, at most one per tile.
int wgrad_small_grid(int n_tiles)
{
    int dev = 0, nsm = 152;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        nsm = 152;
    return std::max(1, std::min(n_tiles, 2 * nsm));
}

// Floats of a layer's partial records (one per block, at most two blocks per SM), and
// of all layers: the records stay until one launch adds them all.
size_t wpart_floats(int k)
{
    const size_t rec = k == 0 ? WF_REC : k == NL - 1 ? WL_REC : WG32_REC, n = wgrad_small_grid(1 << 30) * rec;
    return k == 0 || k == NL - 1 ? n : std::max(n, (size_t)cnn_wgrad32_umma_part_floats());
}

size_t wpart_offset(int k)
{
    size_t n = 0;
    for (int j = 0; j < k; j++) n += wpart_floats(j);
    return n;
}

// Mean squared error: per-block partial sums (double), then one block adds them
// in order; gy = 2 (y - t) / N.
__global__ void k_mse(const float *__restrict__ y, const float *__restrict__ t, int64_t n, float *__restrict__ gy,
                      double *__restrict__ partial)
{
    double s = 0.0;
    const float inv = 2.f / (float)n;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float d = y[i] - t[i];
        s += (double)d * d;
        gy[i] = inv * d;
    }
    __shared__ double red[8];
    for (int k = 16; k > 0; k >>= 1) s += __shfl_xor_sync(0xffffffffu, s, k);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) tot += red[w];
        partial[blockIdx.x] = tot;
    }
}

__global__ void __launch_bounds__(256) k_sum_partials(const double *partial, int n, double scale, double *out)
{
    // fixed order: thread t adds entries t, t + 256, ...; then the warps' sums
    // by shuffles and the eight warp totals in order
    __shared__ double red[8];
    const int t = threadIdx.x;
    double s = 0.0;
    for (int i = t; i < n; i += 256) s += partial[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((t & 31) == 0) red[t >> 5] = s;
    __syncthreads();
    if (t == 0) {
        double tot = 0.0;
        for (int w = 0; w < 8; w++) tot += red[w];
        *out = tot * scale;
    }
}

// Adam with bias correction (step t >= 1).
__global__ void k_adam(float *__restrict__ theta, const float *__restrict__ g, float *__restrict__ m,
                       float *__restrict__ v, int64_t n, float lr, float b1, float b2, float eps, float c1, float c2)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        theta[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

// FP32 forward of layer k.
void fwd(int k, const float *in, int H, const float *theta, float *out, int B, cudaStream_t st)
{
    const int Ho = (H + 2 - 3) / LAYERS[k].S + 1;
    if (k == NL - 1) {
        const int total = B * Ho * Ho;
        k_conv_last<<<(total + 127) / 128, 128, 0, st>>>(in, H, theta, out, total);
        return;
    }
    const int nyg = (Ho + PX - 1) / PX, total = B * nyg * Ho;
    const dim3 grid((total + 127) / 128, 32 / OC);
    if (k == 0) k_conv_fwd32<2, 2><<<grid, 128, 0, st>>>(in, H, theta, out, Ho, nyg, total);
    else if (LAYERS[k].S == 2) k_conv_fwd32<32, 2><<<grid, 128, 0, st>>>(in, H, theta, out, Ho, nyg, total);
    else k_conv_fwd32<32, 1><<<grid, 128, 0, st>>>(in, H, theta, out, Ho, nyg, total);
}

// FP32 weight gradient of layer k (records to part, entered in sums for grad) and, for k > 0, its data gradient with
// the ReLU mask of the layer below into gx.
void bwd(int k, const float *in, int H, const float *gz, const float *theta, float *gx, float *grad, int B,
         cudaStream_t st, float *part, CnnSumList &sums)
{
    const int Ho = (H + 2 - 3) / LAYERS[k].S + 1;
    auto tiles = [&](int tr, int tc) { return B * ((Ho + tr - 1) / tr) * ((Ho + tc - 1) / tc); };
    if (k == 0) {
        const int grid = wgrad_small_grid(tiles(WF_TR, WF_TW));
        k_wgrad_first<<<grid, 256, 0, st>>>(in, H, gz, Ho, B, part);
        sums.add(part, grid, WF_REC, grad, false);
        return;
    }
    if (k == NL - 1) {
        const int grid = wgrad_small_grid(tiles(WL_TR, WL_TW)), total = B * H * H;
        k_wgrad_last<false><<<grid, 256, 0, st>>>(in, H, gz, B, part);
        sums.add(part, grid, WL_REC, grad, false);
        k_bwd_data_last<false><<<(total + 127) / 128, 128, 0, st>>>(gz, theta, in, gx, H, total);
        return;
    }
    const int S = LAYERS[k].S, nx = H / S, nyg = (nx + PX - 1) / PX, total = B * nyg * nx;
    const dim3 grid((total + 127) / 128, 32 / OC, S * S);
    if (S == 2) {
        const int wg = wgrad_small_grid(tiles(Wg32<2>::TR, Wg32<2>::TC));
        k_wgrad32<2><<<wg, 256, 0, st>>>(in, H, gz, Ho, B, part);
        sums.add(part, wg, WG32_REC, grad, false);
        k_conv_bwd_data32<2><<<grid, 128, 0, st>>>(gz, Ho, theta, in, gx, H, nyg, total);
    } else {
        const int wg = wgrad_small_grid(tiles(Wg32<1>::TR, Wg32<1>::TC));
        k_wgrad32<1><<<wg, 256, 0, st>>>(in, H, gz, Ho, B, part);
        sums.add(part, wg, WG32_REC, grad, false);
        k_conv_bwd_data32<1><<<grid, 128, 0, st>>>(gz, Ho, theta, in, gx, H, nyg, total);
    }
}

}  // namespace

struct reg_cnn {
    cudaStream_t stream = nullptr;
    int side = 0, max_batch = 0;
    int64_t n = 0;
    float *theta = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;
    float *act[NL] = {nullptr};  // layer outputs (post-ReLU, the last one raw)
    float *g0 = nullptr, *g1 = nullptr;  // gradient ping-pong (largest activation)
    float *gy = nullptr;
    double *partial = nullptr, *loss = nullptr;
    uint16_t *actb[5] = {nullptr};  // tensor-core path: outputs of layers 0..4, BF16 planar [b][c/8][y][x][c%8]
    uint32_t *wpack_u = nullptr;  // the 32 -> 32 layers' weights in the tcgen05 operand layout
    uint32_t *wpack_d = nullptr;  // the same, flipped and transposed for the data gradients
    uint32_t *wpack_first = nullptr, *wpack_last = nullptr;  // the first and last layers, tcgen05 layouts
    // parameter version (set_params, adam_step) and the version the packed
    // copies were made from: the packing runs only after a change
    int64_t version = 0, packed = -1;
    int *uerr = nullptr;          // error word of the tcgen05 kernels (a wait ran out): device view
    int *uerr_host = nullptr;     // the same word, pinned host memory mapped into the device
    float *wpart = nullptr;     // per-block partial weight gradients, a region per layer
    int64_t step = 0;
};

namespace {

reg_status cnn_fail(reg_status st, const char *msg) { return reg_internal_fail(st, msg); }

#define CKC(x)                                                          \
    do {                                                                \
        cudaError_t e_ = (x);                                           \
        if (e_ != cudaSuccess) return cnn_fail(REG_ECUDA, cudaGetErrorString(e_)); \
    } while (0)

int out_side(int k, int side)
{
    int H = side;
    for (int j = 0; j <= k; j++) H = (H + 2 - 3) / LAYERS[j].S + 1;
    return H;
}

int in_side(int k, int side) { return k == 0 ? side : out_side(k - 1, side); }

int64_t act_elems(int k, int side) { return (int64_t)LAYERS[k].O * out_side(k, side) * out_side(k, side); }

}  // namespace

int64_t cnn_output_side(const reg_cnn *h) { return out_side(NL - 1, h->side); }

reg_status cnn_check_device_error(reg_cnn *h)
{
    volatile int *w = h->uerr_host;
    const int e = *w;
    if (e == 0) return REG_OK;
    *w = 0;
    return cnn_fail(REG_ECUDA, e == 1   ? "tcgen05 convolution: a copy did not complete in time"
                               : e == 2 ? "tcgen05 convolution: the tensor-core work did not complete in time"
                                        : "tcgen05 convolution: shared memory not 128-byte aligned");
}
int cnn_input_side(const reg_cnn *h) { return h->side; }
int cnn_max_batch(const reg_cnn *h) { return h->max_batch; }

// Forward of a batch of pairs x (device, B x 2 x side x side) into y (device,
// B x 2 x side/4 x side/4) on the given stream; the layer outputs stay in the
// handle for a backward pass.
reg_status cnn_forward(reg_cnn *h, const float *x, int B, float *y, cudaStream_t st, bool tc)
{
    const int S = h->side;
    const float *a = x;
    if (tc && h->packed != h->version) {
        const float *th[NL];
        for (int k = 0; k < NL; k++) th[k] = h->theta + param_offset(k);
        const reg_status rs = cnn_pack_umma(th, h->wpack_first, h->wpack_u, h->wpack_last, h->wpack_d, st);
        if (rs != REG_OK) return rs;
        h->packed = h->version;
    }
    for (int k = 0; k < NL; k++) {
        const int H = in_side(k, S);
        const float *th = h->theta + param_offset(k);
        float *out = (k == NL - 1 && y) ? y : h->act[k];
        if (tc) {
            // tensor-core path, all six layers on tcgen05: layer 0 from the FP32
            // input, the others from the BF16 planar activations, which layers
            // 0..4 write; layer 5 writes the FP32 output
            reg_status rs;
            if (k == 0)
                rs = cnn_first_umma(a, H, th, h->actb[0], B, st, h->wpack_first, h->uerr);
            else if (k == NL - 1)
                rs = cnn_last_umma(h->actb[k - 1], H, th, out, B, st, h->wpack_last, h->uerr);
            else
                rs = cnn_conv32_umma(h->actb[k - 1], H, th, h->actb[k], B, LAYERS[k].S, st,
                                     h->wpack_u + (k - 1) * cnn_conv32_umma_words(), h->uerr);
            if (rs != REG_OK) return rs;
        } else {
            fwd(k, a, H, th, out, B, st);
        }
        if (k == NL - 1 && y && y != h->act[k])
            CKC(cudaMemcpyAsync(h->act[k], y, sizeof(float) * act_elems(k, S) * B, cudaMemcpyDeviceToDevice, st));
        a = out;
    }
    CKC(cudaGetLastError());
    return REG_OK;
}

extern "C" {

int64_t reg_cnn_num_params(void) { return total_params(); }
reg_status reg_cnn_loss_grad_tc(reg_cnn_t h, const float *x, const float *target, int32_t batch, double *loss,
                                float *grad_out);

reg_status reg_cnn_create(int32_t side, int32_t max_batch, void *cuda_stream, reg_cnn_t *out)
{
    if (!out || side < 16 || side % 4 != 0 || side > 4096 || max_batch < 1) return cnn_fail(REG_EINVAL, "bad argument");
    reg_cnn *h = new reg_cnn();
    h->stream = (cudaStream_t)cuda_stream;
    h->side = side;
    h->max_batch = max_batch;
    h->n = total_params();
    auto alloc = [&](void **p, size_t bytes) { return cudaMalloc(p, bytes) == cudaSuccess; };
    bool ok = alloc((void **)&h->theta, sizeof(float) * h->n) && alloc((void **)&h->grad, sizeof(float) * h->n) &&
              alloc((void **)&h->m, sizeof(float) * h->n) && alloc((void **)&h->v, sizeof(float) * h->n);
    int64_t big = 0;
    for (int k = 0; k < NL && ok; k++) {
        ok = alloc((void **)&h->act[k], sizeof(float) * act_elems(k, side) * max_batch);
        if (ok && k < 5) ok = alloc((void **)&h->actb[k], sizeof(uint16_t) * act_elems(k, side) * max_batch);
        big = std::max(big, act_elems(k, side));
    }
    big = std::max(big, (int64_t)2 * side * side);
    ok = ok && alloc((void **)&h->g0, sizeof(float) * big * max_batch) &&
         alloc((void **)&h->g1, sizeof(float) * big * max_batch) &&
         alloc((void **)&h->gy, sizeof(float) * act_elems(NL - 1, side) * max_batch) &&
         alloc((void **)&h->partial, sizeof(double) * 1024) && alloc((void **)&h->loss, sizeof(double)) &&
         alloc((void **)&h->wpack_u, sizeof(uint32_t) * 4 * cnn_conv32_umma_words()) &&
         alloc((void **)&h->wpack_d, sizeof(uint32_t) * 4 * cnn_conv32_umma_words()) &&
         alloc((void **)&h->wpack_first, sizeof(uint32_t) * cnn_first_umma_words()) &&
         alloc((void **)&h->wpack_last, sizeof(uint32_t) * cnn_last_umma_words()) &&
         cudaHostAlloc((void **)&h->uerr_host, sizeof(int), cudaHostAllocMapped) == cudaSuccess &&
         cudaHostGetDevicePointer((void **)&h->uerr, h->uerr_host, 0) == cudaSuccess &&
         alloc((void **)&h->wpart, sizeof(float) * wpart_offset(NL));
    if (!ok) {
        reg_cnn_destroy(h);
        return cnn_fail(REG_ENOMEM, "device allocation failed");
    }
    cudaMemsetAsync(h->theta, 0, sizeof(float) * h->n, h->stream);
    cudaMemsetAsync(h->m, 0, sizeof(float) * h->n, h->stream);
    cudaMemsetAsync(h->v, 0, sizeof(float) * h->n, h->stream);
    if (cudaStreamSynchronize(h->stream) != cudaSuccess) {
        reg_cnn_destroy(h);
        return cnn_fail(REG_ECUDA, "init");
    }
    *reinterpret_cast<volatile int *>(h->uerr_host) = 0;
    *out = h;
    return REG_OK;
}

reg_status reg_cnn_set_params(reg_cnn_t h, const float *theta, int32_t on_device)
{
    if (!h || !theta) return cnn_fail(REG_EINVAL, "bad argument");
    CKC(cudaMemcpyAsync(h->theta, theta, sizeof(float) * h->n,
                        on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, h->stream));
    CKC(cudaMemsetAsync(h->m, 0, sizeof(float) * h->n, h->stream));
    CKC(cudaMemsetAsync(h->v, 0, sizeof(float) * h->n, h->stream));
    h->step = 0;
    h->version++;
    CKC(cudaStreamSynchronize(h->stream));
    return REG_OK;
}

reg_status reg_cnn_get_params(reg_cnn_t h, float *theta, int32_t on_device)
{
    if (!h || !theta) return cnn_fail(REG_EINVAL, "bad argument");
    CKC(cudaMemcpyAsync(theta, h->theta, sizeof(float) * h->n,
                        on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, h->stream));
    CKC(cudaStreamSynchronize(h->stream));
    return REG_OK;
}

reg_status reg_cnn_forward(reg_cnn_t h, const float *x, int32_t batch, float *y, int32_t tensor_cores)
{
    if (!h || !x || !y || batch < 1 || batch > h->max_batch) return cnn_fail(REG_EINVAL, "bad argument");
    reg_status st = cnn_forward(h, x, batch, y, h->stream, tensor_cores != 0);
    if (st != REG_OK) return st;
    CKC(cudaStreamSynchronize(h->stream));
    return cnn_check_device_error(h);
}

static reg_status loss_grad(reg_cnn_t h, const float *x, const float *target, int32_t batch, double *loss,
                            float *grad_out, bool tc);

reg_status reg_cnn_loss_grad(reg_cnn_t h, const float *x, const float *target, int32_t batch, double *loss,
                             float *grad_out)
{
    return loss_grad(h, x, target, batch, loss, grad_out, false);
}

reg_status reg_cnn_loss_grad_tc(reg_cnn_t h, const float *x, const float *target, int32_t batch, double *loss,
                                float *grad_out)
{
    return loss_grad(h, x, target, batch, loss, grad_out, true);
}

// Loss and gradient; tc: the forward of all six layers, the four 32 -> 32
// layers' weight and data gradients on the tensor cores (BF16 operands, FP32
// accumulation); the weight gradients of the 2 -> 32 and 32 -> 2 layers
// (k_wgrad_first, k_wgrad_last) and the last layer's data gradient on the CUDA
// cores in FP32.
static reg_status loss_grad(reg_cnn_t h, const float *x, const float *target, int32_t batch, double *loss,
                            float *grad_out, bool tc)
{
    if (!h || !x || !target || batch < 1 || batch > h->max_batch) return cnn_fail(REG_EINVAL, "bad argument");
    cudaStream_t st = h->stream;
    const int S = h->side, B = batch;
    reg_status rs = cnn_forward(h, x, B, nullptr, st, tc);
    if (rs != REG_OK) return rs;
    const int64_t ny = act_elems(NL - 1, S) * B;
    const int nb = (int)std::min<int64_t>(1024, (ny + 255) / 256);
    k_mse<<<nb, 256, 0, st>>>(h->act[NL - 1], target, ny, h->gy, h->partial);
    k_sum_partials<<<1, 256, 0, st>>>(h->partial, nb, 1.0 / (double)ny, h->loss);
    const float *gz = h->gy;
    float *bufs[2] = {h->g0, h->g1};
    CnnSumList sums;
    for (int k = NL - 1; k >= 0; k--) {
        const int H = in_side(k, S);
        const float *in = k == 0 ? x : h->act[k - 1];
        const float *th = h->theta + param_offset(k);
        float *gr = h->grad + param_offset(k);
        float *gx = k == 0 ? nullptr : bufs[k & 1];
        float *part = h->wpart + wpart_offset(k);
        if (tc && k >= 1 && k <= 4) {
            // the layer's input and the mask below: BF16 planar
            const uint16_t *inb = h->actb[k - 1];
            rs = cnn_wgrad32_umma(inb, H, gz, B, LAYERS[k].S, gr, part, sums, st, h->uerr);
            if (rs != REG_OK) return rs;
            const uint32_t *wp = h->wpack_d + (k - 1) * cnn_conv32_umma_words();
            if (LAYERS[k].S == 1) rs = cnn_dgrad32_umma(gz, H, inb, gx, B, st, wp, h->uerr);
            else rs = cnn_dgrad32s2_umma(gz, H / 2, inb, gx, B, st, wp, h->uerr);
            if (rs != REG_OK) return rs;
            gz = gx;
            continue;
        }
        if (tc && k == NL - 1) {
            // the last layer's input (and the mask below) is the planar BF16
            // output of layer 4
            const int nt = B * ((H + WL_TW - 1) / WL_TW) * ((H + WL_TR - 1) / WL_TR), grid = wgrad_small_grid(nt);
            k_wgrad_last<true><<<grid, 256, 0, st>>>(h->actb[k - 1], H, gz, B, part);
            sums.add(part, grid, WL_REC, gr, false);
            const int total = B * H * H;
            k_bwd_data_last<true><<<(total + 127) / 128, 128, 0, st>>>(gz, th, h->actb[k - 1], gx, H, total);
            gz = gx;
            continue;
        }
        if (tc && k == 0) {
            const int Ho = H / 2, nt = B * ((Ho + WF_TW - 1) / WF_TW) * ((Ho + WF_TR - 1) / WF_TR);
            const int grid = wgrad_small_grid(nt);
            k_wgrad_first<<<grid, 256, 0, st>>>(x, H, gz, Ho, B, part);
            sums.add(part, grid, WF_REC, gr, false);
            continue;
        }
        bwd(k, in, H, gz, th, gx, gr, B, st, part, sums);
        gz = gx;
    }
    cnn_sum_records(sums, st);
    CKC(cudaGetLastError());
    if (loss) CKC(cudaMemcpyAsync(loss, h->loss, sizeof(double), cudaMemcpyDeviceToHost, st));
    if (grad_out) CKC(cudaMemcpyAsync(grad_out, h->grad, sizeof(float) * h->n, cudaMemcpyDeviceToHost, st));
    CKC(cudaStreamSynchronize(st));
    return cnn_check_device_error(h);
}

reg_status reg_cnn_adam_step(reg_cnn_t h, double lr, double beta1, double beta2, double eps)
{
    if (!h || !(lr > 0.0) || !(beta1 >= 0.0 && beta1 < 1.0) || !(beta2 >= 0.0 && beta2 < 1.0) || !(eps > 0.0))
        return cnn_fail(REG_EINVAL, "bad argument");
    h->step++;
    h->version++;
    const double c1 = 1.0 - std::pow(beta1, (double)h->step), c2 = 1.0 - std::pow(beta2, (double)h->step);
    k_adam<<<(int)std::min<int64_t>(1024, (h->n + 255) / 256), 256, 0, h->stream>>>(
        h->theta, h->grad, h->m, h->v, h->n, (float)lr, (float)beta1, (float)beta2, (float)eps, (float)c1, (float)c2);
    CKC(cudaGetLastError());
    CKC(cudaStreamSynchronize(h->stream));
    return REG_OK;
}

reg_status reg_cnn_destroy(reg_cnn_t h)
{
    if (!h) return REG_OK;
    cudaFree(h->theta);
    cudaFree(h->grad);
    cudaFree(h->m);
    cudaFree(h->v);
    for (int k = 0; k < NL; k++) cudaFree(h->act[k]);
    for (int k = 0; k < 5; k++) cudaFree(h->actb[k]);
    cudaFree(h->g0);
    cudaFree(h->g1);
    cudaFree(h->gy);
    cudaFree(h->wpack_u);
    cudaFree(h->wpack_d);
    cudaFree(h->wpack_first);
    cudaFree(h->wpack_last);
    if (h->uerr_host) cudaFreeHost(h->uerr_host);
    cudaFree(h->wpart);
    cudaFree(h->partial);
    cudaFree(h->loss);
    delete h;
    return REG_OK;
}

}  // extern "C"
