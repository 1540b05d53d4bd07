// Internal device data structures of libreg (not part of the public ABI).
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "arith.h"

#define REG_MAX_LEVELS 8
#define REG_MAX_TRIALS 8
#define REG_CTL_THREADS 512  // threads per block of the control kernel
// Warp strips of the gradient and trial kernels: the 32 lanes of a warp hold 32
// adjacent node columns and walk down the rows of a tile together, so that
// vertical neighbours stay in registers and horizontal ones are a shuffle away.
#define REG_GW 30  // gradient tile: owned node columns (lanes 1..30; lanes 0, 31 are halo)
#define REG_CW 31  // trial tile: owned cell columns (lanes 0..30; lane 31 is the right corner)
#define REG_TRIAL_ROWS 32  // most cell rows of a trial tile (its nodes lie in shared memory)
#define REG_STRIP_THREADS 128  // threads per block of the strip kernels (a tile per block, or per warp in the
                               // gradient pass of many tiles)
// Rows per strip tile at a level of n nodes per side (owned node rows of a
// gradient tile, owned cell rows of a trial tile): short strips on the coarse
// levels, where a tile's row walk is latency bound, long ones on the fine
// levels, where the halo rows cost bandwidth.
// Default strip rows of a level of n nodes per side (the tile autotuner may
// pick others per level): short strips where a tile's row walk is latency
// bound, long ones where there are enough tiles.
__host__ __device__ __forceinline__ int strip_rows(int n) { return n <= 65 ? 8 : (n <= 257 ? 16 : 32); }
#define PT_STRIDE (3 * REG_MAX_TRIALS + 3)  // floats per trial-tile partial record
#define PG_STRIDE 2                         // floats per gradient-tile partial record

// Phases of the per-operator state machine.
enum {
    PH_START = 0,    // evaluate the energy at the level's initial u (tau = 0)
    PH_GRAD = 1,     // apply the pending step, then gradient + first trial pass
    PH_TRIAL = 2,    // more step sizes of the same Armijo search
    PH_PROLONG = 3,  // prolongate u + pending step from the level below, START at the result
    PH_DONE = 4      // the batch's final pass applies the pending step and writes the output slot
};
enum { SEARCH_INIT = 0, SEARCH_WIDEN = 1, SEARCH_SHRINK = 2 };
enum { OPST_CONVERGED = 0, OPST_MAXITER = 1, OPST_STALLED = 2, OPST_NONFINITE = 3, OPST_ZERO_GRAD = 4 };

// Device work counters (nodes swept per kernel family, summed over steps).
enum { KW_G = 0,         // gradient pass nodes
       KW_T = 1,         // trial pass nodes (u, d, R, T read)
       KW_TSTART = 2,    // level-start energy nodes (u, R, T read)
       KW_TSAMPLES = 3,  // trial samples (nodes x step sizes)
       KW_PPROL = 4,     // prolongation: fine nodes written
       KW_PFIN = 5,      // final write: nodes
       KW_TEXACT = 6,    // trial nodes whose largest move leaves the cell (exact path)
       KW_TSEQ = 7,      // nodes x sequential Armijo trials decided (the one-at-a-time rule's trials)
       KW_COUNT = 8 };

// State of one operator at one node of a level, read and written as two
// 16-byte words: the displacement in grid units of the level as a float pair
// per component (value = (x, y) + (z, w), "double-float"), the descent
// direction d = -g / w, and the per-node weights of the current search
// (M~ That at u, M~ R~) that the trial passes use.
struct __align__(16) NodeRec {
    float4 u;
    float2 d;
    float mt;  // 36 M~ That (integer stencil weights, unscaled)
    float mr;  // M~ R~
};

struct LevelDesc {
    int n;            // nodes per side (2^l + 1)
    int pitch;        // row pitch in elements (float2 for U/D, scalar for images)
    int hg, ht;       // strip rows of the gradient and trial tiles at this level
    int tg, tt;       // tiles of a gradient and a trial pass at this level
    float h2;         // h^2 = 4^-l (as float for scaling, exact)
    double h2d;       // h^2 in double
    const void *R;    // normalised reference frame (mean 0, FE sigma 1) at this level
    const void *T;    // normalised template frame
    const float *MR;  // M~ R~: the reference frame times the FE mass matrix (units h^2)
    NodeRec *V[2];    // node records, double-buffered (the gradient pass reads one, writes the other)
    const float2 *sm_tab;  // H1-type smoother: Thomas coefficients (c'_i, m_i) of the level's 1D system
};

struct OpDesc {
    int nl;                 // number of levels
    int init;               // 0 identity, 1 copy left, 2 compose(left, right)
    const float2 *left;     // finest-level slot fields (px == grid units of level L)
    const float2 *right;
    float2 *out;            // destination slot (finest level)
    int slot_pitch;
    int judge;              // the output slot holds a learned start: measure the correction
    int part0;              // first of the operator's tile records in partG and partT
    // Lockstep replay (diagnostic; null: free-running search).  Level k
    // (0 = coarsest) takes exactly the accepted step sizes
    // lock_tau[lock_off[k] .. lock_off[k+1]), one per gradient iteration, and
    // ends after the last of them.
    const double *lock_tau;
    int lock_off[REG_MAX_LEVELS + 1];
    LevelDesc lv[REG_MAX_LEVELS];  // index 0 = coarsest level m0
};

// What the gradient and trial passes of a step read of an operator, gathered by
// the control kernel in two cache lines: the passes reach their first node
// records three dependent loads after their start (plan, this, record), and the
// scalars are rounded to float once per step instead of once per tile.
struct __align__(16) StepDesc {
    const void *T;       // template at the level
    const float *MR;
    const NodeRec *Vs;   // records before the gradient pass (or the only ones of a level start)
    NodeRec *Vc;         // records the gradient pass writes and the trial pass reads
    const NodeRec *VC;   // PH_PROLONG: the coarser level's records
    int cpitch;          // and their pitch
    int phase, n, pitch, hg, ht, ntr, part0;
    float ih2;           // 1 / h^2 (exact: a power of two)
    float tau_acc;       // pending step
    float isig, c36, cT; // 1 / sigma, NCC / sigma^2 / 36, NCC / sigma^2 T_bar at u
    float tau[REG_MAX_TRIALS];  // step sizes of the trial pass
};

// An evaluated energy: the FE sums S1 = int That, S2 = int That^2, S3 = int That
// R~ (R~ normalised: mean 0, FE sigma 1; S1 is That's mean), NCC = S3 / sigma with
// sigma = sqrt(S2 - S1^2), the gradient pass's coefficients there, and of a trial the energy
// change, the Armijo test and the stopping test.
struct EvalAt {
    double S1, S2, S3, ncc, dE;
    float isig, c36, cT;
    int acc, conv, pad;
};

struct OpState {
    StepDesc step;
    int phase, lvl, cur, src;
    int iter, iters_total, trials_seq, evals;
    int status, nonfinite_seen, search, ntr;
    int tG, tT;       // gradient and trial tiles of this step
    double tau;       // base step of the current search
    double tau_acc;   // step to apply at the start of the next gradient pass, prolongation or result
    double sh_tau;    // shrinking: last rejected step
    double btau;      // last accepted step of the search
    double E;         // at the current u
    double slope;
    double Qud, Qdd;  // Dirichlet forms u^T K d and d^T K d of the current search
    EvalAt cur_ev;    // at the current u
    EvalAt best_ev;   // last accepted trial of a search that goes on in another pass
    double trial_tau[REG_MAX_TRIALS];
    double corr;  // judged ops: sum over finest nodes of |u_final - u_start| (x + y, px)
};

// Device-side batch: everything the step kernels need, passed by value.
// Sizes that change per batch live in device memory (ctr) so that a captured
// graph stays valid across batches.
struct BatchDev {
    OpDesc *ops;
    OpState *st;
    int2 *plan;                  // per op: {gradient tiles, trial tiles} of the next step
    int *listG, *listT;          // batches of more than 32 ops: compacted op indices per family
    int *prefG, *prefT;          // and exclusive prefix of tile counts (n+1 entries)
    int *ctr;                    // [0] n_ops [2] nG [3] nT [5] itemsG [6] itemsT [7] n_active
                                 // [8] error flag [9] blocks of the control kernel that are done
    float *partG;                // per gradient tile: slope and u^T K d partials (PG_STRIDE)
    float *partT;                // per trial tile: 3 sums per step size, .., the Dirichlet form of d (PT_STRIDE)
    double *partU;               // per tile of a level-start pass: 3 sums and the Dirichlet form of u
    unsigned long long *work;    // per kernel family: nodes processed
    double *trace;               // optional Armijo trial records (7 doubles each)
    unsigned long long *trace_len;
    long long trace_cap;
    double lambda, sigma, tau_init, tau_max, tau_min, eps;
    float lam6;                  // lambda / 6
    int iter_max, J, bf16;
    // H1-type smoother (smooth != 0): per op and column chunk of
    // REG_GW columns, the partial sums {sum omega d_L2 . d, sum d . 6 K u}
    float *partS;
    int smooth, rch, cch;  // row chunks and column chunks of REG_GW per op (maxima)
    float sm_a;            // off-diagonal of the dimensionless 1D system (1/6 - s^2/2)
};

// Raw levels of the images whose pyramids are being built (0 = coarsest): node
// (r, c) of image z is img[z stride + min(r, lim) pitch + min(c, lim)] (lim < n - 1:
// a frame embedded on the vertex grid by repeating its last row and column); out
// and opitch: the level inside a pyramid block.
struct RawLevel {
    const float *img;
    int64_t stride, pitch, out;
    int n, lim, opitch;
};
struct RawLevels {
    RawLevel l[REG_MAX_LEVELS];
    int tiles[REG_MAX_LEVELS];  // 32 x 32 node tiles per level
    int nl;
};

// Rigid variant: one level of one operator, and one requested parameter set
// (element 0 of an operator's REG_MAX_TRIALS requests carries the count n_e
// and, with grad, the scalars of the gradient at that parameter set).
struct RigidLevel {
    int n, pitch;
    const void *T;     // normalised template at this level
    const float *MR;   // M~ R~ of the normalised reference
};
struct RigidReq {
    float a, b, tx, ty;           // cos(alpha) - 1, sin(alpha), translation in grid units
    float ca, sa, h, nm1;         // cos, sin, grid spacing 1/(n-1) and n-1 (gradient only)
    float inv_sig, ncc_over_var, tbar;  // 1/sigma_T, NCC/sigma_T^2, T_bar at the gradient's parameters
    int n_e, grad;                // request 0: number of parameter sets, gradient wanted
};
#define RIGID_SUMS (3 * REG_MAX_TRIALS + 3)  // 3 energy sums per set, then 3 gradient sums

static inline int cdiv(int a, int b) { return (a + b - 1) / b; }

// Compensated ("double-float") displacement arithmetic.  The accepted steps of
// a level shrink to ~1e-6 grid units while |u| is several units: one float
// cannot take such a step without rounding it by percents, so u is kept as an
// unevaluated sum hi + lo of two floats and updated with an exact two-sum.
// (hi + lo) + v, renormalised so that |lo| <= ulp(hi) / 2
__device__ __forceinline__ void df_add(float &hi, float &lo, float v)
{
    float s, e;
    two_sum(hi, v, s, e);
    e = __fadd_rn(e, lo);
    hi = __fadd_rn(s, e);
    lo = __fsub_rn(e, __fsub_rn(hi, s));
}

__device__ __forceinline__ float4 df_add2(float4 u, float vx, float vy)
{
    df_add(u.x, u.z, vx);
    df_add(u.y, u.w, vy);
    return u;
}

// floor(x) as an int and as a float without a float-to-int conversion
// instruction (conversions run on the narrow double-precision pipe of this
// GPU): adding 1.5 * 2^23 rounds x to an integer held in the low mantissa
// bits, one correction step turns round-to-nearest into floor.  |x| < 2^22.
__device__ __forceinline__ int floor_i(float x, float &fl)
{
    const float magic = 12582912.0f;  // 1.5 * 2^23
    float t = __fadd_rn(x, magic);
    int i = __float_as_int(t) - 0x4B400000;
    float r = __fsub_rn(t, magic);
    if (r > x) {
        i -= 1;
        r -= 1.f;
    }
    fl = r;
    return i;
}

// Integer part and fraction of hi + lo.  The fraction is rounded to float, the
// integer part is exact: hi - floor(hi) is exact and is either 0 or at least
// ulp(hi) > |lo|, so hi + lo lies below floor(hi) only when that fraction is 0
// and lo < 0.
__device__ __forceinline__ void df_split(float hi, float lo, int &ip, float &fr)
{
    float f;
    int i = floor_i(hi, f);
    float a = (hi - f) + lo;
    if (a < 0.f) {
        i -= 1;
        a += 1.f;
    }
    ip = i;
    fr = a;
}
