// batch_lu.cu -- one persistent kernel that factorizes, solves and refines a
// batch of small independent sparse systems (static-pivot LU, Sec. III).
//
// Each CTA takes whole systems from a device queue (largest first) and runs,
// for its system, everything the single-system path spreads over launches:
// assembly, then the panels level by level -- diagonal-block LU with static
// pivot replacement, the two panel TRSMs (L and U^T sides), and the updates
// of the facing panels with the scatter fused (Sec. V-B) -- then the
// triangular solves and FP64 iterative refinement.  No CTA ever waits on
// another, so the kernel needs no grid-wide synchronisation.
//
// Schedule inside a CTA (the leaf-versus-top choice is a launch parameter):
//  * panels at most `leaf_width` wide with at most kLeafRows rows below go one
//    per warp, all panels of a level at once, their updates added atomically
//    (siblings may share targets);
//  * the others use the whole CTA one at a time (plain read-modify-write);
//  * the solves go one panel per warp, level by level, on a copy of the
//    right-hand side in shared memory.
//
// What bounds it: chains.  A system's panels of a level rarely fill the CTA's
// warps, each is a string of loads, pivots and barriers, and of 19 resident
// warps' cycles a scheduler spends 6.5 at barriers and 5.9 on loads per issued
// instruction, so FP32 batches of many systems run four CTAs an SM (64 registers;
// three: 29.3 ms, four: 27.8), smaller ones as many as hold them all at once, with
// the registers that this leaves (24 systems of 5 to 40 a side, FP32: 1.62 -> 1.23
// ms; registers spilled, bytes of stores: 16 to 20 at two CTAs an SM, 56 to 68 at
// three, 164 to 232 at four, 128 to 136 in FP64).  4096 systems (grids of 12 to 80 a side, FP32 with refinement) 37.5 ->
// 27.7 ms, 24 systems (5 to 40 a side, FP64) 3.29 -> 2.66 ms, by narrow panels
// and sweeps with their rows in registers and blocked pivots of the wide ones;
// in FP64 the FP64 unit's rate for narrow panels bounds the leaves.
#include "batch_kernel.cuh"
#include "lublock.cuh"

#include <cmath>

namespace spx {
namespace {

constexpr int kWarps = kBatchThreads / 32;
constexpr int kLeafRows = 32;              // one a lane; taller by one warp: same time, more code
constexpr int kLdC = kBatchMaxWidth + 1;   // odd leading dimensions: no bank conflicts
constexpr int kLdW = kBatchLeafMax + 1;
constexpr int kChunkC = 64;                // TRSM rows per pass and side, CTA mode
constexpr int kChunkW = 32;                // TRSM rows per pass, warp mode
constexpr int kCtaElems = kBatchMaxWidth * kLdC + 2 * kChunkC * kLdC + kBatchMaxWidth;
constexpr int kWarpElems = kBatchLeafMax * kLdW + kChunkW * kLdW + kBatchLeafMax;
static_assert(8 * 9 + 8 + 2 * 32 * 9 + 32 * 2 <= kWarpElems, "panel_warp8's shared memory");
constexpr int kRedDoubles = 3 * kWarps + 2;   // reductions + 4 ints

__device__ __forceinline__ double inf_if_nan(double v) { return v != v ? INFINITY : v; }

// a / d with r = 1 / d at hand: the quotient a r corrected by its remainder
// (Markstein, "Computation of elementary functions on the IBM RISC System/6000
// processor", 1990), as accurate as the division, whose chain of dependent
// operations is several times as long.  What leaves the normal range takes the
// division.
__device__ __forceinline__ float quot(float a, float d, float r)
{
    const float q = a * r, x = fabsf(q);
    if (!((x > 0x1p-60f && x < 0x1p60f) || a == 0.0f) || !(fabsf(d) > 0x1p-60f && fabsf(d) < 0x1p60f)) return a / d;
    return fmaf(fmaf(-q, d, a), r, q);
}
__device__ __forceinline__ double quot(double a, double d, double r)
{
    const double q = a * r;
    const int eq = (__double2hiint(q) >> 20) & 0x7FF, ed = (__double2hiint(d) >> 20) & 0x7FF;
    if (((unsigned)(eq - 600) > 850u && a != 0.0) || (unsigned)(ed - 600) > 850u) return a / d;
    return fma(fma(-q, d, a), r, q);
}

// Static pivoting (Sec. III): a pivot whose magnitude is below tau is replaced
// by +-tau (+tau for 0).  With tau == 0 a zero pivot in column k is recorded in
// *zero_k and replaced by 1 so the work completes.  `least` is tau rounded up to
// T, so that comparing with it is comparing with tau.
template <typename T>
struct Tau {
    bool on;
    T least, value;
    __device__ __forceinline__ explicit Tau(double tau)
    {
        on = tau > 0.0;
        if constexpr (sizeof(T) == 4) least = __double2float_ru(tau);
        else least = tau;
        value = (T)tau;
    }
    __device__ __forceinline__ T pivot(T d, int k, int *nrep, int *zero_k) const
    {
        const T ad = d < (T)0 ? -d : d;
        if (on) {
            if (!(ad >= least)) {
                d = d < (T)0 ? -value : value;
                ++*nrep;
            }
        } else if (!(ad > (T)0)) {
            if (*zero_k < 0) *zero_k = k;
            d = (T)1;
        }
        return d;
    }
};

// LU without row exchanges of the w x w block a (column-major, leading
// dimension ld) by one warp.  Returns the number of replaced pivots (the same
// on every lane).
template <typename T>
__device__ __forceinline__ int getrf_warp(T *a, int w, int ld, const Tau<T> &tau, int lane, int *zero_k)
{
    int nrep = 0;
    for (int k = 0; k < w; ++k) {
        const T d = tau.pivot(a[k + k * ld], k, &nrep, zero_k);
        const T r = (T)1 / d;
        __syncwarp();
        if (lane == 0) a[k + k * ld] = d;
        for (int i = k + 1 + lane; i < w; i += 32) a[i + k * ld] *= r;
        __syncwarp();
        for (int i = k + 1 + lane; i < w; i += 32) {
            const T lik = a[i + k * ld];
            for (int j = k + 1; j < w; ++j) a[i + j * ld] -= lik * a[k + j * ld];
        }
        __syncwarp();
    }
    return nrep;
}

// One row x (length w, in shared memory) of the off-diagonal part:
//   side 0 (L panel):   x <- x U^{-1},  U = upper(lu)
//   side 1 (U^T panel): x <- x L^{-T},  L = unit lower(lu)
// by substitution, two partial sums to halve the dependent chain; rv: the
// reciprocals of lu's diagonal.
template <typename T>
__device__ __forceinline__ void trsm_row(T *x, const T *lu, const T *rv, int ld, int w, int side)
{
    for (int j = 0; j < w; ++j) {
        T s0 = x[j], s1 = (T)0;
        int k = 0;
        if (side == 0) {
            for (; k + 1 < j; k += 2) {
                s0 -= x[k] * lu[k + j * ld];
                s1 -= x[k + 1] * lu[k + 1 + j * ld];
            }
            if (k < j) s0 -= x[k] * lu[k + j * ld];
            x[j] = quot(s0 + s1, lu[j + j * ld], rv[j]);
        } else {
            for (; k + 1 < j; k += 2) {
                s0 -= x[k] * lu[j + k * ld];
                s1 -= x[k + 1] * lu[j + (k + 1) * ld];
            }
            if (k < j) s0 -= x[k] * lu[j + k * ld];
            x[j] = s0 + s1;
        }
    }
}

template <typename T>
__device__ __forceinline__ void sub_to(T *dst, T v, bool atomic)
{
    if (atomic) atomicAdd(dst, -v);
    else *dst -= v;
}

// Updates of every panel facing source panel p (Sec. III step 3), scatter
// fused (Sec. V-B).  For task (p -> t) with facing rows [r0, r1):
//   L side, rows i in [r0, h):  C_L(relmap(i), row(j) - fcol(t)) -= sum_k L(i,k) U^T(j,k)
//   U side, rows i in [r1, h):  C_U(relmap(i), row(j) - fcol(t)) -= sum_k U^T(i,k) L(j,k)
// Threads t0.. of a group of nt; RT rows per thread (spaced so that the
// loads of consecutive threads are consecutive).  Threads run through the
// tasks without waiting for one another.
template <typename T, int RT>
__device__ __forceinline__ void update_group(const BClass &c, int p, T *Ls, T *Us, int t0, int nt, bool atomic)
{
    const int w = c.pw[p], h = c.ph[p];
    const T *Lp = Ls + c.pval[p];
    const T *Up = Us + c.pval[p];
    const int32_t *rows = c.rows + c.prow[p];
    for (int q = c.task_ptr[p]; q < c.task_ptr[p + 1]; ++q) {
        const BTask tk = c.tasks[q];
        const int ht = c.ph[tk.tgt];
        const int fct = c.pfcol[tk.tgt];
        const int32_t *rmap = c.relmap + tk.relmap_off - tk.r0;
        const int N = tk.r1 - tk.r0;
#pragma unroll
        for (int side = 0; side < 2; ++side) {
            const int lo = side == 0 ? tk.r0 : tk.r1;
            const int M = h - lo;
            if (M <= 0) continue;
            const T *Ai = side == 0 ? Lp : Up;     // row operand
            const T *Bj = side == 0 ? Up : Lp;     // facing operand
            T *C = (side == 0 ? Ls : Us) + c.pval[tk.tgt];
            const int MR = (M + RT - 1) / RT;
            for (int e = t0; e < MR * N; e += nt) {
                const int ig = e % MR, j = tk.r0 + e / MR;
                T acc[RT];
#pragma unroll
                for (int r = 0; r < RT; ++r) acc[r] = (T)0;
                for (int k = 0; k < w; ++k) {
                    const T b = Bj[j + (int64_t)k * h];
#pragma unroll
                    for (int r = 0; r < RT; ++r) {
                        const int i = lo + ig + r * MR;
                        if (i < h) acc[r] += Ai[i + (int64_t)k * h] * b;
                    }
                }
                const int64_t coff = (int64_t)(rows[j] - fct) * ht;
#pragma unroll
                for (int r = 0; r < RT; ++r) {
                    const int i = lo + ig + r * MR;
                    if (i < h) sub_to<T>(C + rmap[i] + coff, acc[r], atomic);
                }
            }
        }
    }
}

// Panel p of w <= 8 columns and R <= kLeafRows rows below by one warp (columns
// past w: the identity's).  The diagonal block a row a lane and by shuffles; then
// the rows of both sides in registers, by substitution; then the updates: the
// row operand from the registers, the facing rows from shared memory, one after
// another.  In FP64, where each warp instruction holds the FP64 unit for ~19
// cycles, R <= 16 rows of both sides share the lanes, and groups of lanes take
// the sides and every other facing row at the same time (24 systems 3.2 -> 2.7
// ms; in FP32 the extra registers cost as much as the instructions saved).
template <typename T>
__device__ __forceinline__ void panel_warp8(const BClass &c, int p, T *Ls, T *Us, T *sm, const Tau<T> &tau, int lane,
                                            int *nrep, int *zero_col)
{
    constexpr int W = 8, LDR = W + 1;
    const int w = c.pw[p], h = c.ph[p], R = h - w;
    // FP64 instructions past the panel's width cost more than the branch around them
    auto column = [&](int k) { return sizeof(T) == 4 || k < w; };
    T *Lp = Ls + c.pval[p];
    T *Up = Us + c.pval[p];
    T *lu = sm, *rv = sm + W * LDR, *st = rv + W;   // lu by rows; rows of L, then 32 of U^T
    int64_t *start = reinterpret_cast<int64_t *>(st + 64 * LDR);
    // a task a lane (each faces one row at least), its loads under way with the block's
    const int nt = c.task_ptr[p + 1] - c.task_ptr[p];
    BTask tk{0, 0, 0, 0};
    int tht = 0, tfc = 0, row = 0;
    int64_t tpv = 0;
    if (lane < nt) {
        tk = c.tasks[c.task_ptr[p] + lane];
        tht = c.ph[tk.tgt];
        tfc = c.pfcol[tk.tgt];
        tpv = c.pval[tk.tgt];
    }
    if (lane < R) row = c.rows[c.prow[p] + w + lane];
    T a[W];
#pragma unroll
    for (int k = 0; k < W; ++k) a[k] = lane < w && k < w ? Lp[lane + k * h] : (T)(lane == k ? 1 : 0);
    int zk = -1, nr = 0;
#pragma unroll
    for (int k = 0; k < W; ++k) {
        if (k < w) {
            const T d = tau.pivot(__shfl_sync(0xffffffffu, a[k], k), k, &nr, &zk);
            const T r = (T)1 / d;
            if (lane == k) {
                a[k] = d;
                rv[k] = r;
            }
            const T l = a[k] * r;
            if (lane > k) a[k] = l;
#pragma unroll
            for (int j = k + 1; j < W; ++j)
                if (column(j)) {
                    const T u = __shfl_sync(0xffffffffu, a[j], k);
                    if (lane > k) a[j] -= l * u;
                }
        }
    }
    if (lane == 0) {
        if (nr) atomicAdd(nrep, nr);
        if (zk >= 0) atomicMin(zero_col, c.pfcol[p] + zk);
    }
#pragma unroll
    for (int k = 0; k < W; ++k) {
        if (lane < w && k < w) Lp[lane + k * h] = a[k];
        if (lane < W) lu[lane * LDR + k] = a[k];
    }
    __syncwarp();
    if (R == 0) return;                             // a root: no rows, no updates
    T x[W], y[W];
    constexpr bool kSplit = sizeof(T) == 8;
    if (kSplit && R <= 16) {                    // lanes 0 .. R-1: rows of L, R .. 2R-1: of U^T
        const bool us = lane >= R, in = lane < 2 * R;
        T *X = (us ? Up : Lp) + w + (us ? lane - R : lane);
#pragma unroll
        for (int k = 0; k < W; ++k) x[k] = in && k < w ? X[k * h] : (T)0;
        const int sk = us ? 1 : LDR, sj = us ? LDR : 1;
#pragma unroll
        for (int k = 0; k < W; ++k)
            if (k < w) {
                const T q = quot(x[k], lu[k * LDR + k], rv[k]);
                if (!us) x[k] = q;
#pragma unroll
                for (int j = k + 1; j < W; ++j)
                    if (column(j)) x[j] -= x[k] * lu[k * sk + j * sj];
            }
#pragma unroll
        for (int k = 0; k < W; ++k) {
            if (in && k < w) X[k * h] = x[k];
            if (in) st[(us ? lane - R + 32 : lane) * LDR + k] = x[k];
        }
    } else {                                    // a row of both a lane
        T *Xl = Lp + w + lane, *Xu = Up + w + lane;
#pragma unroll
        for (int k = 0; k < W; ++k) {
            x[k] = lane < R && k < w ? Xl[k * h] : (T)0;
            y[k] = lane < R && k < w ? Xu[k * h] : (T)0;
        }
#pragma unroll
        for (int k = 0; k < W; ++k)
            if (k < w) {
                x[k] = quot(x[k], lu[k * LDR + k], rv[k]);
#pragma unroll
                for (int j = k + 1; j < W; ++j)
                    if (column(j)) {
                        x[j] -= x[k] * lu[k * LDR + j];
                        y[j] -= y[k] * lu[j * LDR + k];
                    }
            }
#pragma unroll
        for (int k = 0; k < W; ++k) {
            if (lane < R && k < w) {
                Xl[k * h] = x[k];
                Xu[k * h] = y[k];
            }
            st[lane * LDR + k] = x[k];
            st[(lane + 32) * LDR + k] = y[k];
        }
    }
    // where facing row j's column starts in its target
    int64_t mine = 0;
    for (int q = 0; q < nt; ++q) {
        const int r0 = __shfl_sync(0xffffffffu, tk.r0, q), r1 = __shfl_sync(0xffffffffu, tk.r1, q);
        const int ht = __shfl_sync(0xffffffffu, tht, q), fct = __shfl_sync(0xffffffffu, tfc, q);
        const int64_t off = __shfl_sync(0xffffffffu, tpv, q);
        if (w + lane >= r0 && w + lane < r1) mine = off + (int64_t)(row - fct) * ht;
    }
    start[lane] = mine;
    __syncwarp();
    const int lg = !kSplit || R > 16 ? 5 : R > 8 ? 4 : R > 4 ? 3 : 2;   // 2^lg lanes a group
    const int v = lane & ((1 << lg) - 1), g = lane >> lg, i = w + v;
    const int side = lg == 5 ? 0 : g & 1, j0 = lg == 5 ? 0 : g >> 1, step = lg == 5 ? 1 : 16 >> lg;
    if (lg < 5) {
#pragma unroll
        for (int k = 0; k < W; ++k) x[k] = v < R ? st[(v + 32 * side) * LDR + k] : (T)0;
    }
    auto relative = [&](int q) {
        const int r0 = __shfl_sync(0xffffffffu, tk.r0, q), off = __shfl_sync(0xffffffffu, tk.relmap_off, q);
        return i < h && i >= r0 ? c.relmap[off + i - r0] : 0;
    };
    const T *fl = st + (side ? 0 : 32 * LDR), *fu = st;      // the facing rows of x and of y
    T *C = side ? Us : Ls;
    int m = nt > 0 ? relative(0) : 0;
    for (int q = 0; q < nt; ++q) {
        const int r0 = __shfl_sync(0xffffffffu, tk.r0, q), r1 = __shfl_sync(0xffffffffu, tk.r1, q);
        const int next = q + 1 < nt ? relative(q + 1) : 0;
        const bool in = i < h && i >= (side ? r1 : r0);
        for (int j = r0 - w + j0; j < r1 - w; j += step) {
            const int64_t o = start[j] + m;
            T s = (T)0;
#pragma unroll
            for (int k = 0; k < W; ++k)
                if (column(k)) s += x[k] * fl[j * LDR + k];
            if (in) atomicAdd(C + o, -s);
            if (lg == 5) {
                s = (T)0;
#pragma unroll
                for (int k = 0; k < W; ++k)
                    if (column(k)) s += y[k] * fu[j * LDR + k];
                if (i < h && i >= r1) atomicAdd(Us + o, -s);
            }
        }
        m = next;
    }
    __syncwarp();
}

// Panel p by one warp (w <= kBatchLeafMax).  sm: kWarpElems elements.
template <typename T, int RT>
__device__ __forceinline__ void panel_warp(const BClass &c, int p, T *Ls, T *Us, T *sm, const Tau<T> &tau, int lane,
                           int *nrep, int *zero_col)
{
    const int w = c.pw[p], h = c.ph[p];
    if (w <= 8) return panel_warp8<T>(c, p, Ls, Us, sm, tau, lane, nrep, zero_col);
    T *lu = sm;
    T *st = sm + kBatchLeafMax * kLdW, *rv = st + kChunkW * kLdW;
    T *Lp = Ls + c.pval[p];
    T *Up = Us + c.pval[p];
    for (int e = lane; e < w * w; e += 32) lu[e % w + (e / w) * kLdW] = Lp[e % w + (e / w) * h];
    __syncwarp();
    int zk = -1;
    const int nr = getrf_warp<T>(lu, w, kLdW, tau, lane, &zk);
    if (lane == 0) {
        if (nr) atomicAdd(nrep, nr);
        if (zk >= 0) atomicMin(zero_col, c.pfcol[p] + zk);
    }
    if (lane < w) rv[lane] = (T)1 / lu[lane + lane * kLdW];
    for (int e = lane; e < w * w; e += 32) Lp[e % w + (e / w) * h] = lu[e % w + (e / w) * kLdW];
    for (int side = 0; side < 2; ++side) {
        T *X = side ? Up : Lp;
        for (int c0 = w; c0 < h; c0 += kChunkW) {
            const int m = min(kChunkW, h - c0);
            for (int e = lane; e < m * w; e += 32) st[(e % m) * kLdW + e / m] = X[c0 + e % m + (int64_t)(e / m) * h];
            __syncwarp();
            if (lane < m) trsm_row<T>(st + lane * kLdW, lu, rv, kLdW, w, side);
            __syncwarp();
            for (int e = lane; e < m * w; e += 32) X[c0 + e % m + (int64_t)(e / m) * h] = st[(e % m) * kLdW + e / m];
            __syncwarp();
        }
    }
    update_group<T, RT>(c, p, Ls, Us, lane, 32, true);
}

// Panel p by the whole CTA (w <= kBatchMaxWidth).  sm: kCtaElems elements.
template <typename T, int RT>
__device__ __forceinline__ void panel_cta(const BClass &c, int p, T *Ls, T *Us, T *sm, const Tau<T> &tau, int *nrep,
                          int *zero_col)
{
    const int tid = threadIdx.x;
    const int w = c.pw[p], h = c.ph[p];
    T *lu = sm;
    T *stL = sm + kBatchMaxWidth * kLdC;
    T *stU = stL + kChunkC * kLdC, *rv = stU + kChunkC * kLdC;
    T *Lp = Ls + c.pval[p];
    T *Up = Us + c.pval[p];
    for (int e = tid; e < w * w; e += kBatchThreads) lu[e % w + (e / w) * kLdC] = Lp[e % w + (e / w) * h];
    __syncthreads();
    int zk = -1;
    int nr = 0;
    getrf_cta<T, 2>(lu, w, kLdC, [&](T d, int k) { return tau.pivot(d, k, &nr, &zk); },
                    [](T d) { return (T)1 / d; });
    if (tid == 0) {
        if (nr) atomicAdd(nrep, nr);
        if (zk >= 0) atomicMin(zero_col, c.pfcol[p] + zk);
    }
    if (tid < w) rv[tid] = (T)1 / lu[tid + tid * kLdC];   // the first chunk's barrier follows
    for (int e = tid; e < w * w; e += kBatchThreads) Lp[e % w + (e / w) * h] = lu[e % w + (e / w) * kLdC];
    for (int c0 = w; c0 < h; c0 += kChunkC) {
        const int m = min(kChunkC, h - c0);
        for (int e = tid; e < m * w; e += kBatchThreads) {
            const int r = e % m, k = e / m;
            stL[r * kLdC + k] = Lp[c0 + r + (int64_t)k * h];
            stU[r * kLdC + k] = Up[c0 + r + (int64_t)k * h];
        }
        __syncthreads();
        if (tid < kChunkC) {
            if (tid < m) trsm_row<T>(stL + tid * kLdC, lu, rv, kLdC, w, 0);
        } else if (tid >= 128 && tid < 128 + kChunkC) {
            if (tid - 128 < m) trsm_row<T>(stU + (tid - 128) * kLdC, lu, rv, kLdC, w, 1);
        }
        __syncthreads();
        for (int e = tid; e < m * w; e += kBatchThreads) {
            const int r = e % m, k = e / m;
            Lp[c0 + r + (int64_t)k * h] = stL[r * kLdC + k];
            Up[c0 + r + (int64_t)k * h] = stU[r * kLdC + k];
        }
        __syncthreads();
    }
    update_group<T, RT>(c, p, Ls, Us, tid, kBatchThreads, false);
    __syncthreads();
}

// Forward sweep of panel p by one warp: y = L11^{-1} w_p (unit lower), then
// w(rows below) -= L21 y, added atomically (panels of a level run at once).
// Eight columns at a time: the 8 x 8 triangle a row a lane, its y passed on by
// shuffles; then a row a lane with eight loads in flight.
template <typename T>
__device__ __forceinline__ void fwd_panel_warp(const BClass &c, int p, const T *Ls, T *wv, int lane)
{
    const int w = c.pw[p], h = c.ph[p], fc = c.pfcol[p];
    const T *Lp = Ls + c.pval[p];
    const int32_t *rows = c.rows + c.prow[p];
    T y[8], l[8];
    for (int k0 = 0; k0 < w; k0 += 8) {
        const int kc = min(8, w - k0);
        const T *Lk = Lp + (int64_t)k0 * h;
        T v = lane < kc ? wv[fc + k0 + lane] : (T)0;
#pragma unroll
        for (int k = 0; k < 8; ++k) l[k] = lane < kc && k < lane ? Lk[k0 + lane + k * h] : (T)0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (k < kc) {
                y[k] = __shfl_sync(0xffffffffu, v, k);
                if (lane > k) v -= l[k] * y[k];
            }
        }
        if (lane < kc) wv[fc + k0 + lane] = v;
        for (int i = k0 + kc + lane; i < w; i += 32) {         // kc == 8 here
            T s = (T)0;
#pragma unroll
            for (int k = 0; k < 8; ++k) s += Lk[i + k * h] * y[k];
            wv[fc + i] -= s;
        }
        __syncwarp();
    }
    for (int i = w + lane; i < h; i += 32) {
        T s = (T)0;
        int k0 = 0;
        for (; k0 + 8 <= w; k0 += 8) {
#pragma unroll
            for (int k = 0; k < 8; ++k) l[k] = Lp[i + (int64_t)(k0 + k) * h];
#pragma unroll
            for (int k = 0; k < 8; ++k) s += l[k] * wv[fc + k0 + k];
        }
        if (k0 < w) {
#pragma unroll
            for (int k = 0; k < 8; ++k) l[k] = k0 + k < w ? Lp[i + (int64_t)(k0 + k) * h] : (T)0;
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (k0 + k < w) s += l[k] * wv[fc + k0 + k];
        }
        atomicAdd(&wv[rows[i]], -s);
    }
}

// Backward sweep of panel p by one warp: z = w_p - U12 w(rows below), then
// x_p = U11^{-1} z.  U12(k, row i) is U^T(i, k).  Eight columns at a time: the
// rows below over the lanes, eight sums a lane, added up by halving shuffles
// (the sum of column k ends in lane k); the triangles as in the forward sweep.
template <typename T>
__device__ __forceinline__ void bwd_panel_warp(const BClass &c, int p, const T *Ls, const T *Us, T *wv, int lane)
{
    const int w = c.pw[p], h = c.ph[p], fc = c.pfcol[p];
    const T *Lp = Ls + c.pval[p];
    const T *Up = Us + c.pval[p];
    const int32_t *rows = c.rows + c.prow[p];
    if (sizeof(T) == 8 && h > w && h - w <= 8) {
        // few rows: a column a lane (in FP64 eight sums' shuffles cost more than the
        // rows; in FP32 the branch costs as much as it saves)
        for (int k = lane; k < w; k += 32) {
            T s0 = wv[fc + k], s1 = (T)0;
            int i = w;
            for (; i + 1 < h; i += 2) {
                s0 -= Up[i + (int64_t)k * h] * wv[rows[i]];
                s1 -= Up[i + 1 + (int64_t)k * h] * wv[rows[i + 1]];
            }
            if (i < h) s0 -= Up[i + (int64_t)k * h] * wv[rows[i]];
            wv[fc + k] = s0 + s1;
        }
        __syncwarp();
    } else if (h > w) {
        for (int k0 = 0; k0 < w; k0 += 8) {
            const int kc = min(8, w - k0);
            T s[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) s[k] = (T)0;
            for (int i = w + lane; i < h; i += 32) {
                const T v = wv[rows[i]];
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (k < kc) s[k] += Up[i + (int64_t)(k0 + k) * h] * v;
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1)
#pragma unroll
                for (int k = 0; k < o; ++k) {
                    const bool up = (lane & o) != 0;
                    const T give = up ? s[k] : s[k + o], keep = up ? s[k + o] : s[k];
                    s[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
                }
            s[0] += __shfl_xor_sync(0xffffffffu, s[0], 8);
            s[0] += __shfl_xor_sync(0xffffffffu, s[0], 16);
            if (lane < kc) wv[fc + k0 + lane] -= s[0];
        }
        __syncwarp();
    }
    for (int k0 = (w - 1) & ~7; k0 >= 0; k0 -= 8) {
        const int kc = min(8, w - k0);
        const T *Lk = Lp + (int64_t)k0 * h;
        T v = lane < kc ? wv[fc + k0 + lane] : (T)0, u[8], x[8];
        const T d = lane < kc ? Lk[k0 + lane + lane * h] : (T)1;
#pragma unroll
        for (int k = 0; k < 8; ++k) u[k] = lane < k && k < kc ? Lk[k0 + lane + k * h] : (T)0;
        const T r = (T)1 / d;
#pragma unroll
        for (int k = 7; k >= 0; --k) {
            if (k >= kc) continue;
            x[k] = __shfl_sync(0xffffffffu, quot(v, d, r), k);
            if (lane == k) v = x[k];
            if (lane < k) v -= u[k] * x[k];
        }
        if (lane < kc) wv[fc + k0 + lane] = v;
        for (int i = lane; i < k0; i += 32) {
            T s = (T)0;
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (k < kc) s += Lk[i + k * h] * x[k];
            wv[fc + i] -= s;
        }
        __syncwarp();
    }
}

// Max over the CTA of three values (every thread gets the result).
__device__ __forceinline__ void block_max3(double *v, double *red)
{
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
#pragma unroll
    for (int q = 0; q < 3; ++q)
        for (int o = 16; o > 0; o >>= 1) v[q] = fmax(v[q], __shfl_xor_sync(0xffffffffu, v[q], o));
    __syncthreads();
    if (lane == 0) {
#pragma unroll
        for (int q = 0; q < 3; ++q) red[q * kWarps + warp] = v[q];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        double m = red[q * kWarps];
#pragma unroll
        for (int u = 1; u < kWarps; ++u) m = fmax(m, red[q * kWarps + u]);
        v[q] = m;
    }
}

// r = b - A x (FP64, original numbering) into wv (permuted, T); returns the
// backward error max|r| / (||A||_inf max|x| + max|b|).
template <typename T>
__device__ __forceinline__ double residual(const BClass &c, const BSys &S, const double *vals, const double *b,
                           const double *x, bool x_zero, double anorm, T *wv, double *red)
{
    double v[3] = {0.0, 0.0, 0.0};   // max |r|, max |x|, max |b|
    for (int i = threadIdx.x; i < S.n; i += kBatchThreads) {
        double s = b[i];
        if (!x_zero)
            for (int e = c.csr_ptr[i]; e < c.csr_ptr[i + 1]; ++e)
                s -= vals[S.voff + c.csr_src[e]] * x[c.csr_col[e]];
        wv[c.iperm[i]] = (T)s;
        v[0] = fmax(v[0], inf_if_nan(fabs(s)));
        if (!x_zero) v[1] = fmax(v[1], inf_if_nan(fabs(x[i])));
        v[2] = fmax(v[2], fabs(b[i]));
    }
    block_max3(v, red);
    const double den = anorm * v[1] + v[2];
    if (den > 0.0) return v[0] / den;
    return v[0] == 0.0 ? 0.0 : INFINITY;
}

template <typename T, int RT>
__device__ __forceinline__ void process(const BatchArgs &a, int sid, T *region, double *red, int *si)
{
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const BSys S = a.sys[sid];
    const BClass c = a.cls[S.cls];
    T *Ls = static_cast<T *>(a.L) + S.foff;
    T *Us = static_cast<T *>(a.U) + S.foff;
    const double *vals = a.vals;

    // assembly: zero the panels, ||A||_inf, then scatter the values
    for (int64_t e = tid; e < c.nstored; e += kBatchThreads) {
        Ls[e] = (T)0;
        Us[e] = (T)0;
    }
    double v[3] = {0.0, 0.0, 0.0};
    for (int i = tid; i < S.n; i += kBatchThreads) {
        double s = 0.0;
        for (int e = c.csr_ptr[i]; e < c.csr_ptr[i + 1]; ++e) s += fabs(vals[S.voff + c.csr_src[e]]);
        v[0] = fmax(v[0], s);
    }
    if (tid == 0) {
        si[1] = 0;
        si[2] = 0x7fffffff;
    }
    block_max3(v, red);   // also orders the zero fill before the scatter
    const double anorm = v[0];
    const Tau<T> tau(a.tau_opt >= 0.0 ? a.tau_opt : 0x1p-26 * anorm);   // sqrt(2^-52) ||A||_inf
    for (int e = tid; e < c.nnz; e += kBatchThreads) {
        const int64_t m = c.amap[e];
        const T x = (T)vals[S.voff + e];
        if (m >= 0) Ls[m] = x;
        else if (m <= -2) Us[-2 - m] = x;
    }
    __syncthreads();

    // factorization, level by level
    auto by_warp = [&](int p) { return c.pw[p] <= a.leaf_width && c.ph[p] - c.pw[p] <= kLeafRows; };
    for (int l = 0; l < c.nlevels; ++l) {
        const int q0 = c.level_ptr[l], q1 = c.level_ptr[l + 1];
        if (a.leaf_width > 0) {
            T *wsm = region + warp * kWarpElems;
            for (int q = q0 + warp; q < q1; q += kWarps) {
                const int p = c.level_panels[q];
                if (by_warp(p)) panel_warp<T, RT>(c, p, Ls, Us, wsm, tau, lane, &si[1], &si[2]);
            }
            __syncthreads();
        }
        for (int q = q0; q < q1; ++q) {
            const int p = c.level_panels[q];
            if (!by_warp(p)) panel_cta<T, RT>(c, p, Ls, Us, region, tau, &si[1], &si[2]);
        }
    }
    __syncthreads();
    const int nrep = si[1];
    const int zero_col = si[2];

    int iters = 0, conv = 1;
    double berr = 0.0;
    if (a.do_solve) {
        const double *b = a.B + S.xoff;
        double *x = a.X + S.xoff;
        T *wv = region;
        for (int i = tid; i < S.n; i += kBatchThreads) x[i] = 0.0;
        residual<T>(c, S, vals, b, x, true, anorm, wv, red);   // w = P b
        __syncthreads();
        for (int s = 1;; ++s) {
            for (int l = 0; l < c.nlevels; ++l) {
                for (int q = c.level_ptr[l] + warp; q < c.level_ptr[l + 1]; q += kWarps)
                    fwd_panel_warp<T>(c, c.level_panels[q], Ls, wv, lane);
                __syncthreads();
            }
            for (int l = c.nlevels - 1; l >= 0; --l) {
                for (int q = c.level_ptr[l] + warp; q < c.level_ptr[l + 1]; q += kWarps)
                    bwd_panel_warp<T>(c, c.level_panels[q], Ls, Us, wv, lane);
                __syncthreads();
            }
            for (int i = tid; i < S.n; i += kBatchThreads) x[c.perm[i]] += (double)wv[i];
            __syncthreads();
            berr = residual<T>(c, S, vals, b, x, false, anorm, wv, red);
            __syncthreads();
            iters = s - 1;
            if (a.tol > 0.0 && berr <= a.tol) break;
            if (s > a.max_iter) break;
        }
        conv = a.tol > 0.0 ? (berr <= a.tol) : 1;
    }
    if (tid == 0) {
        a.iters[sid] = iters;
        a.converged[sid] = conv;
        a.berr[sid] = berr;
        a.nrepl[sid] = nrep;
        a.bad_col[sid] = zero_col == 0x7fffffff ? -1 : zero_col;
        if (!conv) atomicAdd(&a.summary[0], 1u);
        if (zero_col != 0x7fffffff) atomicAdd(&a.summary[1], 1u);
    }
}

template <typename T, int RT, int CTAS>
__global__ void __launch_bounds__(kBatchThreads, CTAS) batch_lu_kernel(BatchArgs a)
{
    extern __shared__ double smd[];
    double *red = smd;
    int *si = reinterpret_cast<int *>(smd + 3 * kWarps);
    T *region = reinterpret_cast<T *>(smd + kRedDoubles);
    for (;;) {
        if (threadIdx.x == 0) si[0] = (int)atomicAdd(a.queue, 1u);
        __syncthreads();
        const int q = si[0];
        __syncthreads();
        if (q >= a.nsys) break;
        process<T, RT>(a, a.order[q], region, red, si);
    }
}

}  // namespace

size_t batch_smem_bytes(int elem_bytes, int n_max)
{
    int elems = kCtaElems;
    if (kWarps * kWarpElems > elems) elems = kWarps * kWarpElems;
    if (n_max > elems) elems = n_max;
    return sizeof(double) * kRedDoubles + (size_t)elem_bytes * (size_t)elems;
}

// fn(kernel) with the kernel for `ctas` CTAs an SM: its registers are what that
// many leave (FP32: 128, 80 or 64 a thread for up to two, three, four; FP64, whose
// shared memory lets two on an SM, 128).
template <typename T, int RT, typename F>
static auto with_ctas(int ctas, F fn)
{
    if constexpr (sizeof(T) == 4) {
        if (ctas > 3) return fn(batch_lu_kernel<T, RT, 4>);
        if (ctas == 3) return fn(batch_lu_kernel<T, RT, 3>);
    }
    return fn(batch_lu_kernel<T, RT, 2>);
}

template <typename F>
static auto with_kernel(int elem_bytes, int rows_per_thread, int ctas, F fn)
{
    if (elem_bytes == 8) {
        if (rows_per_thread == 1) return with_ctas<double, 1>(ctas, fn);
        if (rows_per_thread == 2) return with_ctas<double, 2>(ctas, fn);
        return with_ctas<double, 4>(ctas, fn);
    }
    if (rows_per_thread == 1) return with_ctas<float, 1>(ctas, fn);
    if (rows_per_thread == 2) return with_ctas<float, 2>(ctas, fn);
    return with_ctas<float, 4>(ctas, fn);
}

int batch_max_ctas_per_sm(int elem_bytes, int n_max, int rows_per_thread, int ctas)
{
    const size_t smem = batch_smem_bytes(elem_bytes, n_max);
    return with_kernel(elem_bytes, rows_per_thread, ctas, [&](auto *kernel) {
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        int blocks = 0;
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, kernel, kBatchThreads, smem) == cudaSuccess
                   ? blocks
                   : 0;
    });
}

// The shared-memory attribute is set by batch_max_ctas_per_sm, which the
// caller runs first (outside any stream capture).
void launch_batch(const BatchArgs &a, int elem_bytes, int rows_per_thread, int ctas, int grid, int n_max,
                  cudaStream_t s)
{
    with_kernel(elem_bytes, rows_per_thread, ctas, [&](auto *kernel) {
        kernel<<<grid, kBatchThreads, batch_smem_bytes(elem_bytes, n_max), s>>>(a);
        return 0;
    });
}

}  // namespace spx
