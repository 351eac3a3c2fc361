// sweep.cu -- forward and backward substitution on the panel factor, each
// direction one launch over a device-resident queue of work items.
//
// The items are the per-panel steps of the triangular solves in elimination
// order (Sec. III orders the factorization tasks the same way): a panel item
// applies the inverted diagonal block, a chunk item moves 64 off-diagonal
// rows of a panel between the panel and its ancestors.  CTAs take items from
// one atomic counter in queue order; an item waits on per-panel counters for
// the items it depends on, all of which sit earlier in the queue, so the
// earliest unfinished item always has its inputs and the walk cannot stall.
// Every wait is bounded: past the limit the kernel sets *err and its CTAs
// return, which the host reports as a failed solve.
//
// Forward (L y = b):
//   panel p  waits until every chunk writing into rows of p has finished,
//            then Z_p = Linv_p Y_p and flag[p] = 1;
//   chunk    waits for flag[p] of its panel, Y[rows] -= L_chunk Z_p, then
//            counts itself on each panel owning one of its rows.
// Backward (L^T x = y):
//   chunk    waits for flag[q] of each panel q owning one of its rows, then
//            Tacc_p += L_chunk^T X[rows] and counts itself on its panel;
//   panel p  waits for all its chunks, X_p = M (Z_p - Tacc_p), flag[p] = 1.
// Right-hand sides are column-major n x nrhs in the permuted numbering.
//
// An item is one or two 64 x 64 by 64 x NC products and a hand-off, and the
// sweep is a chain of a few hundred of them, so what counts is the time of one
// item on one SM.  The products are cut accordingly:
//   FP32, NC = 4: 4 x 4 results a thread, k in 16 parts (a loop of four dependent
//     steps instead of 64), joined by shuffles and shared memory; more columns:
//     the kernels at the end, one row and four columns a thread (measured a few
//     per cent faster there than split sums);
//   FP64, NC = 8: one 8 x 8 tile a warp by mma.m8n8k4.f64 (fewer instructions;
//     the rate is the FP64 unit's), without the zero halves of the triangles;
//   FP64, NC = 1: one row a thread, k split in four.
// On this part a 64 x 64 x NC product in FP64 takes 2,400 NC cycles of one
// SM's FP64 unit, so in FP64 the columns are dealt to `groups` independent
// walks of the same queue (group g: column blocks g, g + groups, ...), which
// run on different SMs at the same time.  64^3 diffusion, a forward and a
// backward sweep in ms, before (16 columns on one SM whatever their number)
// and now: FP64 1 column 26.3 -> 5.0, 4 26.6 -> 11.5, 16 27.0 -> 22.5; FP32 1
// column 4.0 -> 3.1.
#include "blocks.cuh"

#include <algorithm>

namespace spx {

namespace {

constexpr int kQThreads = 256;

__device__ __forceinline__ int ld_acquire(const int32_t *p)
{
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Polled by one thread.  False, with *err set, after `limit` polls (of
// about 256 ns each), or as soon as another CTA has reported a timeout.
__device__ bool wait_geq(const int32_t *p, int target, int32_t *err, uint32_t limit)
{
    if (ld_acquire(p) >= target) return true;
    for (uint32_t it = 0; it < limit; ++it) {
        __nanosleep(it < 256 ? 32 : 256);
        if (ld_acquire(p) >= target) return true;
        if ((it & 1023) == 1023 && ld_acquire(err) != 0) return false;
    }
    atomicExch(err, 1);
    return false;
}

// Data written by other CTAs of the same launch is read through L2.
template <typename T>
__device__ __forceinline__ T ld_l2(const T *p)
{
    return __ldcg(p);
}

// Whole CTA: true once every polled counter reached its target.  Thread t
// polls cnt[ids[t]] (ids == nullptr: thread 0 polls cnt[0]) for t < m.
__device__ __forceinline__ bool cta_wait(const int32_t *cnt, const int32_t *ids, int m, int target,
                                         int32_t *err, uint32_t limit)
{
    int ok = 1;
    if ((int)threadIdx.x < m) ok = wait_geq(cnt + (ids ? ids[threadIdx.x] : 0), target, err, limit);
    return __syncthreads_and(ok) != 0;
}

// Whole CTA, after its writes: they become visible before flag[0] = 1 and
// before each cnt[ids[t]] (t < m; ids == nullptr: cnt[0]) is incremented
// (barrier, then one gpu-scope acquire-release fence by the signalling
// thread, which covers the writes the barrier ordered before it).
__device__ __forceinline__ void cta_release(int32_t *flag, int32_t *cnt, const int32_t *ids, int m)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        asm volatile("fence.acq_rel.gpu;" ::: "memory");
        if (flag) atomicExch(flag, 1);
        for (int t = 0; t < m; ++t) atomicAdd(cnt + (ids ? ids[t] : 0), 1);
    }
}

// The factor's blocks (read-only during a sweep) go to shared memory by
// asynchronous copies (cp.async, one element each, zero-filled past the
// panel): every copy of an item is in flight at once, beside the item's
// dependency wait, and stage_wait() before the barrier that precedes their
// first use completes them.  The right-hand sides, written by other CTAs
// of the same launch, are read through L2 after the wait; those staging
// loops issue every load of a batch before its first store.
template <typename T>
__device__ __forceinline__ void cp_async_elem(T *dst, const T *src, bool valid)
{
    static_assert(sizeof(T) == 4 || sizeof(T) == 8, "4- or 8-byte elements");
    const unsigned saddr = (unsigned)__cvta_generic_to_shared(dst);
    const int bytes = valid ? (int)sizeof(T) : 0;
    if constexpr (sizeof(T) == 4)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(saddr), "l"(src), "r"(bytes) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(saddr), "l"(src), "r"(bytes) : "memory");
}

__device__ __forceinline__ void stage_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

// This thread's asynchronous copies are done (a barrier after it makes
// every thread's visible to the CTA).
__device__ __forceinline__ void stage_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }


template <int N>
__device__ __forceinline__ void stage_wait_but()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// ---------------------------------------------------------------------------
// 64 x 64 by 64 x NC products on matrices staged in shared memory.
//   N form: out(i) = sum_k A(i, k) v(k), A(i, k) at idx_n(i, k);
//   T form: out(i) = sum_k A(k, i) v(k), A(k, i) at idx_t(k, i);
// both staged by copying columns of a column-major source.  v(k, c) at
// Vs[vidx(k, c)].  A thread ends up with the kOut results (row(o), col(o)); rows
// outside the product's are left to the caller to skip.  mul_n reads k < K,
// mul_t reads k < K rounded up to 4: the caller zeroes that much of A and v.
// ---------------------------------------------------------------------------
template <typename T, int NC>
struct Prod;

// What a product can leave out: rows past `rows`; tri < 0: A is lower
// triangular (k <= i), tri > 0: the sum starts at k = i.
struct Range {
    int rows, tri;
};

// FP32 operand layout of both forms; k quads of a row are swizzled by the row
// in the T form, so that a warp's 16-byte loads of neighbouring rows fall in
// distinct banks.
struct FloatTile {
    static constexpr int kMat = 64 * 64;
    static __device__ __forceinline__ int idx_t(int k, int i)
    {
        return i * 64 + ((((k >> 2) ^ i) & 15) << 2) + (k & 3);
    }
};

// FP32, 4 columns: 16 row groups (rows rq + 16 q) x 2 parts of k a warp, 8
// parts over the warps.
template <>
struct Prod<float, 4> : FloatTile {
    static constexpr int kOut = 1, kRed = 2048;
    // the two lane halves take alternate k, kept in distinct banks
    static __device__ __forceinline__ int idx_n(int i, int k) { return k * 64 + (i ^ ((k & 1) << 4)); }
    static __device__ __forceinline__ int vidx(int k, int c) { return k * 4 + c; }
    static __device__ __forceinline__ int col(int) { return threadIdx.x & 3; }
    static __device__ __forceinline__ int row(int) { return threadIdx.x >> 2; }
    static __device__ __forceinline__ void mul_n(const float *A, const float *Vs, int K, Range, float *red,
                                                 float (&out)[1])
    {
        const int rq = threadIdx.x & 15, kh = (threadIdx.x >> 4) & 1, span = (K + 15) / 16 * 2;
        const int k0 = (int)(threadIdx.x >> 5) * span, k1 = min(K, k0 + span);
        float acc[4][4] = {};
#pragma unroll 4
        for (int k = k0 + kh; k < k1; k += 2) {
            const float *a = A + k * 64 + (rq ^ (kh << 4));   // (k0 is even)
            const float4 y = *reinterpret_cast<const float4 *>(Vs + vidx(k, 0));
            const float av[4] = {a[0], a[kh ? -16 : 16], a[32], a[kh ? 16 : 48]}, yv[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], yv[j], acc[i][j]);
        }
        join(acc, red, out);
    }
    static __device__ __forceinline__ void mul_t(const float *A, const float *Vs, int K, Range, float *red,
                                                 float (&out)[1])
    {
        const int rq = threadIdx.x & 15, span = ((K + 15) / 16 + 3) & ~3;
        const int k0 = (int)(threadIdx.x >> 4) * span, k1 = min((K + 3) & ~3, k0 + span);
        float acc[4][4] = {};
        for (int k = k0; k < k1; k += 4) {
            float4 y[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) y[u] = *reinterpret_cast<const float4 *>(Vs + vidx(k + u, 0));
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 a = *reinterpret_cast<const float4 *>(A + idx_t(k, rq + 16 * i));
                const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    acc[i][0] = fmaf(av[u], y[u].x, acc[i][0]);
                    acc[i][1] = fmaf(av[u], y[u].y, acc[i][1]);
                    acc[i][2] = fmaf(av[u], y[u].z, acc[i][2]);
                    acc[i][3] = fmaf(av[u], y[u].w, acc[i][3]);
                }
            }
        }
        join(acc, red, out);
    }
    // the lane halves added up by shuffles, the warps through shared memory
    static __device__ __forceinline__ void join(float (&acc)[4][4], float *red, float (&out)[1])
    {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, kh = lane >> 4;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] += __shfl_xor_sync(0xffffffffu, acc[i][j], 16);
        float4 *r4 = reinterpret_cast<float4 *>(red);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if ((i >> 1) == kh)
                r4[warp * 64 + (lane & 15) + 16 * i] = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
        __syncthreads();
        float s = 0.0f;
#pragma unroll
        for (int p = 0; p < 8; ++p) s += red[p * 256 + threadIdx.x];
        out[0] = s;
    }
};

// FP64, 8 columns: an 8 x 8 tile of results a warp on the FP64 tensor path,
// two accumulators (leading dimensions such that a fragment's 32 elements
// fall in distinct banks).
template <>
struct Prod<double, 8> {
    static constexpr int kOut = 2, kMat = 64 * 72, kRed = 0;
    static __device__ __forceinline__ int idx_n(int i, int k) { return k * 72 + i; }
    static __device__ __forceinline__ int idx_t(int k, int i) { return i * 68 + k; }
    static __device__ __forceinline__ int vidx(int k, int c) { return k * 8 + c; }
    static __device__ __forceinline__ int col(int o) { return 2 * (threadIdx.x & 3) + o; }
    static __device__ __forceinline__ int row(int)
    {
        return 8 * (int)(threadIdx.x >> 5) + (int)((threadIdx.x & 31) >> 2);
    }
    template <bool kT>
    static __device__ __forceinline__ void mul(const double *A, const double *Vs, int K, Range g, double (&out)[2])
    {
        const int i = row(0), q = threadIdx.x & 3, n = (threadIdx.x & 31) >> 2;
        double c0 = 0.0, c1 = 0.0, e0 = 0.0, e1 = 0.0;
        out[0] = out[1] = 0.0;
        const int t8 = 8 * (int)(threadIdx.x >> 5);   // this warp's rows t8 .. t8 + 7
        if (t8 >= g.rows) return;
        const int K4 = min((K + 3) & ~3, g.tri < 0 ? t8 + 8 : 64);
#pragma unroll 2
        for (int k = g.tri > 0 ? t8 : 0; k < K4; k += 8) {
            dmma_f64(c0, c1, A[kT ? idx_t(k + q, i) : idx_n(i, k + q)], Vs[vidx(k + q, n)]);
            if (k + 4 < K4)
                dmma_f64(e0, e1, A[kT ? idx_t(k + 4 + q, i) : idx_n(i, k + 4 + q)], Vs[vidx(k + 4 + q, n)]);
        }
        out[0] = c0 + e0;
        out[1] = c1 + e1;
    }
    static __device__ __forceinline__ void mul_n(const double *A, const double *Vs, int K, Range g, double *, double (&out)[2])
    {
        mul<false>(A, Vs, K, g, out);
    }
    static __device__ __forceinline__ void mul_t(const double *A, const double *Vs, int K, Range g, double *, double (&out)[2])
    {
        mul<true>(A, Vs, K, g, out);
    }
};

// FP64, one column: row tid % 64, part tid / 64 of k.
template <>
struct Prod<double, 1> {
    static constexpr int kOut = 1, kMat = 64 * 65, kRed = 256;
    static __device__ __forceinline__ int idx_n(int i, int k) { return k * 64 + i; }
    static __device__ __forceinline__ int idx_t(int k, int i) { return i * 65 + k; }
    static __device__ __forceinline__ int vidx(int k, int) { return k; }
    static __device__ __forceinline__ int col(int) { return 0; }
    static __device__ __forceinline__ int row(int)
    {
        return threadIdx.x;   // threads 64 .. hold no result
    }
    template <bool kT>
    static __device__ __forceinline__ void mul(const double *A, const double *Vs, int K, Range g, double *red,
                                               double (&out)[1])
    {
        // by warps of 32 rows: the k range of their triangle, none past the rows
        const int i = threadIdx.x & 63, lo = i & 32;
        const int ka = g.tri > 0 ? lo : 0, kb = lo >= g.rows ? ka : min(K, g.tri < 0 ? lo + 32 : 64);
        const int span = (max(kb - ka, 0) + 3) / 4, k0 = ka + (threadIdx.x >> 6) * span, k1 = min(kb, k0 + span);
        double s0 = 0.0, s1 = 0.0;
        int k = k0;
        for (; k + 1 < k1; k += 2) {
            s0 = fma(A[kT ? idx_t(k, i) : idx_n(i, k)], Vs[k], s0);
            s1 = fma(A[kT ? idx_t(k + 1, i) : idx_n(i, k + 1)], Vs[k + 1], s1);
        }
        if (k < k1) s0 = fma(A[kT ? idx_t(k, i) : idx_n(i, k)], Vs[k], s0);
        red[threadIdx.x] = s0 + s1;
        __syncthreads();
        out[0] = threadIdx.x < 64 ? (red[threadIdx.x] + red[64 + threadIdx.x]) +
                                        (red[128 + threadIdx.x] + red[192 + threadIdx.x])
                                  : 0.0;
    }
    static __device__ __forceinline__ void mul_n(const double *A, const double *Vs, int K, Range g, double *red, double (&out)[1])
    {
        mul<false>(A, Vs, K, g, red, out);
    }
    static __device__ __forceinline__ void mul_t(const double *A, const double *Vs, int K, Range g, double *red, double (&out)[1])
    {
        mul<true>(A, Vs, K, g, red, out);
    }
};

// Staging of rows x cols (rows rounded up to 8, columns to 4) of a
// column-major source (leading dimension ld) by asynchronous copies; (i, k)
// outside [0, rows) x [0, cols) as zeros.  kMask 0: everything; 1: lower triangle;
// 2: strictly lower, ones on the diagonal; 3: upper triangle ((i, k) counted
// from row io, column ko of the diagonal block).
enum Mask { kAll = 0, kLower = 1, kUnitLower = 2, kUpper = 3 };
template <typename P, bool kT, typename T>
__device__ __forceinline__ void stage_mat(T *dst, const T *src, int64_t ld, int rows, int cols, Mask mask, int io = 0,
                                          int ko = 0)
{
    const int nk = (cols + 3) & ~3, i = threadIdx.x & 63;
    if (i >= ((rows + 7) & ~7)) {
        stage_commit();   // an empty group, to count with the others
        return;
    }
    const bool in = i < rows;
    for (int k = threadIdx.x >> 6; k < nk; k += kQThreads / 64) {
        const int d = (i + io) - (k + ko);
        T *to = dst + (kT ? P::idx_t(i, k) : P::idx_n(i, k));
        if (mask == kUnitLower && d == 0) {
            *to = (T)1;
            continue;
        }
        const bool ok = in && k < cols && (mask == kAll || (mask == kUpper ? d <= 0 : d >= 0));
        cp_async_elem(to, ok ? src + i + (int64_t)k * ld : src, ok);
    }
    stage_commit();
}

// Vs(k, c) = V[f + k, c0 + c] for k < w (zeros past nc, and rows up to the
// next multiple of 8), read through L2, a thread's loads before its stores.
template <typename P, int NC, typename T>
__device__ __forceinline__ void load_vec(T *Vs, const T *V, int64_t f, int w, int nc, int64_t n, int c0)
{
    constexpr int kC = (NC + kQThreads / 64 - 1) / (kQThreads / 64);   // columns a thread
    const int c1 = threadIdx.x >> 6, wp = (w + 7) & ~7;
    for (int k = threadIdx.x & 63; k < wp; k += 64) {
        T v[kC];
#pragma unroll
        for (int q = 0; q < kC; ++q) {
            const int c = c1 + 4 * q;
            v[q] = k < w && c < nc ? ld_l2(V + f + k + (int64_t)(c0 + c) * n) : (T)0;
        }
#pragma unroll
        for (int q = 0; q < kC; ++q)
            if (c1 + 4 * q < NC) Vs[P::vidx(k, c1 + 4 * q)] = v[q];
    }
}

constexpr int kQRhs = 16;                   // right-hand sides per pass of the 16-column kernels

// Rows [r0, r0 + 64) of a panel's off-diagonal block to dst[k * ld + r]
// (rows past the panel as zeros).
template <typename T>
__device__ __forceinline__ void stage_chunk(T *dst, int ld, const T *Pn, int h, int w, int r0, int nr)
{
    const int total = w * 64;
    for (int e = threadIdx.x; e < total; e += kQThreads) {
        const int r = e & 63, k = e >> 6;
        const bool ok = r < nr;
        cp_async_elem(dst + k * ld + r, ok ? Pn + r0 + r + (int64_t)k * h : Pn, ok);
    }
    stage_commit();
}

// dst[e] = src[e], e < total (a diagonal block's inverse, column-major).
template <typename T>
__device__ __forceinline__ void stage_copy(T *dst, const T *src, int total)
{
    for (int e = threadIdx.x; e < total; e += kQThreads) cp_async_elem(dst + e, src + e, true);
    stage_commit();
}

// Right-hand-side blocks in shared memory hold kQRhs columns per row, the
// four column quads of row k in the order q ^ ((k >> 1) & 3): a thread
// reads its quad of one row with one vector load (the same address across
// a warp), and the column-wise staging stores spread over eight banks.
__device__ __forceinline__ int vslot(int k, int c)
{
    return k * kQRhs + ((((c >> 2) ^ (k >> 1)) & 3) << 2) + (c & 3);
}
template <typename T>
__device__ __forceinline__ void ld_quad(const T *Vs, int k, int g, T (&v)[4])
{
    const T *p = Vs + vslot(k, 4 * g);
    if constexpr (sizeof(T) == 4) {
        const float4 x = *reinterpret_cast<const float4 *>(p);
        v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
    } else {
        const double2 x = *reinterpret_cast<const double2 *>(p);
        const double2 y = *reinterpret_cast<const double2 *>(p + 2);
        v[0] = x.x; v[1] = x.y; v[2] = y.x; v[3] = y.y;
    }
}
template <typename T>
__device__ __forceinline__ void st_quad(T *Vs, int k, int g, const T (&v)[4])
{
    T *p = Vs + vslot(k, 4 * g);
    if constexpr (sizeof(T) == 4) {
        *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
        *reinterpret_cast<double2 *>(p) = make_double2(v[0], v[1]);
        *reinterpret_cast<double2 *>(p + 2) = make_double2(v[2], v[3]);
    }
}

// Vs(k, c) = V[f + k, c0 + c] for k < w (zero past nc), read through L2.
template <typename T>
__device__ __forceinline__ void stage_vec(T *Vs, const T *V, int64_t f, int w, int nc, int64_t n, int c0)
{
    constexpr int NB = 4;
    const int total = w * kQRhs;
    for (int base = threadIdx.x; base < total; base += kQThreads * NB) {
        T v[NB];
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            const int e = base + q * kQThreads, k = e % w, c = e / w;
            v[q] = (e < total && c < nc) ? ld_l2(V + f + k + (int64_t)(c0 + c) * n) : (T)0;
        }
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            const int e = base + q * kQThreads;
            if (e < total) Vs[vslot(e % w, e / w)] = v[q];
        }
    }
}

// Xs(r, c) = X[row_r, c0 + c] (r < 64, zero past nr or nc); the thread's
// rows are all r = tid & 63, whose index `row` it loaded beforehand.
template <typename T>
__device__ __forceinline__ void stage_rows(T *Xs, const T *X, int64_t row, int nr, int nc, int64_t n, int c0)
{
    constexpr int NC = kQRhs / (kQThreads / 64);   // columns per thread
    const int r = threadIdx.x & 63, cf = threadIdx.x >> 6;
    T v[NC];
#pragma unroll
    for (int q = 0; q < NC; ++q) {
        const int c = cf + q * (kQThreads / 64);
        v[q] = (r < nr && c < nc) ? ld_l2(X + row + (int64_t)(c0 + c) * n) : (T)0;
    }
#pragma unroll
    for (int q = 0; q < NC; ++q) Xs[vslot(r, cf + q * (kQThreads / 64))] = v[q];
}

// Y[row_r, c0 + 4g + u] -= sum_k Lc(r, k) Zs(k, 4g + u) for thread (r, g) =
// (tid & 63, tid >> 6); Lc staged [k * 64 + r].
template <typename T>
__device__ __forceinline__ void fwd_chunk_pass(const T *Lc, const T *Zs, int w, int nr, int nc, int64_t row,
                                               T *Y, int64_t n, int c0)
{
    const int r = threadIdx.x & 63, g = threadIdx.x >> 6;
    if (r >= nr) return;
    T acc[4] = {(T)0, (T)0, (T)0, (T)0};
#pragma unroll 4
    for (int k = 0; k < w; ++k) {
        const T l = Lc[k * 64 + r];
        T z[4];
        ld_quad(Zs, k, g, z);
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[u] += l * z[u];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int c = 4 * g + u;
        if (c < nc) atomicAdd(Y + row + (int64_t)(c0 + c) * n, -acc[u]);
    }
}

// acc[u] += sum over r of Lc(r, k) Xs(r, 4g + u), Lc staged [k * 65 + r].
template <typename T>
__device__ __forceinline__ void chunk_dot4(const T *Lc, const T *Xs, int k, int g, T (&acc)[4])
{
#pragma unroll 4
    for (int r = 0; r < 64; ++r) {
        const T l = Lc[k * 65 + r];
        T x[4];
        ld_quad(Xs, r, g, x);
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[u] += l * x[u];
    }
}

}  // namespace

// Shared memory: two 64 x 64 matrices, two vectors of the widest panel (at
// least 64 rows) x NC, the partial sums.  Four CTAs an SM in FP32 (one more
// measured slower, where registers spill), three for one FP64 column (two
// measured slower), two for eight, as many as 82 KB of shared memory let on.
template <typename T, int NC>
constexpr int kCtas = sizeof(T) == 4 ? 4 : NC == 1 ? 3 : 2;

template <typename T, int NC>
__global__ void __launch_bounds__(kQThreads, kCtas<T, NC>)
    fwd_queue_kernel(DevPlan p, SweepQueue q, const T *__restrict__ Dinv, int unit,
                     const T *__restrict__ L, T *Y, T *Z, int nrhs)
{
    using P = Prod<T, NC>;
    extern __shared__ __align__(16) unsigned char smraw[];
    T *const mat = reinterpret_cast<T *>(smraw);   // two matrices, block b in b & 1
    T *vec = mat + 2 * P::kMat, *vec2 = vec + q.vec_rows * NC, *red = vec2 + 64 * NC;
    __shared__ int s_next;
    __shared__ SweepItem s_item[2];
    __shared__ int32_t s_row[64];
    const int tid = threadIdx.x;
    const int64_t n = p.n;
    const int total = q.nitems * q.groups;
    // the items are handed out one ahead: while an item is worked on, the
    // counter gives the next one's place and its description is read
    auto describe = [&](int idx) {
        const SweepItem *at = q.desc + (q.groups == 1 ? idx : idx / q.groups);
        return tid < 4 && idx < total ? reinterpret_cast<const int4 *>(at)[tid] : make_int4(0, 0, 0, 0);
    };
    if (tid == 0) s_next = atomicAdd(q.head, 1);
    __syncthreads();
    int idx = s_next;
    {
        const int4 d = describe(idx);
        if (tid < 4) reinterpret_cast<int4 *>(s_item)[tid] = d;
    }
    __syncthreads();
    for (int turn = 0; idx < total; turn ^= 1) {
        const SweepItem &it = s_item[turn];   // read as needed (registers are short)
        const int grp = q.groups == 1 ? 0 : idx % q.groups;
        int next = 0;
        if (tid == 0) next = atomicAdd(q.head, 1);   // not waited for here
        int32_t *cnt = q.cnt + (int64_t)grp * p.npanels, *flag = q.flag + (int64_t)grp * p.npanels;
        const bool isp = it.panel_item, chunk = it.nr > 0;
        const int pid = it.panel, w = it.w, h = it.h, nr = it.nr, nb = (w + 63) / 64;
        const int64_t f = it.f;
        const T *Mi = Dinv + it.inv, *Lp = L + it.chunk;
        // the item's 64 x 64 blocks in order of use: a panel's inverse by block
        // rows, then (or, for a chunk item, only) the chunk by block columns
        const int ninv = isp ? nb * (nb + 1) / 2 : 0, nall = ninv + (chunk ? nb : 0);
        auto stage = [&](int b) {
            T *dst = mat + (b & 1) * P::kMat;
            if (b < ninv) {
                int ib = 0, kb = b;
                while (kb > ib) kb -= ++ib;
                stage_mat<P, false>(dst, Mi + 64 * ib + (int64_t)64 * kb * w, w, min(64, w - 64 * ib),
                                    min(64, w - 64 * kb), unit ? kUnitLower : kLower, 64 * ib, 64 * kb);
            } else {
                const int kb = b - ninv;
                stage_mat<P, false>(dst, Lp + (int64_t)64 * kb * h, h, nr, min(64, w - 64 * kb), kAll);
            }
        };
        stage(0);
        if (nall > 1) stage(1);
        const int32_t row = (tid & 63) < nr ? p.rows[it.rows + (tid & 63)] : 0;   // not waited for here
        if (tid == 0) s_next = next;
        if (!cta_wait(isp ? cnt + pid : flag + pid, nullptr, 1, isp ? it.need : 1, q.err, q.spin_limit)) {
            stage_wait();   // no copy left in flight on the way out
            return;
        }
        if (tid < 64) s_row[tid] = row;
        idx = s_next;
        const int4 ahead = describe(idx);
        bool first = true;
        for (int c0 = grp * NC; c0 < nrhs; c0 += q.groups * NC, first = false) {
            const int nc = min(NC, nrhs - c0);
            if (!first) {
                stage(0);
                if (nall > 1) stage(1);
            }
            load_vec<P, NC>(vec, isp ? Y : Z, f, w, nc, n, c0);
            T acc[P::kOut];
            int ib = 0, kb = 0;
            for (int b = 0; b < nall; ++b) {
                if (b + 1 < nall) stage_wait_but<1>();
                else stage_wait();
                __syncthreads();
                T out[P::kOut];
                const bool inv = b < ninv;
                const int k = inv ? kb : b - ninv;
                // a chunk taken along multiplies Z_p, which the inverse left in vec2 (one block)
                const Range g{inv ? min(64, w - 64 * ib) : nr, inv && kb == ib ? -1 : 0};
                P::mul_n(mat + (b & 1) * P::kMat, (isp && !inv) ? vec2 : vec + P::vidx(64 * k, 0), min(64, w - 64 * k),
                         g, red, out);
                const bool start = inv ? kb == 0 : k == 0, end = inv ? kb == ib : k == nb - 1;
#pragma unroll
                for (int o = 0; o < P::kOut; ++o) acc[o] = start ? out[o] : acc[o] + out[o];
                if (end) {
#pragma unroll
                    for (int o = 0; o < P::kOut; ++o) {
                        const int i = P::row(o), c = P::col(o);
                        if (i >= 64) continue;
                        if (inv) {
                            if (64 * ib + i < w && c < nc) Z[f + 64 * ib + i + (int64_t)(c0 + c) * n] = acc[o];
                            if (chunk) vec2[P::vidx(i, c)] = acc[o];   // (rows past w: zero)
                        } else if (i < nr && c < nc) {
                            atomicAdd(Y + s_row[i] + (int64_t)(c0 + c) * n, -acc[o]);
                        }
                    }
                }
                if (inv && kb++ == ib) {
                    kb = 0;
                    ++ib;
                }
                __syncthreads();
                if (b + 2 < nall) stage(b + 2);
            }
        }
        if (tid < 4) reinterpret_cast<int4 *>(s_item + (turn ^ 1))[tid] = ahead;
        cta_release(isp ? flag + pid : nullptr, cnt, q.tgt + it.t0, it.t1 - it.t0);
    }
}

// lu: 0 Cholesky (M = Linv^T), 1 LU (M = U^{-1}), 2 LDL^T
// (X_p = l^{-T} (D^{-1} Z_p - Tacc_p), 1/d on the diagonal of Dinv).
template <typename T, int NC>
__global__ void __launch_bounds__(kQThreads, kCtas<T, NC>)
    bwd_queue_kernel(DevPlan p, SweepQueue q, const T *__restrict__ Dinv, int lu,
                     const T *__restrict__ Lop, const T *__restrict__ Z, T *Tacc, T *X, int nrhs)
{
    using P = Prod<T, NC>;
    extern __shared__ __align__(16) unsigned char smraw[];
    T *const mat = reinterpret_cast<T *>(smraw);   // two matrices, block b in b & 1
    T *vec = mat + 2 * P::kMat, *vec2 = vec + q.vec_rows * NC, *red = vec2 + 64 * NC;
    __shared__ int s_next;
    __shared__ SweepItem s_item[2];
    const int tid = threadIdx.x;
    const int64_t n = p.n;
    const int total = q.nitems * q.groups;
    // the items are handed out one ahead: while an item is worked on, the
    // counter gives the next one's place and its description is read
    auto describe = [&](int idx) {
        const SweepItem *at = q.desc + (q.groups == 1 ? idx : idx / q.groups);
        return tid < 4 && idx < total ? reinterpret_cast<const int4 *>(at)[tid] : make_int4(0, 0, 0, 0);
    };
    if (tid == 0) s_next = atomicAdd(q.head, 1);
    __syncthreads();
    int idx = s_next;
    {
        const int4 d = describe(idx);
        if (tid < 4) reinterpret_cast<int4 *>(s_item)[tid] = d;
    }
    __syncthreads();
    for (int turn = 0; idx < total; turn ^= 1) {
        const SweepItem &it = s_item[turn];   // read as needed (registers are short)
        const int grp = q.groups == 1 ? 0 : idx % q.groups;
        int next = 0;
        if (tid == 0) next = atomicAdd(q.head, 1);   // not waited for here
        int32_t *cnt = q.cnt + (int64_t)grp * p.npanels, *flag = q.flag + (int64_t)grp * p.npanels;
        const bool isp = it.panel_item, chunk = it.nr > 0;
        const int pid = it.panel, w = it.w, h = it.h, nr = it.nr, nb = (w + 63) / 64;
        const int64_t f = it.f;
        const T *Mi = Dinv + it.inv, *Lp = Lop + it.chunk;
        // the chunk's block columns first, then the inverse: block row ib of
        // X_p takes the blocks kb = ib .. of M
        const int nchk = chunk ? nb : 0, nall = nchk + (isp ? nb * (nb + 1) / 2 : 0);
        auto block = [&](int b, int &ib, int &kb) {
            ib = 0;
            kb = b - nchk;
            while (kb >= nb - ib) {
                kb -= nb - ib;
                ++ib;
            }
            kb += ib;
        };
        auto stage = [&](int b) {
            T *dst = mat + (b & 1) * P::kMat;
            if (b < nchk) {
                stage_mat<P, true>(dst, Lp + (int64_t)64 * b * h, h, nr, min(64, w - 64 * b), kAll);
                return;
            }
            int ib, kb;
            block(b, ib, kb);
            const int ni = min(64, w - 64 * ib), nk = min(64, w - 64 * kb);
            if (lu == 1) stage_mat<P, false>(dst, Mi + 64 * ib + (int64_t)64 * kb * w, w, ni, nk, kUpper, 64 * ib, 64 * kb);
            else stage_mat<P, true>(dst, Mi + 64 * kb + (int64_t)64 * ib * w, w, nk, ni, lu == 2 ? kUnitLower : kLower,
                                    64 * kb, 64 * ib);
        };
        stage(0);
        if (nall > 1) stage(1);
        const int32_t row = (tid & 63) < nr ? p.rows[it.rows + (tid & 63)] : 0;
        if (tid == 0) s_next = next;
        const int t0 = it.t0, m = it.t1 - it.t0;
        {
            // one wait: threads < m on the panels owning the chunk's rows,
            // thread m (of a panel item) on the panel's own chunks
            int ok = 1;
            if (tid < m) ok = wait_geq(flag + q.tgt[t0 + tid], 1, q.err, q.spin_limit);
            else if (tid == m && isp) ok = wait_geq(cnt + pid, it.need, q.err, q.spin_limit);
            if (!__syncthreads_and(ok)) {
                stage_wait();
                return;
            }
        }
        idx = s_next;
        const int4 ahead = describe(idx);
        bool first = true;
        for (int c0 = grp * NC; c0 < nrhs; c0 += q.groups * NC, first = false) {
            const int nc = min(NC, nrhs - c0);
            if (!first) {
                stage(0);
                if (nall > 1) stage(1);
            }
            // vec2 = the chunk's rows of X, vec = Z_p (LDL^T: D^{-1} Z_p) - Tacc_p:
            // every load through L2 is issued before the first store waits for one
            {
                constexpr int kC = (NC + kQThreads / 64 - 1) / (kQThreads / 64);
                const int r = tid & 63, c1 = tid >> 6, wp = isp ? (w + 7) & ~7 : 0;
                T xv[kC];
                if (chunk) {
#pragma unroll
                    for (int u = 0; u < kC; ++u) {
                        const int c = c1 + 4 * u;
                        xv[u] = r < nr && c < nc ? ld_l2(X + row + (int64_t)(c0 + c) * n) : (T)0;
                    }
                    if constexpr (kC == 1)   // (one column a thread: nothing to batch)
                        if (c1 < NC) vec2[P::vidx(r, c1)] = xv[0];
                }
                for (int k = r; k < wp; k += 64) {
                    T zv[kC], tv[kC];
#pragma unroll
                    for (int u = 0; u < kC; ++u) {
                        const int c = c1 + 4 * u;
                        const bool in = k < w && c < nc;
                        const int64_t at = f + k + (int64_t)(c0 + c) * n;
                        tv[u] = in ? ld_l2(Tacc + at) : (T)0;
                        zv[u] = in ? Z[at] : (T)0;
                    }
                    const T dg = lu == 2 && k < w ? Mi[k + (int64_t)k * w] : (T)1;
#pragma unroll
                    for (int u = 0; u < kC; ++u)
                        if (c1 + 4 * u < NC) vec[P::vidx(k, c1 + 4 * u)] = (lu == 2 ? zv[u] * dg : zv[u]) - tv[u];
                }
                if (kC > 1 && chunk) {
#pragma unroll
                    for (int u = 0; u < kC; ++u)
                        if (c1 + 4 * u < NC) vec2[P::vidx(r, c1 + 4 * u)] = xv[u];
                }
            }
            T acc[P::kOut];
            for (int b = 0; b < nall; ++b) {
                if (b + 1 < nall) stage_wait_but<1>();
                else stage_wait();
                __syncthreads();
                T out[P::kOut];
                if (b < nchk) {
                    const Range g{min(64, w - 64 * b), 0};
                    P::mul_t(mat + (b & 1) * P::kMat, vec2, nr, g, red, out);
#pragma unroll
                    for (int o = 0; o < P::kOut; ++o) {
                        const int i = P::row(o), c = P::col(o), k = 64 * b + i;
                        if (i >= 64 || k >= w) continue;
                        if (isp) vec[P::vidx(k, c)] -= out[o];
                        else if (c < nc) atomicAdd(Tacc + f + k + (int64_t)(c0 + c) * n, out[o]);
                    }
                } else {
                    int ib, kb;
                    block(b, ib, kb);
                    const T *v = vec + P::vidx(64 * kb, 0);
                    const int K = min(64, w - 64 * kb);
                    const Range g{min(64, w - 64 * ib), kb == ib ? 1 : 0};
                    if (lu == 1) P::mul_n(mat + (b & 1) * P::kMat, v, K, g, red, out);
                    else P::mul_t(mat + (b & 1) * P::kMat, v, K, g, red, out);
#pragma unroll
                    for (int o = 0; o < P::kOut; ++o) acc[o] = kb == ib ? out[o] : acc[o] + out[o];
                    if (kb == nb - 1) {
#pragma unroll
                        for (int o = 0; o < P::kOut; ++o) {
                            const int c = P::col(o), i = P::row(o);
                            if (i < 64 && 64 * ib + i < w && c < nc)
                                X[f + 64 * ib + i + (int64_t)(c0 + c) * n] = acc[o];
                        }
                    }
                }
                __syncthreads();
                if (b + 2 < nall) stage(b + 2);
            }
        }
        if (tid < 4) reinterpret_cast<int4 *>(s_item + (turn ^ 1))[tid] = ahead;
        if (isp) cta_release(flag + pid, nullptr, nullptr, 0);
        else cta_release(nullptr, cnt + pid, nullptr, 1);
    }
}

// FP32, more than four right-hand sides: 16 columns a pass, threads as (row,
// column quad) = (tid & 63, tid >> 6), each sum whole (the triangles' zero
// halves are left out).  Shared memory: A (q.mat_elems: a diagonal block, or a
// chunk), B (q.matb_elems: the chunk a panel item takes along), a vector of
// q.vec_elems and, when panel items take chunks along, a second one.  Five CTAs
// an SM (41.5 KB of shared memory each for 64-wide panels, at most 48
// registers a thread), so that more items' loads are in flight.  64^3
// diffusion, 16 right-hand sides, a forward and a backward sweep: 4.48 ms,
// 4.57 with split sums as above.
__global__ void __launch_bounds__(kQThreads, 5)
    fwd_rhs16_kernel(DevPlan p, SweepQueue q, const RowChunk *__restrict__ chunks, const float *__restrict__ Dinv,
                     int unit, const float *__restrict__ L, float *Y, float *Z, int nrhs)
{
    using T = float;
    extern __shared__ __align__(16) unsigned char smraw[];
    T *matA = reinterpret_cast<T *>(smraw);
    T *matB = matA + q.mat_elems;
    T *vec = matB + q.matb_elems;
    T *vec2 = vec + q.vec_elems;
    __shared__ int s_next;
    const int tid = threadIdx.x, rt = tid & 63, g = tid >> 6;
    const int64_t n = p.n;
    if (tid == 0) s_next = atomicAdd(q.head, 1);
    __syncthreads();
    for (;;) {
        const int idx = s_next;
        __syncthreads();
        if (idx >= q.nitems) return;
        const int item = q.items[idx];
        if (tid == 0) s_next = atomicAdd(q.head, 1);   // the next item, fetched early
        if (item < 0) {
            // panel: Z_p = Linv_p Y_p (LU / LDL^T: unit Linv), then its
            // first chunk when it takes one along
            const int pid = -item - 1;
            const int w = p.pw[pid], h = p.ph[pid];
            const int64_t f = p.pfcol[pid];
            const T *Mi = Dinv + p.pinv[pid];
            const int mc = q.merge[pid];
            stage_copy(matA, Mi, w * w);   // column-major, ld w
            int nr = 0;
            int64_t row = 0;
            if (mc >= 0) {
                nr = min(64, h - w);
                stage_chunk(matB, 64, L + p.pval[pid], h, w, w, nr);
                if (rt < nr) row = p.rows[p.prow[pid] + w + rt];
            }
            if (!cta_wait(q.cnt + pid, nullptr, 1, q.need[pid], q.err, q.spin_limit)) {
                stage_wait();   // no copy left in flight on the way out
                return;
            }
            for (int c0 = 0; c0 < nrhs; c0 += kQRhs) {
                const int nc = min(kQRhs, nrhs - c0);
                stage_vec(vec, Y, f, w, nc, n, c0);
                stage_wait();
                __syncthreads();
                for (int i = rt; i < w; i += 64) {
                    T acc[4];
                    if (unit) ld_quad(vec, i, g, acc);
                    else acc[0] = acc[1] = acc[2] = acc[3] = (T)0;
                    const int kl = unit ? i : i + 1;
#pragma unroll 4
                    for (int k = 0; k < kl; ++k) {
                        const T a = matA[i + k * w];
                        T y[4];
                        ld_quad(vec, k, g, y);
#pragma unroll
                        for (int u = 0; u < 4; ++u) acc[u] += a * y[u];
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int c = 4 * g + u;
                        if (c < nc) Z[f + i + (int64_t)(c0 + c) * n] = acc[u];
                    }
                    if (mc >= 0) st_quad(vec2, i, g, acc);
                }
                __syncthreads();
                if (mc >= 0) {
                    fwd_chunk_pass(matB, vec2, w, nr, nc, row, Y, n, c0);
                    __syncthreads();
                }
            }
            const int t0 = mc >= 0 ? q.tptr[mc] : 0, t1 = mc >= 0 ? q.tptr[mc + 1] : 0;
            cta_release(q.flag + pid, q.cnt, q.tgt + t0, t1 - t0);
        } else {
            // chunk: Y[rows] -= L(rows, :) Z_p
            const RowChunk ch = chunks[item];
            const int pid = ch.panel;
            const int w = p.pw[pid], h = p.ph[pid];
            const int64_t f = p.pfcol[pid];
            const int nr = min(64, h - ch.r0);
            stage_chunk(matA, 64, L + p.pval[pid], h, w, ch.r0, nr);
            const int64_t row = rt < nr ? p.rows[p.prow[pid] + ch.r0 + rt] : 0;
            if (!cta_wait(q.flag + pid, nullptr, 1, 1, q.err, q.spin_limit)) {
                stage_wait();   // no copy left in flight on the way out
                return;
            }
            for (int c0 = 0; c0 < nrhs; c0 += kQRhs) {
                const int nc = min(kQRhs, nrhs - c0);
                stage_vec(vec, Z, f, w, nc, n, c0);
                stage_wait();
                __syncthreads();
                fwd_chunk_pass(matA, vec, w, nr, nc, row, Y, n, c0);
                __syncthreads();
            }
            const int t0 = q.tptr[item], t1 = q.tptr[item + 1];
            cta_release(nullptr, q.cnt, q.tgt + t0, t1 - t0);
        }
    }
}

// lu: 0 Cholesky (M = Linv^T), 1 LU (M = U^{-1}), 2 LDL^T
// (X_p = l^{-T} (D^{-1} Z_p - Tacc_p), 1/d on the diagonal of Dinv).
__global__ void __launch_bounds__(kQThreads, 5)
    bwd_rhs16_kernel(DevPlan p, SweepQueue q, const RowChunk *__restrict__ chunks, const float *__restrict__ Dinv,
                     int lu, const float *__restrict__ Lop, const float *__restrict__ Z, float *Tacc, float *X, int nrhs)
{
    using T = float;
    extern __shared__ __align__(16) unsigned char smraw[];
    T *matA = reinterpret_cast<T *>(smraw);
    T *matB = matA + q.mat_elems;
    T *vec = matB + q.matb_elems;
    T *vec2 = vec + q.vec_elems;
    __shared__ int s_next;
    const int tid = threadIdx.x, rt = tid & 63, g = tid >> 6;
    const int64_t n = p.n;
    if (tid == 0) s_next = atomicAdd(q.head, 1);
    __syncthreads();
    for (;;) {
        const int idx = s_next;
        __syncthreads();
        if (idx >= q.nitems) return;
        const int item = q.items[idx];
        if (tid == 0) s_next = atomicAdd(q.head, 1);
        if (item < 0) {
            // panel: X_p = M (Z_p - Tacc_p - Lc^T X[rows of its first chunk])
            const int pid = -item - 1;
            // ld odd, so that a warp's rows i of M(i, k) = matA[k + i ld] fall
            // in distinct banks
            const int w = p.pw[pid], h = p.ph[pid], ld = (w & 1) ? w + 2 : w + 1;
            const int64_t f = p.pfcol[pid];
            const T *Mi = Dinv + p.pinv[pid];
            const int mc = q.merge[pid];
            // the stored inverse as it is, column-major with leading dimension ld (by
            // asynchronous copies): M(i, k) is matA[i + k ld] for LU (U^{-1})
            // and matA[k + i ld] = Linv(k, i) otherwise; only k >= i is read
            for (int e = tid; e < w * w; e += kQThreads) cp_async_elem(matA + (e % w) + (e / w) * ld, Mi + e, true);
            stage_commit();
            int nr = 0, t0 = 0, m = 0;
            int64_t row = 0;
            if (mc >= 0) {
                nr = min(64, h - w);
                stage_chunk(matB, 65, Lop + p.pval[pid], h, w, w, nr);
                if (rt < nr) row = p.rows[p.prow[pid] + w + rt];
                t0 = q.tptr[mc];
                m = q.tptr[mc + 1] - t0;
            }
            // the first pass's Z_p (LDL^T: D^{-1} Z_p) is fixed: staged
            // before the wait, Tacc_p subtracted after it by the same threads
            const int nc0 = min(kQRhs, nrhs);
            for (int base = tid; base < w * kQRhs; base += kQThreads * 4) {
                T v[4], dg[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int e = base + q * kQThreads, k = e % w, c = e / w;
                    const bool ok = e < w * kQRhs && c < nc0;
                    v[q] = ok ? Z[f + k + (int64_t)c * n] : (T)0;
                    dg[q] = (ok && lu == 2) ? Mi[k + k * w] : (T)1;
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int e = base + q * kQThreads;
                    if (e < w * kQRhs) vec[vslot(e % w, e / w)] = lu == 2 ? v[q] * dg[q] : v[q];
                }
            }
            // one wait: threads < m on the panels owning the chunk's rows,
            // thread m on the panel's own chunks
            {
                int ok = 1;
                if (tid < m) ok = wait_geq(q.flag + q.tgt[t0 + tid], 1, q.err, q.spin_limit);
                else if (tid == m) ok = wait_geq(q.cnt + pid, q.need[pid], q.err, q.spin_limit);
                if (!__syncthreads_and(ok)) {
                    stage_wait();
                    return;
                }
            }
            for (int c0 = 0; c0 < nrhs; c0 += kQRhs) {
                const int nc = min(kQRhs, nrhs - c0);
                if (c0 > 0) {
                    __syncthreads();
                    for (int e = tid; e < w * kQRhs; e += kQThreads) {
                        const int k = e % w, c = e / w;
                        const int64_t gk = f + k + (int64_t)(c0 + c) * n;
                        vec[vslot(k, c)] = c < nc ? (lu == 2 ? Z[gk] * Mi[k + k * w] : Z[gk]) : (T)0;
                    }
                }
                // vec -= Tacc_p, and the chunk's rows of X: both read through
                // L2 in one batch (the X rows' loads go first, their stores
                // after Tacc's loads are in flight)
                constexpr int NCX = kQRhs / (kQThreads / 64);
                const int xr = tid & 63, xc = tid >> 6;
                T xv[NCX];
                if (mc >= 0) {
#pragma unroll
                    for (int q = 0; q < NCX; ++q) {
                        const int c = xc + q * (kQThreads / 64);
                        xv[q] = (xr < nr && c < nc) ? ld_l2(X + row + (int64_t)(c0 + c) * n) : (T)0;
                    }
                }
                for (int base = tid; base < w * kQRhs; base += kQThreads * 4) {
                    T t[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int e = base + q * kQThreads, k = e % w, c = e / w;
                        t[q] = (e < w * kQRhs && c < nc) ? ld_l2(Tacc + f + k + (int64_t)(c0 + c) * n) : (T)0;
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int e = base + q * kQThreads;
                        if (e < w * kQRhs && e / w < nc) vec[vslot(e % w, e / w)] -= t[q];
                    }
                }
                if (mc >= 0) {
#pragma unroll
                    for (int q = 0; q < NCX; ++q) vec2[vslot(xr, xc + q * (kQThreads / 64))] = xv[q];
                }
                stage_wait();
                __syncthreads();
                if (mc >= 0) {   // vec -= Lc^T X[rows]
                    for (int k = rt; k < w; k += 64) {
                        T part[4] = {(T)0, (T)0, (T)0, (T)0};
                        chunk_dot4(matB, vec2, k, g, part);
                        T v[4];
                        ld_quad(vec, k, g, v);
#pragma unroll
                        for (int u = 0; u < 4; ++u) v[u] -= part[u];
                        st_quad(vec, k, g, v);
                    }
                    __syncthreads();
                }
                for (int i = rt; i < w; i += 64) {
                    T acc[4] = {(T)0, (T)0, (T)0, (T)0};
                    int k = i;
                    if (lu == 2) {   // LDL^T: l^{-T} has a unit diagonal
                        ld_quad(vec, i, g, acc);
                        ++k;
                    }
                    const int sa = lu == 1 ? 1 : ld, sk = lu == 1 ? ld : 1;   // M(i, k) = matA[i sa + k sk]
#pragma unroll 4
                    for (; k < w; ++k) {
                        const T a = matA[i * sa + k * sk];
                        T v[4];
                        ld_quad(vec, k, g, v);
#pragma unroll
                        for (int u = 0; u < 4; ++u) acc[u] += a * v[u];
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int c = 4 * g + u;
                        if (c < nc) X[f + i + (int64_t)(c0 + c) * n] = acc[u];
                    }
                }
            }
            cta_release(q.flag + pid, nullptr, nullptr, 0);
        } else {
            // chunk: Tacc_p += Lop(rows, :)^T X[rows]
            const RowChunk ch = chunks[item];
            const int pid = ch.panel;
            const int w = p.pw[pid], h = p.ph[pid];
            const int64_t f = p.pfcol[pid];
            const int nr = min(64, h - ch.r0);
            stage_chunk(matA, 65, Lop + p.pval[pid], h, w, ch.r0, nr);
            const int64_t row = rt < nr ? p.rows[p.prow[pid] + ch.r0 + rt] : 0;
            const int t0 = q.tptr[item], t1 = q.tptr[item + 1];
            if (!cta_wait(q.flag, q.tgt + t0, t1 - t0, 1, q.err, q.spin_limit)) {
                stage_wait();   // no copy left in flight on the way out
                return;
            }
            for (int c0 = 0; c0 < nrhs; c0 += kQRhs) {
                const int nc = min(kQRhs, nrhs - c0);
                stage_rows(vec, X, row, nr, nc, n, c0);
                stage_wait();
                __syncthreads();
                for (int k = rt; k < w; k += 64) {
                    T acc[4] = {(T)0, (T)0, (T)0, (T)0};
                    chunk_dot4(matA, vec, k, g, acc);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int c = 4 * g + u;
                        if (c < nc) atomicAdd(Tacc + f + k + (int64_t)(c0 + c) * n, acc[u]);
                    }
                }
                __syncthreads();
            }
            cta_release(nullptr, q.cnt + pid, nullptr, 1);
        }
    }
}

namespace {

template <typename K>
unsigned queue_grid(K kernel, size_t smem, int64_t items)
{
    int dev = 0, sms = 0, occ = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    set_max_carveout(kernel);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, kQThreads, smem);
    const int64_t g = (int64_t)std::max(occ, 1) * std::max(sms, 1);
    return (unsigned)std::max<int64_t>(1, std::min(g, items));
}

size_t rhs16_smem(const SweepQueue &q)
{
    return sizeof(float) * ((size_t)q.mat_elems + (size_t)q.matb_elems + (q.matb_elems ? 2 : 1) * (size_t)q.vec_elems);
}

template <typename T, int NC>
size_t queue_smem(const SweepQueue &q)
{
    using P = Prod<T, NC>;
    return sizeof(T) * ((size_t)2 * P::kMat + (size_t)(q.vec_rows + 64) * NC + P::kRed);
}

template <typename T, int NC>
void fwd(const DevPlan &p, const SweepQueue &q, const T *Dinv, int unit, const T *L, T *Y, T *Z,
         int nrhs, cudaStream_t s)
{
    const size_t smem = queue_smem<T, NC>(q);
    const unsigned grid = queue_grid(fwd_queue_kernel<T, NC>, smem, (int64_t)q.nitems * q.groups);
    fwd_queue_kernel<T, NC><<<grid, kQThreads, smem, s>>>(p, q, Dinv, unit, L, Y, Z, nrhs);
}

template <typename T, int NC>
void bwd(const DevPlan &p, const SweepQueue &q, const T *Dinv, int lu, const T *Lop, const T *Z,
         T *Tacc, T *X, int nrhs, cudaStream_t s)
{
    const size_t smem = queue_smem<T, NC>(q);
    const unsigned grid = queue_grid(bwd_queue_kernel<T, NC>, smem, (int64_t)q.nitems * q.groups);
    bwd_queue_kernel<T, NC><<<grid, kQThreads, smem, s>>>(p, q, Dinv, lu, Lop, Z, Tacc, X, nrhs);
}

}  // namespace

int sweep_groups(bool fp64, int nrhs)
{
    if (!fp64) return 1;
    return std::max(1, std::min(kSweepGroups, nrhs <= kSweepGroups ? nrhs : (nrhs + 7) / 8));
}

template <typename T>
void launch_fwd_queue(const DevPlan &p, const SweepQueue &q, const RowChunk *chunks, const T *Dinv,
                      int unit, const T *L, T *Y, T *Z, int nrhs, cudaStream_t s)
{
    if (q.nitems <= 0) return;
    if constexpr (sizeof(T) == 8) {
        if (nrhs <= kSweepGroups) fwd<T, 1>(p, q, Dinv, unit, L, Y, Z, nrhs, s);
        else fwd<T, 8>(p, q, Dinv, unit, L, Y, Z, nrhs, s);
    } else {
        if (nrhs <= 4) return fwd<T, 4>(p, q, Dinv, unit, L, Y, Z, nrhs, s);
        const size_t smem = rhs16_smem(q);
        const unsigned grid = queue_grid(fwd_rhs16_kernel, smem, q.nitems);
        fwd_rhs16_kernel<<<grid, kQThreads, smem, s>>>(p, q, chunks, Dinv, unit, L, Y, Z, nrhs);
    }
}

template <typename T>
void launch_bwd_queue(const DevPlan &p, const SweepQueue &q, const RowChunk *chunks, const T *Dinv,
                      int lu, const T *Lop, const T *Z, T *Tacc, T *X, int nrhs, cudaStream_t s)
{
    if (q.nitems <= 0) return;
    if constexpr (sizeof(T) == 8) {
        if (nrhs <= kSweepGroups) bwd<T, 1>(p, q, Dinv, lu, Lop, Z, Tacc, X, nrhs, s);
        else bwd<T, 8>(p, q, Dinv, lu, Lop, Z, Tacc, X, nrhs, s);
    } else {
        if (nrhs <= 4) return bwd<T, 4>(p, q, Dinv, lu, Lop, Z, Tacc, X, nrhs, s);
        const size_t smem = rhs16_smem(q);
        const unsigned grid = queue_grid(bwd_rhs16_kernel, smem, q.nitems);
        bwd_rhs16_kernel<<<grid, kQThreads, smem, s>>>(p, q, chunks, Dinv, lu, Lop, Z, Tacc, X, nrhs);
    }
}

template void launch_fwd_queue<double>(const DevPlan &, const SweepQueue &, const RowChunk *, const double *, int,
                                       const double *, double *, double *, int, cudaStream_t);
template void launch_fwd_queue<float>(const DevPlan &, const SweepQueue &, const RowChunk *, const float *, int,
                                      const float *, float *, float *, int, cudaStream_t);
template void launch_bwd_queue<double>(const DevPlan &, const SweepQueue &, const RowChunk *, const double *, int,
                                       const double *, const double *, double *, double *, int, cudaStream_t);
template void launch_bwd_queue<float>(const DevPlan &, const SweepQueue &, const RowChunk *, const float *, int,
                                      const float *, const float *, float *, float *, int, cudaStream_t);

}  // namespace spx
