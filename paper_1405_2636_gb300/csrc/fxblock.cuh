// fxblock.cuh -- a panel's diagonal block in Cholesky form (Sec. III step 1)
// in fixed-point integers.
//
// The block's chain of pivots runs on one SM, whose FP64 unit starts one warp
// instruction per ~19 cycles and returns it after ~64; its integer units
// return a 32 x 32 -> 64-bit multiply-add after ~5 cycles and start 40 times
// as many lane operations.  A positive definite block makes fixed point safe:
// with row and column i scaled by 2^-s_i so that 1 <= a_ii < 4, every entry
// and every partial sum of the factorization stays below sqrt(a_ii a_jj) < 4
// in magnitude, every entry of L below 2 (Cauchy-Schwarz on A = L L^T).
// Entries are held as 64-bit numbers a 2^59 and l 2^60, so a rounding error is
// 2^-60 of sqrt(a_ii a_jj), where FP64's is 2^-53 of the entry's own
// magnitude, at most that of sqrt(a_ii a_jj): the backward error of the block
// does not grow.  Products use two signed limbs (31 bits and the rest), three
// 32 x 32-bit multiply-adds each; the product of the low limbs is below half
// a unit and is left out.
//
// What fixed point cannot hold is left to the floating-point path: the
// function changes nothing and returns false when an entry is not finite,
// when |a_ij| or an entry of L breaks its bound (not positive definite), or
// when a pivot falls below 2^-44 of its bound (it is zero, negative, or so
// small that static replacement may apply).
#pragma once

#include "blocks.cuh"

namespace spx {
namespace fx {

constexpr int kFA = 59;                    // entries of A: a 2^59
constexpr long long kMinPivot = 1LL << (kFA - 44);
constexpr int kThreads = 256;
constexpr int kMaxW = 152;                 // widest block whose square fits the shared memory

__host__ __device__ constexpr int width8(int w) { return (w + 7) & ~7; }

// Shared memory for a block of width up to wmax: the square with L in its
// lower triangle and the inverse, transposed, above it; the digit limbs of two
// block columns; one block row of products; per-column scales and pivots.
__host__ __device__ constexpr size_t smem_bytes(int wmax)
{
    return (size_t)8 * (width8(wmax) + 1) * (width8(wmax) + 1) + (size_t)2 * 8 * 8 * width8(wmax) +
           (size_t)8 * 8 * width8(wmax) + (size_t)width8(wmax) * (8 + 4 + 4 + 4) + 16;
}

struct Limbs {
    int hi, lo;                            // value = hi 2^31 + lo, |lo| <= 2^30
};
__device__ __forceinline__ Limbs limbs(long long v)
{
    Limbs r;
    r.hi = (int)((v + (1LL << 30)) >> 31);
    r.lo = (int)(v - ((long long)r.hi << 31));
    return r;
}

__device__ __forceinline__ long long wide(int a, int b) { return (long long)a * b; }

// (l 2^60)(m 2^60) as a 2^59 entry's decrement
__device__ __forceinline__ long long mul_ll(Limbs a, Limbs b)
{
    return (wide(a.hi, b.hi) << 1) + ((wide(a.hi, b.lo) + wide(a.lo, b.hi) + (1LL << 29)) >> 30);
}

__device__ __forceinline__ long long shfl_ll(long long v, int src)
{
    const int lo = __shfl_sync(0xffffffffu, (int)v, src), hi = __shfl_sync(0xffffffffu, (int)(v >> 32), src);
    return ((long long)hi << 32) | (unsigned)lo;
}

// 1 / sqrt(d) for d = D 2^-59 > 0: y 2^-62 2^e, y in [2^61, 2^62].  The seed
// is rsqrt.approx of d's leading 24 bits (error below 2^-20 with the cut),
// then one step y0 (1 + h / 2 + 3 h^2 / 8), h = 1 - m y0^2, whose error is
// 5 h^3 / 16 < 2^-61; h comes from the exact product m y0^2 modulo 2^77.
__device__ __forceinline__ long long rsqrt_fx(long long D, int *e)
{
    const int n = __clzll(D), s = (n - 1) & ~1;
    const unsigned long long M = (unsigned long long)D << s;   // m = M 2^-61 in [1, 4)
    const unsigned t = (unsigned)(((unsigned long long)D << n) >> 32);
    const unsigned fb = ((unsigned)(128 + s + 1 - n) << 23) | ((t >> 8) & 0x7FFFFFu);
    float yf;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(yf) : "f"(__uint_as_float(fb)));
    const unsigned yb = min(max(__float_as_uint(yf), 0x3F000000u), 0x3F7FFFFFu);   // [1/2, 1)
    const unsigned y0 = (yb & 0x7FFFFFu) | 0x800000u;                              // y0 2^-24
    const unsigned long long q = (unsigned long long)y0 * y0;
    const unsigned ql = (unsigned)q, qh = (unsigned)(q >> 32), Mh = (unsigned)(M >> 32), Ml = (unsigned)M;
    unsigned long long P = (unsigned long long)Mh * ql + __umulhi(Ml, ql);
    P += (unsigned long long)Ml * qh;
    P += (unsigned long long)(Mh * qh) << 32;
    const long long H = -(long long)P;                          // h 2^77
    const int h = (int)(H >> 32);
    const long long C = (H >> 15) + ((wide(h, h) * 3) >> 30);   // (h / 2 + 3 h^2 / 8) 2^63
    *e = s / 2 - 1;
    return ((long long)y0 << 38) + (wide((int)(C >> 32), (int)y0) << 7) +
           (long long)(((unsigned long long)(unsigned)C * y0) >> 25);
}

// v 2^e as a double, rounded to nearest (ties away), the result in range.
__device__ __forceinline__ double to_double(long long v, int e)
{
    if (v == 0) return 0.0;
    const unsigned long long m = (unsigned long long)(v < 0 ? -v : v);
    const int n = __clzll((long long)m);
    const unsigned long long f = m << n;
    const unsigned long long bits =
        ((unsigned long long)(1023 + 63 - n + e - 1) << 52) + (f >> 11) + ((f >> 10) & 1u);
    return __longlong_as_double((long long)(bits | (v < 0 ? 0x8000000000000000ULL : 0ULL)));
}

// d 2^k (the exponent moved with integers; past the normal range by scalbn).
__device__ __forceinline__ double scale2(double d, int k)
{
    const long long b = __double_as_longlong(d);
    const int ef = (int)((b >> 52) & 0x7FF);
    if (ef == 0) return d == 0.0 ? d : scalbn(d, k);
    if ((unsigned)(ef + k - 1) >= 2046u) return scalbn(d, k);
    return __longlong_as_double(b + ((long long)k << 52));
}

// The block columns' pivots by nw warps: every one of them factors the 8 x 8
// diagonal part in its lanes 0 .. 7 (the same operations, so the same bits)
// and applies it to its own rows in lanes 8 .. 31, NR rows a lane, so no warp
// waits for another.  Per column the chain is: the pivot from its lane, its
// reciprocal square root, the column's entry of the next row times it, the
// square subtracted from the next pivot.
template <int NR>
__device__ __forceinline__ void panel(long long *a, int LD, int W8, int kb, int v, int nw, int2 *lim, long long *rfix,
                                      int *rexp, float *rowsum, int *bad)
{
    const int lane = threadIdx.x & 31;
    int row[NR];
    long long q[NR][kDB];
    float sum[NR];
#pragma unroll
    for (int t = 0; t < NR; ++t) {
        row[t] = lane < 8 ? (t == 0 ? kb + lane : W8) : kb + 8 + 24 * (v + t * nw) + lane - 8;
        const bool in = row[t] < W8;
#pragma unroll
        for (int c = 0; c < kDB; ++c) q[t][c] = in && row[t] >= kb + c ? a[row[t] + (kb + c) * LD] : 0;
        sum[t] = in ? rowsum[row[t]] : 0.0f;
    }
    bool wrong = false;
    long long d = shfl_ll(q[0][0], 0);
#pragma unroll
    for (int c = 0; c < kDB; ++c) {
        const int k = kb + c;
        if ((unsigned long long)(d - kMinPivot) >= (1ULL << (kFA + 2)) - kMinPivot) {
            wrong = true;
            d = 1LL << kFA;
        }
        int e;
        const long long y = rsqrt_fx(d, &e);
        const Limbs r = limbs(y >> 1);                     // 2^61
        if (v == 0 && lane == c) {
            rfix[k] = y;
            rexp[k] = e;
        }
        Limbs l[NR];
#pragma unroll
        for (int t = 0; t < NR; ++t) {
            const long long x = q[t][c];
            // |a_ik| 2^e <= sqrt(a_ii d) 2^e < 4
            if (row[t] > k && row[t] < W8 && ((x < 0 ? -x : x) >> (kFA + 2 - e)) != 0) wrong = true;
            const Limbs s = limbs((long long)((unsigned long long)x << e));
            const long long lv =
                (wide(s.hi, r.hi) << 2) + ((wide(s.hi, r.lo) + wide(s.lo, r.hi) + (1LL << 28)) >> 29);
            l[t] = limbs(lv);
            q[t][c] = lv;
        }
        if (c + 1 < kDB) {
            // the next pivot from its own lane's entry, ahead of the others' updates
            const int c1 = c + 1 < kDB ? c + 1 : c;
            d = shfl_ll(q[0][c1] - mul_ll(l[0], l[0]), c1);
        }
#pragma unroll
        for (int t = 0; t < NR; ++t) {
            const float lf = (float)l[t].hi * 0x1p-29f;
            sum[t] = fmaf(lf, lf, sum[t]);
            // sum_k l_ik^2 <= a_ii (the sum starts from -a_ii), with room for FP32's rounding
            if (row[t] > k && row[t] < W8 && !(sum[t] <= 5e-4f)) wrong = true;
        }
#pragma unroll
        for (int c2 = c + 1; c2 < kDB; ++c2) {
            Limbs o;
            o.hi = __shfl_sync(0xffffffffu, l[0].hi, c2);
            o.lo = __shfl_sync(0xffffffffu, l[0].lo, c2);
#pragma unroll
            for (int t = 0; t < NR; ++t) q[t][c2] -= mul_ll(l[t], o);
        }
    }
#pragma unroll
    for (int t = 0; t < NR; ++t) {
        if (row[t] >= W8 || (lane < 8 && v != 0)) continue;
        rowsum[row[t]] = sum[t];
#pragma unroll
        for (int c = 0; c < kDB; ++c) {
            const bool lower = row[t] >= kb + c;
            const Limbs l = limbs(q[t][c]);
            if (lower) a[row[t] + (kb + c) * LD] = q[t][c];
            lim[c * W8 + row[t]] = lower ? make_int2(l.hi, l.lo) : make_int2(0, 0);
        }
    }
    if (wrong) *bad = 1;
}

// Columns [j0, j1), rows >= j: a -= the rank-8 product of the block column in
// lim; the pairs in turns over threads t0, t0 + ts, ...
__device__ __forceinline__ void rank8(long long *a, int LD, int W8, const int2 *lim, int j0, int j1, int t0, int ts)
{
    int j = j0, rem = t0;
    while (j < j1 && rem >= W8 - j) {
        rem -= W8 - j;
        ++j;
    }
    while (j < j1) {
        const int i = j + rem;
        long long hh = 0, mid = 0;
#pragma unroll
        for (int c = 0; c < kDB; ++c) {
            const int2 x = lim[c * W8 + i], y = lim[c * W8 + j];
            hh += wide(x.x, y.x);
            mid += wide(x.x, y.y);
            mid += wide(x.y, y.x);
        }
        a[i + j * LD] -= (hh << 1) + ((mid + (1LL << 29)) >> 30);
        rem += ts;
        while (j < j1 && rem >= W8 - j) {
            rem -= W8 - j;
            ++j;
        }
    }
}

// Block column b of L as doubles, in place.
__device__ __forceinline__ void convert(long long *a, int LD, int W8, int b, int t0, int ts)
{
    for (int e = t0; e < kDB * (W8 - kDB * b); e += ts) {
        const int c = e & 7, i = kDB * b + (e >> 3), j = kDB * b + c;
        if (i >= j) a[i + j * LD] = __double_as_longlong(to_double(a[i + j * LD], -60));
    }
}

// Block row b of X = L^{-1}, first half: T_j = sum_k L_bk X_kj for the blocks
// j < b, on the FP64 tensor path (which no other part of this kernel uses), and
// the inverse of the 8 x 8 diagonal block, by the last of nw warps.
__device__ __forceinline__ void inverse_products(double *a, int LD, int b, int wi, int nw, double *Tm,
                                                 const long long *rfix, const int *rexp)
{
    const int lane = threadIdx.x & 31, r = lane >> 2, q = lane & 3, kb = kDB * b;
    if (wi == nw - 1) {
        if (lane < kDB) {
            double x[kDB];
#pragma unroll
            for (int i = 0; i < kDB; ++i) x[i] = 0.0;
#pragma unroll
            for (int i = 0; i < kDB; ++i) {
                const double ri = to_double(rfix[kb + i], rexp[kb + i] - 62);
                double s0 = 0.0, s1 = 0.0;
#pragma unroll
                for (int k = 0; k < i; ++k) {
                    const double l = a[(kb + i) + (kb + k) * LD];
                    if (k & 1) s1 = fma(l, x[k], s1);
                    else s0 = fma(l, x[k], s0);
                }
                x[i] = i == lane ? ri : (i > lane ? -ri * (s0 + s1) : 0.0);
            }
            __syncwarp(0xffu);
#pragma unroll
            for (int i = 0; i < kDB; ++i)
                if (i >= lane) a[(kb + lane) + (kb + i + 1) * LD] = x[i];
        }
        __syncwarp();
        if (nw > 1) return;
    }
    for (int j = wi; j < b; j += max(nw - 1, 1)) {
        double c0 = 0.0, c1 = 0.0, e0 = 0.0, e1 = 0.0;
        for (int k = j; k < b; ++k) {
            const double a0 = a[(kb + r) + (kDB * k + q) * LD], a1 = a[(kb + r) + (kDB * k + 4 + q) * LD];
            double b0 = a[(kDB * j + r) + (kDB * k + q + 1) * LD], b1 = a[(kDB * j + r) + (kDB * k + q + 5) * LD];
            if (k == j) {   // X_jj is lower triangular
                if (q < r) b0 = 0.0;
                if (q + 4 < r) b1 = 0.0;
            }
            dmma_f64(c0, c1, a0, b0);
            dmma_f64(e0, e1, a1, b1);
        }
        Tm[(kDB * j + 2 * q) * kDB + r] = c0 + e0;
        Tm[(kDB * j + 2 * q + 1) * kDB + r] = c1 + e1;
    }
}

// ... second half: X_bj = -X_bb T_j.
__device__ __forceinline__ void inverse_finish(double *a, int LD, int b, int wi, int nw, const double *Tm)
{
    const int lane = threadIdx.x & 31, r = lane >> 2, q = lane & 3, kb = kDB * b;
    double a0 = -a[(kb + q) + (kb + r + 1) * LD], a1 = -a[(kb + q + 4) + (kb + r + 1) * LD];
    if (q > r) a0 = 0.0;
    if (q + 4 > r) a1 = 0.0;
    for (int j = wi; j < b; j += nw) {
        double c0 = 0.0, c1 = 0.0;
        dmma_f64(c0, c1, a0, Tm[(kDB * j + r) * kDB + q]);
        dmma_f64(c0, c1, a1, Tm[(kDB * j + r) * kDB + q + 4]);
        a[(kDB * j + 2 * q) + (kb + r + 1) * LD] = c0;
        a[(kDB * j + 2 * q + 1) + (kb + r + 1) * LD] = c1;
    }
}

__device__ __forceinline__ void bar_some(int threads)
{
    asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory");
}

// The whole block: L over its lower triangle, L^{-1} at Mi (w x w, zeros
// above).  All 256 threads; false (and nothing written) when the block has to
// go the floating-point way.  While the chain of block column b runs on up to
// three warps (NR = 2 rows a lane: four), the others finish the rank-8 update of block column b - 1 and
// extend the inverse by its block row.
template <typename T, int NR>
__device__ bool diag_block(T *__restrict__ D, T *__restrict__ Mi, int w, int h, unsigned char *smraw)
{
    const int W8 = width8(w), LD = W8 + 1, nb = W8 / kDB;
    long long *a = reinterpret_cast<long long *>(smraw);
    double *ad = reinterpret_cast<double *>(smraw);
    int2 *lim = reinterpret_cast<int2 *>(a + (size_t)LD * LD);     // [2][8][W8]
    double *Tm = reinterpret_cast<double *>(lim + 2 * kDB * W8);   // [W8][8]
    long long *rfix = reinterpret_cast<long long *>(Tm + kDB * W8);
    int *rexp = reinterpret_cast<int *>(rfix + W8);
    int *sc = rexp + W8;
    float *rowsum = reinterpret_cast<float *>(sc + W8);
    int *bad = reinterpret_cast<int *>(rowsum + W8);
    const int tid = threadIdx.x, warp = tid >> 5;

    if (tid == 0) *bad = 0;
    __syncthreads();
    if (tid < W8) {
        int s = 0;
        float diag = 1.0f;
        if (tid < w) {
            const double d = to_f64<T>(__ldcg(D + tid + (int64_t)tid * h));
            const long long b = __double_as_longlong(d);
            const int ef = (int)(b >> 52);   // 0 .. 0x7FE for a positive finite d
            if (ef < 128 || ef > 1918) *bad = 1;
            s = (ef - 1023) >> 1;
            diag = __uint_as_float(((unsigned)(127 + ((ef - 1023) & 1)) << 23) | (unsigned)((b >> 29) & 0x7FFFFF));
        }
        sc[tid] = s;
        rowsum[tid] = -diag;
    }
    __syncthreads();
    {
        constexpr int NB = 8;   // loads in flight a thread
        const int total = W8 * W8;
        for (int base = tid; base < total; base += kThreads * NB) {
            T v[NB];
#pragma unroll
            for (int u = 0; u < NB; ++u) {
                const int e = base + u * kThreads, i = e % W8, j = e / W8;
                v[u] = (e < total && i < w && j < w && i >= j) ? __ldcg(D + i + (int64_t)j * h) : (T)0;
            }
#pragma unroll
            for (int u = 0; u < NB; ++u) {
                const int e = base + u * kThreads, i = e % W8, j = e / W8;
                if (e >= total || i < j) continue;
                long long f = 0;
                if (i >= w || j >= w) {
                    f = i == j ? 1LL << kFA : 0;
                } else {
                    const long long b = __double_as_longlong(to_f64<T>(v[u]));
                    const int ef = (int)((b >> 52) & 0x7FF);
                    long long m = b & 0xFFFFFFFFFFFFFLL;
                    if (ef > 0) m |= 0x10000000000000LL;
                    const int sh = (ef > 0 ? ef : 1) - 1075 - sc[i] - sc[j] + kFA;   // 2^sh m
                    if (m != 0 && sh > 8) *bad = 1;          // 4 or more, infinite or NaN
                    else if (sh >= 0) m <<= sh;
                    else m = sh < -60 ? 0 : (m + (1LL << (-sh - 1))) >> -sh;
                    f = b < 0 ? -m : m;
                }
                a[i + j * LD] = f;
            }
        }
    }
    __syncthreads();
    if (*bad) return false;

    auto others = [&](int b, int wi, int nw) {
        // block column b is done: its updates past the next block column, its
        // conversion, its row of the inverse
        rank8(a, LD, W8, lim + (b & 1) * kDB * W8, kDB * (b + 2), W8, 32 * wi + (tid & 31), 32 * nw);
        convert(a, LD, W8, b, 32 * wi + (tid & 31), 32 * nw);
        bar_some(32 * nw);
        inverse_products(ad, LD, b, wi, nw, Tm, rfix, rexp);
        bar_some(32 * nw);
        inverse_finish(ad, LD, b, wi, nw, Tm);
    };
    for (int b = 0; b < nb; ++b) {
        const int kb = kDB * b;
        const int nw = min(NR == 1 ? 3 : 4, max(1, (W8 - kb - kDB + 24 * NR - 1) / (24 * NR)));
        if (warp < nw) panel<NR>(a, LD, W8, kb, warp, nw, lim + (b & 1) * kDB * W8, rfix, rexp, rowsum,
                                  bad);
        else if (b > 0) others(b - 1, warp - nw, kThreads / 32 - nw);
        __syncthreads();
        if (*bad) return false;
        if (b + 1 < nb) {
            rank8(a, LD, W8, lim + (b & 1) * kDB * W8, kb + kDB, kb + 2 * kDB, tid, kThreads);
            __syncthreads();
        }
    }
    others(nb - 1, warp, kThreads / 32);
    __syncthreads();
    for (int e = tid; e < w * w; e += kThreads) {
        const int i = e % w, j = e / w;
        if (i >= j) {
            D[i + (int64_t)j * h] = from_f64<T>(scale2(ad[i + j * LD], sc[i]));
            Mi[e] = from_f64<T>(scale2(ad[j + (i + 1) * LD], -sc[j]));
        } else {
            Mi[e] = (T)0;
        }
    }
    return true;
}

}  // namespace fx
}  // namespace spx
