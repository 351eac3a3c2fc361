// fxblock.cuh -- a panel's diagonal block in Cholesky form (Sec. III step 1)
// in fixed-point integers.
//
// The block's chain of pivots runs on one SM, whose FP64 unit starts one warp
// instruction per ~19 cycles and returns it after ~64; a 32 x 32 -> 64-bit
// multiply-add returns after ~16, and four warps start one at a time.  A positive definite block makes fixed point safe:
// with row and column i scaled by 2^-s_i so that 1 <= a_ii < 4, every entry
// and every partial sum of the factorization stays below sqrt(a_ii a_jj) < 4
// in magnitude, every entry of L below 2 (Cauchy-Schwarz on A = L L^T).
// Entries are held as 64-bit numbers a 2^59 and l 2^60, so a rounding error is
// 2^-60 of sqrt(a_ii a_jj), where FP64's is 2^-53 of the entry's own
// magnitude, at most that of sqrt(a_ii a_jj): the backward error of the block
// does not grow.  The inverse X of the scaled L is held as x 2^56 while every
// |x| < 8; its rows' largest entries are at least 1/2 (at 2^53 the solves' errors
// were 1.5 times those of FP64's, at 2^56 they are 0.85 of them).  Products use two
// signed limbs (31 bits and the rest), three 32 x 32-bit multiply-adds each;
// the product of the low limbs is below half a unit and of either sign, so it
// is left out -- but for the squares on the diagonal, whose low limbs' squares
// would all add up one way (a relative 2^-57 of every pivot, which the solve of
// a 64^3 grid amplifies a thousandfold): those are summed beside it (low).
//
// What fixed point cannot hold is left to the floating-point path: the
// function changes nothing and returns kRefused when an entry is not finite,
// when |a_ij| or an entry of L breaks its bound (not positive definite), or when
// a pivot falls below 2^-44 of its bound (it is zero, negative, or so small
// that static replacement may apply).  When an entry of X reaches 8, which
// ordinary blocks do (12 on a plate's separator, 48 with coefficients spread over
// e^4), L is as good as ever: it is stored, the caller forms the inverse alone in
// floating point, and kNoInverse says so.
//
// A 64-wide FP64 block takes 49 us (FP64 unit: 69), FP32 47 (53; both start as
// the same integers); 128 wide 0.18 ms (0.58 on the FP64 unit).  With the inverse
// in floating point 69 us and 50, 0.40 ms and 0.25 (the whole block a second time
// on the FP64 unit: 111 and 92, 0.74 and 0.60).  What bounds it: per 8 columns about 6,600 cycles of one warp's
// dependent instructions, a third of them the reciprocal square roots.
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
// lower triangle and the inverse, transposed, above it; the limbs of two block
// columns of L and of a block row of X; per-column scales, pivots and sums.
__host__ __device__ constexpr size_t smem_bytes(int wmax)
{
    return (size_t)8 * (width8(wmax) + 1) * (width8(wmax) + 1) + (size_t)3 * 8 * kDB * width8(wmax) +
           (size_t)width8(wmax) * (8 + 4 + 4 + 4 + 4) + 16;
}
constexpr int kFX = 56;                    // entries of X: x 2^56, |x| < 8
constexpr long long kMaxX = 1LL << (kFX + 3);
constexpr int kMaxXe = 61 - kFX;           // a pivot's reciprocal root above 2^kMaxXe is above that, too

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
    const unsigned f = __float_as_uint(__ll2float_rz(D));
    const int s = (189 - (int)(f >> 23)) & ~1;                  // D in [2^62-s', ...), s even
    const unsigned long long M = (unsigned long long)D << s;   // m = M 2^-61 in [1, 4)
    const unsigned fb = f + ((unsigned)(s - 61) << 23);
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
           (long long)(((unsigned long long)(unsigned)C * y0 + (1u << 24)) >> 25);
}

// A number's fields by integer operations: sign, biased exponent, mantissa
// with the leading bit (subnormal numbers: without, at exponent 1) shifted to
// 62 bits.  value = m 2^(e - kBias); a double's m is one less where a bit from
// the middle of its mantissa is set, so that of the ties in rounding it later
// half go up and half down (all up: 64 entries of a row would add up).
template <typename T>
struct Fields;
template <>
struct Fields<double> {
    static constexpr int kOne = 1023, kBias = 1075 + 9, kMin = 128, kMax = 1918;
    long long b;
    __device__ __forceinline__ explicit Fields(double v) { b = __double_as_longlong(v); }
    __device__ __forceinline__ int top() const { return (int)(b >> 52); }          // sign and exponent
    __device__ __forceinline__ unsigned mant23() const { return (unsigned)(b >> 29) & 0x7FFFFFu; }
    __device__ __forceinline__ int exp() const { return max((int)(b >> 52) & 0x7FF, 1); }
    __device__ __forceinline__ long long sign() const { return b >> 63; }
    __device__ __forceinline__ unsigned long long mant() const
    {
        const unsigned long long m = (unsigned long long)b & 0xFFFFFFFFFFFFFULL;
        return ((((b >> 52) & 0x7FF) != 0 ? m | 0x10000000000000ULL : m) << 9) - ((b >> 40) & 1);
    }
};
template <>
struct Fields<float> {
    static constexpr int kOne = 127, kBias = 150 + 38, kMin = 1, kMax = 254;
    int b;
    __device__ __forceinline__ explicit Fields(float v) { b = __float_as_int(v); }
    __device__ __forceinline__ int top() const { return b >> 23; }
    __device__ __forceinline__ unsigned mant23() const { return (unsigned)b & 0x7FFFFFu; }
    __device__ __forceinline__ int exp() const { return max((b >> 23) & 0xFF, 1); }
    __device__ __forceinline__ long long sign() const { return b >> 31; }
    __device__ __forceinline__ unsigned long long mant() const
    {
        return (unsigned long long)(((b >> 23) & 0xFF) != 0 ? mant23() | 0x800000u : mant23()) << 38;
    }
};

// v 2^e rounded to nearest, the result in range: as a double by integer
// operations (ties away), as a float by the conversion.
__device__ __forceinline__ void to_value(long long v, int e, double *out)
{
    const unsigned long long m = (unsigned long long)(v < 0 ? -v : v);
    const int n = __clzll((long long)m);
    const unsigned long long f = m << n;
    const unsigned long long bits =
        ((unsigned long long)(1023 + 63 - n + e - 1) << 52) + (f >> 11) + ((f >> 10) & 1u);
    *out = v == 0 ? 0.0 : __longlong_as_double((long long)(bits | (v < 0 ? 0x8000000000000000ULL : 0ULL)));
}
__device__ __forceinline__ void to_value(long long v, int e, float *out)
{
    *out = __ll2float_rn(v) * __uint_as_float((unsigned)(127 + e) << 23);
}

// The block columns' pivots by nw warps: every one of them factors the 8 x 8
// diagonal part in its lanes 0 .. 7 (the same operations, so the same bits)
// and applies it to its own rows in lanes 8 .. 31, NR rows a lane, so no warp
// waits for another.  Column c takes its row's earlier columns at once, when
// its turn comes (sums of limb products, cut to a result once a column); the
// next pivot comes from its own lane's running sum of squares.  The chain of a
// column is then: the pivot from its lane, its reciprocal square root, the
// column's entry times it, its square taken from the next pivot.
// True when this thread saw what fixed point cannot hold.
template <int NR>
__device__ __forceinline__ bool panel(long long *a, int LD, int W8, int kb, int v, int nw, int2 *lim, long long *rfix,
                                      int *rexp, const float *low)
{
    const int lane = threadIdx.x & 31;
    int row[NR];
    long long q[NR][kDB];
    Limbs l[NR][kDB];
#pragma unroll
    for (int t = 0; t < NR; ++t) {
        row[t] = lane < 8 ? (t == 0 ? kb + lane : W8) : kb + 8 + 24 * (v + t * nw) + lane - 8;
#pragma unroll
        for (int c = 0; c < kDB; ++c) q[t][c] = row[t] < W8 && row[t] >= kb + c ? a[row[t] + (kb + c) * LD] : 0;
    }
    // this lane's diagonal entry (lanes 0 .. 7) and the sum of squares to take from it
    long long own = 0, dh = 0, dm = 0;
#pragma unroll
    for (int c = 0; c < kDB; ++c)
        if (lane == c) own = q[0][c];
    if (lane < kDB) own -= __float2int_rn(low[kb + lane]);
    int off = 0;
    long long ykeep = 0;
    int ekeep = 0;
    long long d = shfl_ll(own, 0);
#pragma unroll
    for (int c = 0; c < kDB; ++c) {
        const bool low = (unsigned long long)(d - kMinPivot) >= (1ULL << (kFA + 2)) - kMinPivot;
        off |= low;
        d = low ? 1LL << kFA : d;
        int e;
        const long long y = rsqrt_fx(d, &e);
        const Limbs r = limbs(y >> 1);                     // 2^61
        ykeep = lane == c ? y : ykeep;
        ekeep = lane == c ? e : ekeep;
        long long hh[NR], mid[NR];
#pragma unroll
        for (int t = 0; t < NR; ++t) hh[t] = mid[t] = 0;
#pragma unroll
        for (int k = 0; k < c; ++k) {
            const int oh = __shfl_sync(0xffffffffu, l[0][k].hi, c), ol = __shfl_sync(0xffffffffu, l[0][k].lo, c);
#pragma unroll
            for (int t = 0; t < NR; ++t) {
                hh[t] += wide(l[t][k].hi, oh);
                mid[t] += wide(l[t][k].hi, ol);
                mid[t] += wide(l[t][k].lo, oh);
            }
        }
#pragma unroll
        for (int t = 0; t < NR; ++t) {
            long long x = q[t][c] - (hh[t] << 1) - ((mid[t] + (1LL << 29)) >> 30);
            if (t == 0 && lane == c) x = d;
            // |a_ik| 2^e <= sqrt(a_ii d) 2^e < 4 (rows of padding are zero)
            const int xh = (int)(x >> 32), over = (xh ^ (xh >> 31)) >> (kFA + 2 - 32 - e);
            off |= t > 0 || lane > c ? over : 0;
            const Limbs s = limbs((long long)((unsigned long long)x << e));
            l[t][c] = limbs((wide(s.hi, r.hi) << 2) + ((wide(s.hi, r.lo) + wide(s.lo, r.hi) + (1LL << 28)) >> 29));
        }
        dh += wide(l[0][c].hi, l[0][c].hi);
        dm += wide(l[0][c].hi, l[0][c].lo) + __mulhi(l[0][c].lo, l[0][c].lo);
        if (c + 1 < kDB) d = shfl_ll(own - (dh << 1) - ((dm + (1LL << 28)) >> 29), c + 1);
    }
    if (v == 0 && lane < kDB) {
        rfix[kb + lane] = ykeep;
        rexp[kb + lane] = ekeep;
    }
#pragma unroll
    for (int t = 0; t < NR; ++t) {
        if (row[t] >= W8 || (lane < 8 && v != 0)) continue;
#pragma unroll
        for (int c = 0; c < kDB; ++c) {
            const bool lower = row[t] >= kb + c;
            if (lower) a[row[t] + (kb + c) * LD] = ((long long)l[t][c].hi << 31) + l[t][c].lo;
            lim[c * W8 + row[t]] = lower ? make_int2(l[t][c].hi, l[t][c].lo) : make_int2(0, 0);
        }
    }
    return off != 0;
}

// sum over the block's eight terms of x y by limbs: hh 2^62 + mid 2^31
__device__ __forceinline__ void dot8(const int2 *x, int xs, const int2 *y, int ys, long long &hh, long long &mid)
{
    hh = mid = 0;
#pragma unroll
    for (int c = 0; c < kDB; ++c) {
        const int2 u = x[c * xs], v = y[c * ys];
        hh += wide(u.x, v.x);
        mid += wide(u.x, v.y);
        mid += wide(u.y, v.x);
    }
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
        long long hh, mid;
        dot8(lim + i, W8, lim + j, W8, hh, mid);
        a[i + j * LD] -= (hh << 1) + ((mid + (1LL << 29)) >> 30);
        rem += ts;
        while (j < j1 && rem >= W8 - j) {
            rem -= W8 - j;
            ++j;
        }
    }
}

// Block row b of X = L^{-1} by forward substitution, one column j a thread: the
// sums T(i, j) = sum_k L(i, k) X(k, j) over the earlier blocks stand in X's
// places, the block's own terms follow here.  True when an entry breaks its bound.
__device__ __forceinline__ bool inverse_row(long long *a, int LD, int W8, int b, int j, const int2 *lim, int2 *limx,
                                            const long long *rfix, const int *rexp)
{
    const int kb = kDB * b;
    Limbs x[kDB];
    bool wrong = false;
#pragma unroll
    for (int r = 0; r < kDB; ++r) {
        const int i = kb + r, e = rexp[i];
        const long long y = rfix[i];
        long long s = a[j + (i + 1) * LD], hh = 0, mid = 0;
#pragma unroll
        for (int k = 0; k < r; ++k) {
            const int2 l = lim[k * W8 + i];
            hh += wide(l.x, x[k].hi);
            mid += wide(l.x, x[k].lo);
            mid += wide(l.y, x[k].hi);
        }
        s += (hh << 2) + ((mid + (1LL << 28)) >> 29);
        wrong = wrong || e > kMaxXe || (s ^ (s >> 63)) >= (1LL << 61);
        const Limbs u = limbs(s), v = limbs(y >> 1);
        long long xv = (wide(u.hi, v.hi) << 1) + ((wide(u.hi, v.lo) + wide(u.lo, v.hi) + (1LL << 29)) >> 30);
        const int sh = min(max(e, 0), kMaxXe);
        if (j == i) xv = (y + (1LL << (61 - kFX))) >> (62 - kFX);             // 1 / l_ii
        wrong = wrong || (j <= i && (xv ^ (xv >> 63)) >= (kMaxX >> sh));
        xv = (long long)((unsigned long long)(j < i ? -xv : xv) << sh);
        if (j > i) xv = 0;
        x[r] = limbs(xv);
        if (j <= i) a[j + (i + 1) * LD] = xv;
        limx[r * W8 + j] = make_int2(x[r].hi, x[r].lo);
    }
    return wrong;
}

// T(i, j) += sum over block b of L(i, k) X(k, j), rows i past the block,
// columns j up to its end.
__device__ __forceinline__ void inverse_sums(long long *a, int LD, int W8, int b, const int2 *lim, const int2 *limx,
                                             int t0, int ts)
{
    const int i0 = kDB * (b + 1), nj = i0, ni = W8 - i0;
    if (ni <= 0) return;
    int i = t0 % nj, c = t0 / nj;          // column i, row i0 + c: columns side by side in memory
    for (; c < ni;) {
        long long hh, mid;
        dot8(lim + i0 + c, W8, limx + i, W8, hh, mid);
        a[i + (i0 + c + 1) * LD] += (hh << 2) + ((mid + (1LL << 28)) >> 29);
        i += ts;
        while (i >= nj) {
            i -= nj;
            ++c;
        }
    }
}

// sum_k l_ik^2 <= a_ii, with room for FP32's rounding (the sum starts from
// -a_ii), or true; the squares of the low limbs, in units of an entry.
__device__ __forceinline__ bool check_row(int i, int W8, const int2 *lim, float *rowsum, float *low)
{
    float s = rowsum[i], t = low[i];
#pragma unroll
    for (int c = 0; c < kDB; ++c) {
        const int2 l = lim[c * W8 + i];
        const float f = (float)l.x * 0x1p-29f, g = (float)l.y * 0x1p-30f;
        s = fmaf(f, f, s);
        t = fmaf(g * 0.5f, g, t);
    }
    low[i] = t;
    rowsum[i] = s;
    return !(s <= 5e-4f);
}

__device__ __forceinline__ void bar_some(int threads)
{
    asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory");
}

// The whole block: L over its lower triangle, L^{-1} at Mi (w x w, zeros
// above).  All 256 threads.  While the chain of block column b runs on up to
// three warps (NR = 2 rows a lane: four), the others finish the rank-8 update
// of block column b - 1 and extend the inverse by its block row.  What a thread
// finds stays its own until a barrier joins all threads' words, so that all leave
// at the same barrier: a shared flag, read behind one barrier, could already hold
// what a faster warp finds before the next.  (leave_out is such a flag and decides
// nothing: it saves rows of an inverse that is not used, between barriers that
// every thread passes.)
// rowexp (or null): the exponents of about sqrt(a_ii).
enum Outcome { kRefused, kNoInverse, kDone };
enum Found : int { kBad = 1, kWideInv = 2 };
template <typename T, int NR>
__device__ Outcome diag_block(T *__restrict__ D, T *__restrict__ Mi, int w, int h, unsigned char *smraw, int32_t *rowexp)
{
    const int W8 = width8(w), LD = W8 + 1, nb = W8 / kDB;
    long long *a = reinterpret_cast<long long *>(smraw);
    int2 *lim = reinterpret_cast<int2 *>(a + (size_t)LD * LD);     // [2][8][W8]
    int2 *limx = lim + 2 * kDB * W8;                               // [8][W8]
    long long *rfix = reinterpret_cast<long long *>(limx + kDB * W8);
    int *rexp = reinterpret_cast<int *>(rfix + W8);
    int *sc = rexp + W8;
    float *rowsum = reinterpret_cast<float *>(sc + W8);
    float *low = rowsum + W8;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    volatile int *leave_out = reinterpret_cast<int *>(low + W8);   // a thread saw kWideInv: no more of the inverse
    int found = 0;

    if (tid == 0) *leave_out = 0;
    if (tid < W8) {
        int s = 0;
        float diag = 1.0f;
        if (tid < w) {
            const Fields<T> d(__ldcg(D + tid + (int64_t)tid * h));
            const int ef = d.top();          // the exponent alone for a positive d
            found = ef < Fields<T>::kMin || ef > Fields<T>::kMax ? kBad : 0;
            s = (ef - Fields<T>::kOne) >> 1;
            if (sizeof(T) == 8 && rowexp) rowexp[tid] = s;   // (FP64 factors only)
            diag = __uint_as_float(((unsigned)(127 + ((ef - Fields<T>::kOne) & 1)) << 23) | d.mant23());
        }
        sc[tid] = s;
        rowsum[tid] = -diag;
        low[tid] = 0.0f;
    }
    __syncthreads();
    // a warp takes columns, its lanes rows, several columns' loads in flight;
    // X's places (above the diagonal) start as zero sums
    for (int i = lane; i < W8; i += 32) {
        constexpr int NB = 8;
        const int si = sc[i];
        for (int j0 = warp; j0 < W8; j0 += 8 * NB) {
            T v[NB];
#pragma unroll
            for (int u = 0; u < NB; ++u) {
                const int j = j0 + 8 * u;
                v[u] = i < w && j < w && i >= j ? __ldcg(D + i + (int64_t)j * h) : (T)0;
            }
#pragma unroll
            for (int u = 0; u < NB; ++u) {
                const int j = j0 + 8 * u;
                if (j >= W8) continue;
                if (i < j) {
                    a[i + j * LD] = 0;                 // X(j - 1, i)
                    continue;
                }
                long long f = i == j ? 1LL << kFA : 0;
                if (i < w) {
                    const Fields<T> x(v[u]);
                    const unsigned long long m = x.mant();
                    const int n = si + sc[j] + Fields<T>::kBias - kFA - x.exp();   // m 2^-n
                    found |= m != 0 && n < 1 ? kBad : 0;   // 4 or more, infinite or NaN
                    const long long g = (long long)((m >> min(max(n - 1, 0), 63)) + 1) >> 1, sign = x.sign();
                    f = (g ^ sign) - sign;
                }
                a[i + j * LD] = f;
            }
        }
        a[i + W8 * LD] = 0;                            // X(W8 - 1, i)
    }
    if (__syncthreads_or(found)) return kRefused;

    // block column b of L is done: its updates past the next block column, its
    // block row of the inverse, that row's share of the sums below
    auto others = [&](int b, int wi, int nw) {
        const int2 *lb = lim + (b & 1) * kDB * W8;
        const int cols = kDB * (b + 1), nx = min(nw, (cols + 31) / 32);
        if (wi < nx && !*leave_out)
            for (int j = 32 * wi + lane; j < cols; j += 32 * nx)
                if (inverse_row(a, LD, W8, b, j, lb, limx, rfix, rexp)) {
                    found |= kWideInv;
                    *leave_out = 1;
                }
        if (nx == nw) rank8(a, LD, W8, lb, kDB * (b + 2), W8, 32 * wi + lane, 32 * nw);
        else if (wi >= nx) rank8(a, LD, W8, lb, kDB * (b + 2), W8, 32 * (wi - nx) + lane, 32 * (nw - nx));
        bar_some(32 * nw);
        inverse_sums(a, LD, W8, b, lb, limx, 32 * wi + lane, 32 * nw);
    };
    for (int b = 0; b < nb; ++b) {
        const int kb = kDB * b;
        int2 *lb = lim + (b & 1) * kDB * W8;
        const int nw = min(NR == 1 ? 3 : 4, max(1, (W8 - kb - kDB + 24 * NR - 1) / (24 * NR)));
        if (warp < nw) found |= panel<NR>(a, LD, W8, kb, warp, nw, lb, rfix, rexp, low) ? kBad : 0;
        else if (b > 0) others(b - 1, warp - nw, kThreads / 32 - nw);
        __syncthreads();
        if (kb + tid < W8) found |= check_row(kb + tid, W8, lb, rowsum, low) ? kBad : 0;
        if (b + 1 < nb) rank8(a, LD, W8, lb, kb + kDB, kb + 2 * kDB, tid, kThreads);
        if (__syncthreads_or(found & kBad)) return kRefused;
    }
    others(nb - 1, warp, kThreads / 32);
    if (__syncthreads_or(found & kWideInv)) {
        for (int j = warp; j < w; j += 8)
            for (int i = j + lane; i < w; i += 32) to_value(a[i + j * LD], sc[i] - 60, D + i + (int64_t)j * h);
        return kNoInverse;
    }
    for (int j = warp; j < w; j += 8) {
        const int sj = sc[j];
        for (int i = lane; i < w; i += 32) {
            T x = (T)0;
            if (i >= j) {
                T l;
                to_value(a[i + j * LD], sc[i] - 60, &l);
                to_value(a[j + (i + 1) * LD], -kFX - sj, &x);
                D[i + (int64_t)j * h] = l;
            }
            Mi[i + j * w] = x;
        }
    }
    return kDone;
}

}  // namespace fx
}  // namespace spx
