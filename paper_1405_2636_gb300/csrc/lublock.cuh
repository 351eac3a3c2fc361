// lublock.cuh -- a panel's diagonal block in LU form without row exchanges
// (Sec. III: static pivoting), by one CTA, in shared memory.
#pragma once

#include <cuda_runtime.h>

namespace spx {

// LU of the w x w block a (column-major, leading dimension ld, w <= 32 NR): the
// 8 pivots of a block column by warp 0, its rows in registers (NR a lane), then
// the block row of U one column a thread, then the rank-8 update by all warps.
// (A column at a time spends its time at the barriers and on the update's
// shared-memory round trips.)  pivot(d, k) is the pivot to take for column k,
// given the computed one; it is called by every lane of warp 0 alike.  rcp: the
// reciprocal.
template <typename T, int NR, typename Pivot, typename Rcp>
__device__ __forceinline__ void getrf_cta(T *a, int w, int ld, Pivot pivot, Rcp rcp)
{
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = blockDim.x >> 5;
    for (int k0 = 0; k0 < w; k0 += 8) {
        const int kc = min(8, w - k0), k1 = k0 + kc;
        if (warp == 0) {
            T v[NR][8];
#pragma unroll
            for (int t = 0; t < NR; ++t)
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int i = k0 + lane + 32 * t;
                    v[t][k] = i < w && k < kc ? a[i + (k0 + k) * ld] : (T)0;
                }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if (k >= kc) break;
                const T d = pivot(__shfl_sync(0xffffffffu, v[0][k], k), k0 + k);
                const T r = rcp(d);
                if (lane == k) v[0][k] = d;
                else if (lane > k) v[0][k] *= r;
#pragma unroll
                for (int t = 1; t < NR; ++t) v[t][k] *= r;
#pragma unroll
                for (int j = k + 1; j < 8; ++j) {
                    const T u = __shfl_sync(0xffffffffu, v[0][j], k);
                    if (lane > k) v[0][j] -= v[0][k] * u;
#pragma unroll
                    for (int t = 1; t < NR; ++t) v[t][j] -= v[t][k] * u;
                }
            }
#pragma unroll
            for (int t = 0; t < NR; ++t)
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int i = k0 + lane + 32 * t;
                    if (i < w && k < kc) a[i + (k0 + k) * ld] = v[t][k];
                }
        }
        __syncthreads();
        if (k1 >= w) break;                    // kc == 8 from here on
        for (int j0 = k1 + tid; j0 < w; j0 += blockDim.x) {
            T u[8];
            T *col = a + k0 + j0 * ld;
#pragma unroll
            for (int k = 0; k < 8; ++k) u[k] = col[k];
#pragma unroll
            for (int k = 0; k < 8; ++k)
#pragma unroll
                for (int j = k + 1; j < 8; ++j) u[j] -= a[k0 + j + (k0 + k) * ld] * u[k];
#pragma unroll
            for (int k = 1; k < 8; ++k) col[k] = u[k];
        }
        __syncthreads();
        for (int j = k1 + warp; j < w; j += nw)
            for (int i = k1 + lane; i < w; i += 32) {
                T s = a[i + j * ld];
#pragma unroll
                for (int k = 0; k < 8; ++k) s -= a[i + (k0 + k) * ld] * a[k0 + k + j * ld];
                a[i + j * ld] = s;
            }
        __syncthreads();
    }
}

// In-place inverses of the two factors in a (as getrf_cta leaves them): strictly
// below the diagonal that of the unit lower factor, on and above it that of the
// upper one, which is the transpose of a lower triangle; half of the CTA takes
// each.  The 8 x 8 diagonal blocks first, a column a thread; then block row by
// block row X(b, j) = -D_b^{-1} sum_k L(b, k) X(k, j), the sums in tmp (2 x 8 x w),
// two barriers a block row.
template <typename T, typename Rcp>
__device__ __forceinline__ void invert_lu(T *a, int w, int ld, T *tmp, Rcp rcp)
{
    const int half = blockDim.x / 2, up = threadIdx.x >= half, t0 = threadIdx.x - up * half;
    const int ri = up ? ld : 1, rk = up ? 1 : ld;      // element (i, k) of the lower triangle
    T *t = tmp + up * 8 * w;
    for (int j0 = 0; j0 < w; j0 += half) {             // column j of its diagonal block's inverse
        const int j = j0 + t0, kb = j & ~7, n = min(8, w - kb), c = j - kb;
        T x[8];
        if (j < w) {
            const T *d = a + kb * (ld + 1);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                x[i] = (T)0;
                if (i < n && i >= c) {
                    T s = i == c ? (T)1 : (T)0;
#pragma unroll
                    for (int k = 0; k < i; ++k)
                        if (k >= c) s -= d[i * ri + k * rk] * x[k];
                    x[i] = up ? s * rcp(d[i * (ld + 1)]) : s;
                }
            }
        }
        __syncthreads();                               // whole blocks per turn: half is a multiple of 8
        if (j < w) {
            T *d = a + kb * (ld + 1);
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (i < n && i >= c + 1 - up) d[i * ri + c * rk] = x[i];
        }
        __syncthreads();
    }
    for (int kb = 8; kb < w; kb += 8) {
        const int n = min(8, w - kb);
        for (int e = t0; e < 8 * kb; e += half) {
            const int i = e & 7, j = e >> 3;
            if (i >= n) continue;
            const T *l = a + (kb + i) * ri, *x = a + j * rk;
            T s0 = l[j * rk] * (up ? x[j * ri] : (T)1), s1 = (T)0;
            int k = j + 1;
            for (; k + 1 < kb; k += 2) {
                s0 += l[k * rk] * x[k * ri];
                s1 += l[(k + 1) * rk] * x[(k + 1) * ri];
            }
            if (k < kb) s0 += l[k * rk] * x[k * ri];
            t[e] = s0 + s1;
        }
        __syncthreads();
        for (int e = t0; e < 8 * kb; e += half) {
            const int i = e & 7, j = e >> 3;
            if (i >= n) continue;
            const T *d = a + kb * (ld + 1) + i * ri;
            T s = up ? d[i * rk] * t[e] : t[e];
            for (int k = 0; k < i; ++k) s += d[k * rk] * t[8 * j + k];
            a[(kb + i) * ri + j * rk] = -s;
        }
        __syncthreads();
    }
}

}  // namespace spx
