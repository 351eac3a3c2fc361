// update_sl.cu -- FP64 panel TRSM and supernodal updates (Sec. III steps 2
// and 3, Sec. V-B) on the FP16 tensor cores by error-free slices
// (slices.cuh), for Cholesky and LDL^T factors in FP64.
//
// Operand copy, of the off-diagonal rows of the panels whose updates run here,
// in blocks of 128 rows by 64 columns (digit blocks): an array of K-major FP16
// rows of 64 elements (128 bytes), slice s of it from row s * oprows on.  A block
// of a panel at most 32 or 16 columns wide takes half or a quarter of the row
// (columns 16 * chunk on), beside other blocks: SlPlace says where.  Each (row,
// digit block) has its own exponent at exp[block * exprows + prow[p] + r].  The
// TRSM writes the copy; the update loads 128-row (A) and 64-row (B) boxes of it by
// TMA with the 128-byte swizzle, whole rows whatever the width, and its MMAs start
// at the chunk.
#include "blocks.cuh"
#include "slices.cuh"

#include <algorithm>

namespace spx {
namespace {

using namespace tc;
using namespace sl;

constexpr int kBN = 64;                               // accumulator columns of one group
constexpr int kABytes = kM * kRowBytes;               // one slice of A: 128 rows x 64 digits
constexpr int kBBytes = kBN * kRowBytes;
constexpr int kSlotBytes = kABytes + kBBytes;
constexpr int kSlots = 9;                             // slices 0 and 1 twice (see below)
constexpr int kAcc = 8;                               // accumulator ring: 8 x 64 TMEM columns
constexpr uint32_t kSlCols = kAcc * kBN;
constexpr int kEpi = 16;                              // epilogue warps: 16 columns each
constexpr int kEC = kBN / (kEpi / 4);                 // columns of one epilogue warp
constexpr int kSlThreads = 32 * (kEpi + 2);
constexpr size_t kSlSmem = (size_t)kSlots * kSlotBytes + 1024;

__device__ __forceinline__ int slot_of(int s, int lt) { return (s < 2 && (lt & 1)) ? 7 + s : s; }

// ---------------------------------------------------------------------------
// The update.  A tile is 128 off-diagonal rows x 64 off-diagonal rows of one
// source panel x one digit block (K <= 64), whatever target panels its
// columns face (a 64-column tile faces five of them on average on a 48^3
// grid, where a tile per task was a quarter full): column R's entries go to
// colbase[R] + relmap[relbase[R] + row].  Roles of a CTA's eighteen warps, all walking the CTA's tiles:
//   warp 16 (one thread) TMA loads, one barrier per slice;
//   warp 17 (one thread) MMAs: group g's digit pairs into the next of eight
//                        accumulators, g = 6 first;
//   warps 0-15           drain each group as soon as it is complete (warp w:
//                        TMEM lanes 32 (w % 4) .., column blocks of 8 in
//                        turns), put the sums together in integers and
//                        subtract the tile from its target with reductions.
// Descending groups free slice g after group g, so the next tile's slices
// 6 .. 2 arrive while this tile's last groups run; slices 0 and 1, which
// every group needs, have two buffers each.
// What bounds it: a full tile's 28 pairs take 28 x 4 MMAs of 32 cycles
// (3,584 cycles), its drain about 50 integer instructions an element
// (3,200 cycles a warp scheduler), beside each other.  64^3 grid, 64-wide
// panels: all updates 36.5 ms (4.2e11 flops, 11 TFLOP/s; the FP64 unit's tiles
// in the task queue took most of that factorization's 537 ms, now 61.5).  Registers
// (96 a thread for 18 warps) spill: 36 bytes, for panels wider than 64 with their
// carried sums 196.
// ---------------------------------------------------------------------------
template <bool kWide>
__global__ void __launch_bounds__(kSlThreads, 1)
    update_sl_kernel(const __grid_constant__ CUtensorMap mapa, const __grid_constant__ CUtensorMap mapb,
                     int64_t oprows, int64_t exprows, const SlTile *__restrict__ tiles, int count, const int64_t *__restrict__ colbase,
                     const int64_t *__restrict__ relbase, const int32_t *__restrict__ relmap,
                     const int32_t *__restrict__ expa, const int32_t *__restrict__ expb, double *__restrict__ C,
                     int *err)
{
    extern __shared__ unsigned char smraw[];
    unsigned char *base =
        reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t full[kSlots], empty[kSlots], acc_full[kAcc], acc_empty[kAcc], drained;
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_fail;
    __shared__ int s_lt, s_slice;                      // the first load that was not issued
    __shared__ int64_t s_coff[kEpi][kEC], s_rel[kEpi][kEC];
    __shared__ int32_t s_eb[kEpi][kEC];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kSlots; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(&drained, 1);
        for (int b = 0; b < kAcc; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], kEpi);
        }
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(kSlCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem;

    if (warp == kEpi) {
        if (elect_one()) {
            int lt = 0, next = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < count && ok; t += gridDim.x) {
                const SlTile tl = tiles[t];
                for (int kx = 0; ok && (kx == 0 || (kWide && kx < tl.k)); kx += kK) {
#pragma unroll
                    for (int i = 0; i < kSlices; ++i) {
                        const int s = i < 2 ? i : 8 - i;   // 0, 1, 6, 5, 4, 3, 2: the order they fall free in
                        const int slot = slot_of(s, lt);
                        const int u = s < 2 ? lt >> 1 : lt;   // earlier uses of this buffer
                        if (u >= 1 && !mbar_wait_or(&empty[slot], (uint32_t)(u - 1) & 1u, &s_fail)) {
                            ok = false;
                            next = i;
                            break;
                        }
                        unsigned char *dst = base + slot * kSlotBytes;
                        mbar_expect_tx(&full[slot], kSlotBytes);
                        const int ra = tl.aop + (kWide ? kx / kK * tl.nrow : 0);
                        const int rb = tl.bop + (kWide ? kx / kK * tl.bstep : 0);
                        tma_load_2d(dst, &mapa, &full[slot], 0, (int)(s * oprows) + ra);
                        tma_load_2d(dst + kABytes, &mapb, &full[slot], 0, (int)(s * oprows) + rb);
                    }
                    lt += ok;
                }
            }
            if (!ok) s_fail = 1;
            s_lt = lt;
            s_slice = next;
        }
    } else if (warp == kEpi + 1) {
        if (elect_one()) {
            int lt = 0;
            const uint64_t desc0 = sw128_desc(smem_u32(base));
            uint32_t ng = 0;   // groups issued so far: the accumulator ring position
            bool ok = true;
            for (int t = blockIdx.x; t < count && ok; t += gridDim.x) {
                const SlTile tl = tiles[t];
                for (int kx = 0; kx == 0 || (kWide && kx < tl.k && ok); kx += kK, ++lt) {
                    const uint32_t idesc = idesc_f16((tl.ncol + 15) & ~15);
                    const int ksteps = (min(kK, tl.k - kx) + 15) / 16;
                    const uint64_t da0 = desc0 + (uint32_t)(2 * tl.achunk), db0 = desc0 + (uint32_t)(2 * tl.bchunk);
                    auto arrived = [&](int s) {
                        return mbar_wait_or(&full[slot_of(s, lt)], (uint32_t)(s < 2 ? lt >> 1 : lt) & 1u, &s_fail);
                    };
#pragma unroll 1
                    for (int g = kGroups - 1; g >= 0 && ok; --g, ++ng) {
                        const int a = (int)(ng % kAcc);
                        const uint32_t acc = tmem + (uint32_t)(a * kBN);
                        if (ng >= kAcc && !mbar_wait_or(&acc_empty[a], (ng / kAcc - 1) & 1u, &s_fail)) {
                            ok = false;
                            break;
                        }
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        uint32_t more = 0;
                        auto pair = [&](int s, int u) {
                            const uint64_t da = da0 + (uint32_t)(slot_of(s, lt) * (kSlotBytes >> 4));
                            const uint64_t db = db0 + (uint32_t)(slot_of(u, lt) * (kSlotBytes >> 4) + (kABytes >> 4));
                            mma<1>(acc, da, db, idesc, more);
                            if (ksteps > 1) mma<1>(acc, da + 2, db + 2, idesc, 1);
                            if (ksteps > 2) mma<1>(acc, da + 4, db + 4, idesc, 1);
                            if (ksteps > 3) mma<1>(acc, da + 6, db + 6, idesc, 1);
                            more = 1;
                        };
                        if (g == kGroups - 1) {
                            // the pairs as their slices arrive
                            ok = arrived(0) && arrived(6);
                            if (ok) {
                                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                                pair(0, 6), pair(6, 0);
                                ok = arrived(1) && arrived(5);
                            }
                            if (ok) {
                                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                                pair(1, 5), pair(5, 1);
                                ok = arrived(4) && arrived(3);
                            }
                            if (ok) {
                                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                                pair(3, 3);
                                ok = arrived(2);
                            }
                            if (ok) {
                                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                                pair(2, 4), pair(4, 2);
                            }
                            if (!ok) break;
                        } else {
#pragma unroll 1
                            for (int s = 0; s <= g; ++s) pair(s, g - s);
                        }
                        mma_commit(&acc_full[a]);
                        mma_commit(&empty[slot_of(g, lt)]);
                    }
                }
            }
            if (!ok) s_fail = 1;
            mma_commit(&drained);
        }
    } else {
        uint32_t ng = 0;
        const int quad = warp & 3, part = warp >> 2;
        const uint32_t tlane = tmem + ((uint32_t)(quad * 32) << 16);
        double carry[kWide ? kEC : 1];
        SlTile tl{};
        if ((int)blockIdx.x < count) tl = tiles[blockIdx.x];
        bool ok = true;
        for (int t = blockIdx.x; t < count && ok; t += gridDim.x) {
            const SlTile cur = tl;
            if (t + (int)gridDim.x < count) tl = tiles[t + gridDim.x];   // the next tile's, a tile ahead
            // this warp's columns kEC part .. + kEC - 1
            if (lane < kEC) {
                const int c = min(kEC * part + lane, cur.ncol - 1);
                s_coff[warp][lane] = colbase[cur.brow + c];
                s_rel[warp][lane] = relbase[cur.brow + c] + cur.arow;
            }
            const int r = quad * 32 + lane;
            const bool row_ok = r < cur.nrow;
            // nothing to do for a warp without columns, or without rows on or
            // below them: it only passes the groups on
            const bool use = kEC * part < cur.ncol && quad * 32 < cur.nrow && quad * 32 + 31 + cur.diff >= kEC * part;
            auto group_ready = [&]() {
                ok = mbar_wait_or(&acc_full[ng % kAcc], (ng / kAcc) & 1u, &s_fail) && ok;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            };
            auto group_read = [&]() {
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(&acc_empty[ng % kAcc]);
                ++ng;
            };
            for (int kx = 0; kx == 0 || (kWide && kx < cur.k); kx += kK) {
                const int64_t blk = kWide ? (int64_t)(kx / kK) * exprows : 0;
                if (lane < kEC) s_eb[warp][lane] = expb[blk + cur.brow + min(kEC * part + lane, cur.ncol - 1)];
                const int32_t ea = row_ok ? expa[blk + cur.arow + r] : 0;
                __syncwarp();
                if (!use) {
#pragma unroll 1
                    for (int g = 0; g < kGroups; ++g) {
                        group_ready();
                        group_read();
                    }
                    continue;
                }
                Sum sum[kEC];
                auto drain = [&](auto gc) {
                    constexpr int G = decltype(gc)::value;
                    group_ready();
                    uint32_t v[kEC];
                    tmem_read16(tlane + (uint32_t)((int)(ng % kAcc) * kBN + kEC * part), v);
                    group_read();
#pragma unroll
                    for (int i = 0; i < kEC; ++i) add_group<G>(sum[i], __uint_as_float(v[i]));
                };
                drain(std::integral_constant<int, 6>());
                drain(std::integral_constant<int, 5>());
                drain(std::integral_constant<int, 4>());
                drain(std::integral_constant<int, 3>());
                drain(std::integral_constant<int, 2>());
                drain(std::integral_constant<int, 1>());
                drain(std::integral_constant<int, 0>());
                if (ok && row_ok) {
#pragma unroll
                    for (int i = 0; i < kEC; ++i) {
                        const int c = kEC * part + i;
                        if (c < cur.ncol && r + cur.diff >= c) {
                            double v = finish(sum[i], ea + s_eb[warp][i], true);
                            // panels wider than a digit block (kWide): the blocks' products
                            // are added up first, so that the target is rounded once
                            if constexpr (kWide) {
                                if (kx > 0) v += carry[i];
                                carry[i] = v;
                                if (kx + kK < cur.k) continue;
                            }
                            atomicAdd(C + s_coff[warp][i] + relmap[s_rel[warp][i] + r], v);
                        }
                    }
                }
                __syncwarp();
            }
        }
        if (!ok) s_fail = 1;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (s_fail) {
        // one of the roles gave up: no MMA and no load may be left in flight when the
        // accumulators are freed and the CTA's shared memory is another's
        mbar_wait(&drained, 0);
        for (int i = 0; i < kSlices; ++i) {
            const int s = i < 2 ? i : 8 - i, n = s_lt + (i < s_slice ? 1 : 0);   // (see the loads' order)
            const int even = s < 2 ? (n + 1) / 2 : n, odd = s < 2 ? n / 2 : 0;
            if (even > 0) mbar_wait(&full[s], (uint32_t)(even - 1) & 1u);
            if (odd > 0) mbar_wait(&full[7 + s], (uint32_t)(odd - 1) & 1u);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0 && s_fail) atomicExch(err, 1);
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kSlCols));
}

// ---------------------------------------------------------------------------
// Panel TRSM in FP64 as a product with the inverted diagonal block (the forms
// TRSM_LLT, TRSM_LDLT and, for panels up to 64 wide and without the operand
// copy, TRSM_RIGHT_LINV of blocks.cuh), 64 rows a CTA: X's rows and the
// inverse's rows are cut into slices in shared memory, the 28 digit pairs run
// on the tensor cores, the result is put together as in the update, written
// back in place and written again as slices for the updates.  Each row lies
// twice in the 128-row A tile, so that all four TMEM lane quadrants hold
// results: quadrants 0 and 1 drain columns 0 .. 31, 2 and 3 the rest.
// Both operands' columns k are scaled by powers of two first, X's by the
// inverse of about sqrt(a_kk) (LDL^T: of the largest l(k, m) sqrt(|d_m|)), whose
// exponents the diagonal block's kernel leaves in rowexp, and the inverse's by
// the opposite, which the products do not see: X(i, k) grows with the scale of
// unknown k and Linv(j, k) falls with it, and without this one large entry of
// each row, at different k, would set the rows' exponents.  (Not by the pivot
// l_kk, which elimination inside the block may leave far below sqrt(a_kk): on
// smooth covariance matrices of 256 points and a nugget of 1e-8 that left the
// entries of L L^T 2.9e-12 off, where FP64 multiply-adds leave 4.9e-14.)  LDL^T's two operand
// copies for the update are cut with such scales, too: L(i, k) falls and
// (D L^T)(j, k) grows with the scale of unknown k, so L's column k is taken
// times about sqrt(|d_k|) and D L^T's divided by it (unscaled, the update's
// error was that of FP64 multiply-adds times the ratio of the largest to the
// smallest scale in the panel).  Cholesky's L has no such factor.
// Panels wider than 64 go by 64-column blocks, the last one first (block c
// needs the old X of blocks <= c), the partial sums of their digit blocks
// added in FP64.  Bound by the integer work of cutting and joining (about 80
// instructions an element) and, at the top of the tree, where a level has a
// few dozen CTAs, by latency and instruction fetches: 8 elements a thread
// and one loop over both operands keep the code short (a 64-row CTA 17 us; 128
// rows with straight-line code 35).  64^3 grid: 11.9 ms for 245 levels.
// ---------------------------------------------------------------------------
constexpr int kTrRows = 64;
constexpr int kTrThreads = 512;
constexpr int kTC = kK / (kTrThreads / kTrRows);       // columns of one row a thread
constexpr size_t kTrSmem = (size_t)kSlices * kSlotBytes + 1024;
static_assert(kTC == 8, "one 16-byte word of digits a thread and slice");

// Eight neighbouring digits of one operand row, all slices: 16 bytes each.
__device__ __forceinline__ void digits8(const double *x, int field, uint32_t (&w)[kSlices][4],
                                        const int *scale = nullptr)
{
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        uint32_t d[kSlices];
        digits2(fixed_biased(x[2 * q], field, scale ? scale[2 * q] : 0),
                fixed_biased(x[2 * q + 1], field, scale ? scale[2 * q + 1] : 0), d);
#pragma unroll
        for (int s = 0; s < kSlices; ++s) w[s][q] = d[s];
    }
}

// One thread: all digit pairs of an A tile (slices of kABytes) and a B tile
// (kBBytes), n columns, group g into accumulator g; done[g] completes with
// group g, the last first.
__device__ __forceinline__ void issue_pairs(uint32_t tmem, const unsigned char *sA, const unsigned char *sB, int n,
                                            int ksteps, uint64_t *done)
{
    const uint32_t idesc = idesc_f16(n);
    const uint64_t a0 = sw128_desc(smem_u32(sA)), b0 = sw128_desc(smem_u32(sB));
#pragma unroll 1
    for (int g = kGroups - 1; g >= 0; --g) {
        const uint32_t acc = tmem + (uint32_t)(g * kBN);
#pragma unroll 1
        for (int s = 0; s <= g; ++s) {
            const uint64_t da = a0 + (uint32_t)(s * (kABytes >> 4));
            const uint64_t db = b0 + (uint32_t)((g - s) * (kBBytes >> 4));
            mma<1>(acc, da, db, idesc, s > 0);
            if (ksteps > 1) mma<1>(acc, da + 2, db + 2, idesc, 1);
            if (ksteps > 2) mma<1>(acc, da + 4, db + 4, idesc, 1);
            if (ksteps > 3) mma<1>(acc, da + 6, db + 6, idesc, 1);
        }
        mma_commit(&done[g]);
    }
}

__global__ void __launch_bounds__(kTrThreads, 1)
    trsm_sl_kernel(DevPlan p, const RowChunk *__restrict__ chunks, const double *__restrict__ Dinv,
                   double *__restrict__ X, double *__restrict__ Wout, int mode, const int32_t *__restrict__ rowexp,
                   __half *__restrict__ opa,
                   __half *__restrict__ opb, int32_t *__restrict__ expa, int32_t *__restrict__ expb,
                   const SlPlace *__restrict__ places, int64_t oprows, int64_t exprows, int *err)
{
    extern __shared__ unsigned char smraw[];
    unsigned char *base =
        reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~(uintptr_t)1023);
    unsigned char *sA = base, *sB = base + kSlices * kABytes;
    __shared__ __align__(8) uint64_t done[kGroups];
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail;
    __shared__ int s_f[2][8][kTrRows];                // exponent fields, parts of a row: X's, the inverse's
    __shared__ int32_t s_e[2][kTrRows];
    __shared__ int s_sc[kMaxWidth + kK];              // scales of the products' columns (up to whole digit blocks),
    __shared__ int s_sd[kK];                          // and LDL^T's of the operand copies'
    const RowChunk ch = chunks[blockIdx.x];
    const bool ldlt = mode == TRSM_LDLT, right = mode == TRSM_RIGHT_LINV;
    const SlPlace at = right ? SlPlace{-1, 0, 0, 0} : places[blockIdx.x];
    const int pid = ch.panel, w = p.pw[pid], h = p.ph[pid];
    const int nr = min(kTrRows, h - ch.r0);
    double *Xg = X + p.pval[pid] + ch.r0;
    const double *Mi = Dinv + p.pinv[pid];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (tid == 0) {
        for (int g = 0; g < kGroups; ++g) mbar_init(&done[g], 1);
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(kSlCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (const int k = tid - 32; k >= 0 && k < kMaxWidth + kK) {      // (warp 0 allocates the accumulators)
        // column k of X times 2^s_sc, column k of the inverse divided by it
        const int e = k < w && !right ? rowexp[p.pfcol[pid] + k] : 0;
        s_sc[k] = e < -kNoExp / 4 || e > kNoExp / 4 ? 0 : -e;        // (rows of zeros, infinities, NaN)
        if (k < kK) {
            const int d = ldlt && k < w ? lead_exp(high_word(X + p.pval[pid] + k + (int64_t)k * h)) : 0;
            s_sd[k] = d < -kNoExp / 2 || d > kNoExp / 2 ? 0 : d >> 1;
        }
    }
    const int rs = tid & (kTrRows - 1), ps = tid / kTrRows;          // staging: row and 8-column part
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem;

    const int quad = warp & 3;
    const int r = 32 * (quad & 1) + lane, part = 4 * (quad >> 1) + (warp >> 2);   // results: row and part
    const bool row_ok = r < nr;
    const int nblk = (w + kK - 1) / kK;
    uint32_t phase = 0;
    for (int c0 = (nblk - 1) * kK; c0 >= 0; c0 -= kK) {
        double out[kTC];
        for (int k0 = 0; k0 <= c0; k0 += kK) {
            const int ksteps = (min(kK, w - k0) + 15) / 16;
            // operand 0: X(rs, k0 ..), operand 1: the inverse's row c0 + rs
            // (B(k, j) = Linv(j, k)); eight columns of one row a thread
#pragma unroll 1
            for (int o = 0; o < 2; ++o) {
                const int j = c0 + rs, k1 = k0 + kTC * ps;
                const double *src = o == 0  ? Xg + rs + (int64_t)k1 * h
                                    : right ? Mi + k1 + (int64_t)j * w    // L^{-1}: B(k, j) = Linv(k, j)
                                            : Mi + j + (int64_t)k1 * w;
                const int64_t ld = o == 0 ? h : (right ? 1 : w);
                // columns read: k < klim and, for L^{-1}, k >= j
                const int klim = o == 0 ? (rs < nr ? w : 0) : (j < w ? (right ? w : j + 1) : 0);
                const int kmin = o == 1 && right ? j : 0;
                double x[kTC];
#pragma unroll
                for (int q = 0; q < kTC; ++q)
                    x[q] = k1 + q < klim && k1 + q >= kmin ? __ldcg(src + q * ld) : 0.0;
                if (o == 1 && ldlt) {   // unit diagonal (1/d is stored there)
#pragma unroll
                    for (int q = 0; q < kTC; ++q)
                        if (k1 + q == j) x[q] = 1.0;
                }
                int sc[kTC];
#pragma unroll
                for (int q = 0; q < kTC; ++q) sc[q] = o == 0 ? s_sc[k1 + q] : -s_sc[k1 + q];
                int f = kFieldZero;
#pragma unroll
                for (int q = 0; q < kTC; ++q) f = max(f, exp_field(x[q], sc[q]));
                s_f[o][ps][rs] = f;
                __syncthreads();
#pragma unroll
                for (int q = 0; q < 8; ++q) f = max(f, s_f[o][q][rs]);
                if (ps == 0) s_e[o][rs] = row_exp(f);
                if (kTC * ps < 16 * ksteps) {
                    uint32_t wd[kSlices][4];
                    digits8(x, f, wd, sc);
                    unsigned char *t = (o == 0 ? sA : sB) + rs * kRowBytes + ((16 * ps) ^ ((rs & 7) << 4));
                    const int step = o == 0 ? kABytes : kBBytes;
#pragma unroll
                    for (int s = 0; s < kSlices; ++s) {
                        const uint4 v = make_uint4(wd[s][0], wd[s][1], wd[s][2], wd[s][3]);
                        *reinterpret_cast<uint4 *>(t + s * step) = v;
                        if (o == 0) *reinterpret_cast<uint4 *>(t + s * step + kTrRows * kRowBytes) = v;
                    }
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncthreads();
            if (warp == 0) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                if (elect_one()) issue_pairs(tmem, sA, sB, kBN, ksteps, done);
                __syncwarp();
            }
            Sum sum[kTC];
            auto drain = [&](auto gc) {
                constexpr int G = decltype(gc)::value;
                if (!mbar_wait(&done[G], phase)) s_fail = 1;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                uint32_t v[kTC];
                tmem_read8(tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(G * kBN + kTC * part), v);
#pragma unroll
                for (int i = 0; i < kTC; ++i) add_group<G>(sum[i], __uint_as_float(v[i]));
            };
            drain(std::integral_constant<int, 6>());
            drain(std::integral_constant<int, 5>());
            drain(std::integral_constant<int, 4>());
            drain(std::integral_constant<int, 3>());
            drain(std::integral_constant<int, 2>());
            drain(std::integral_constant<int, 1>());
            drain(std::integral_constant<int, 0>());
            phase ^= 1u;
            const int32_t ea = s_e[0][r];
#pragma unroll
            for (int q = 0; q < kTC; ++q) {
                const double v = finish(sum[q], ea + s_e[1][kTC * part + q], false);
                if (k0 == 0) out[q] = v;
                else out[q] += v;
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncthreads();   // the accumulators, the slices and the exponents may be written again
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (s_fail) break;
        }
        if (s_fail) break;
        // columns j0 .. j0 + 7 of row r: back in place, then as slices
        const int j0 = c0 + kTC * part;
#pragma unroll 1
        for (int o = ldlt ? 1 : 0; o >= 0; --o) {
            // LDL^T: out = X l^{-T} is the D L^T row (the update's B operand, o = 1);
            // then L = out D^{-1}
            if (ldlt && o == 0) {
#pragma unroll
                for (int q = 0; q < kTC; ++q)
                    if (j0 + q < w) out[q] *= __ldcg(Mi + (j0 + q) + (int64_t)(j0 + q) * w);
            }
            double *dst = (o == 1 ? Wout + p.pval[pid] + ch.r0 : Xg) + r + (int64_t)j0 * h;
            int sc[kTC], f = kFieldZero;
#pragma unroll
            for (int q = 0; q < kTC; ++q) {
                sc[q] = ldlt ? (o == 1 ? -s_sd[kTC * part + q] : s_sd[kTC * part + q]) : 0;   // (at most 64 wide)
                if (j0 + q >= w) out[q] = 0.0;
                else if (row_ok) dst[(int64_t)q * h] = out[q];
                f = max(f, exp_field(out[q], sc[q]));
            }
            if (at.row < 0) continue;   // no operand copy
            s_f[0][part][r] = f;
            __syncthreads();
#pragma unroll
            for (int q = 0; q < 8; ++q) f = max(f, s_f[0][q][r]);
            __syncthreads();
            if (row_ok) {
                const int64_t orow = p.prow[pid] + ch.r0 + r;
                if (part == 0) (o == 1 ? expb : expa)[(int64_t)(c0 / kK) * exprows + orow] = row_exp(f);
                if (kTC * part >= at.cols) continue;
                uint32_t wd[kSlices][4];
                digits8(out, f, wd, sc);
                __half *op = (o == 1 ? opb : opa) + ((int64_t)at.row + r + c0 / kK * at.step) * kK + 16 * at.chunk +
                             kTC * part;
#pragma unroll
                for (int s = 0; s < kSlices; ++s)
                    *reinterpret_cast<uint4 *>(op + (int64_t)s * oprows * kK) =
                        make_uint4(wd[s][0], wd[s][1], wd[s][2], wd[s][3]);
            }
        }
    }
    if (s_fail) mbar_wait(&done[0], phase ^ 1u);   // no MMA in flight when the accumulators are freed
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (tid == 0 && s_fail) atomicExch(err, 1);
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kSlCols));
}

// ---------------------------------------------------------------------------
// Selected inversion, Z_RJ = -Z_RR Lh for 128 rows i of one panel (selinv.cu
// says what the quantities are): per 64 columns j of Z_RR the gathered 128 x 64
// block of Z and the 64 x w block of Lh are cut into slices, multiplied, and the
// product is added in FP64 to the running result.  Z(i, j) lies in the column
// of the lower of the two rows: at colbase[j] + relmap[relbase[j] + i] for
// i >= j.  Column j of Z is scaled by the leading power of two of L(j, j) and
// row j of Lh by its inverse (see the TRSM).  The next block's entries of Z are
// loaded before this block's sums are drained.  Split over j as in the CUDA-core
// form (gridDim.y parts, added into a zeroed Z).
// Bound by the integer work (about 68 instructions an entry of Z, 72 a result
// and block); the FP64 unit would take 300,000 cycles for a block that this
// does in about 15,000.  48^3 grid: the whole selected inverse 257 -> 46 ms, of
// which these products 39 (150 levels of about 33 us fixed cost each).  Registers
// (128 a thread) spill 240 bytes.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kTrThreads, 1)
    selinv_sl_kernel(DevPlan p, const RowChunk *__restrict__ chunks, const int64_t *__restrict__ colbase,
                     const int64_t *__restrict__ relbase, const int32_t *__restrict__ dexp,
                     const double *__restrict__ Lh, double *__restrict__ Z, int *err)
{
    extern __shared__ unsigned char smraw[];
    unsigned char *base =
        reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~(uintptr_t)1023);
    unsigned char *sA = base, *sB = base + kSlices * kABytes;
    __shared__ __align__(8) uint64_t done[kSlices];
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail;
    __shared__ int s_f[4][kM], s_g[8][kBN];
    __shared__ int32_t s_eb[kBN];
    __shared__ int s_sc[2][kK];                        // this block's column scales, and the next one's
    __shared__ int64_t s_cb[2][kK], s_rb[2][kK];
    constexpr int kQ = kK / (kTrThreads / kM);         // 16 entries of one row of Z a thread
    const RowChunk ch = chunks[blockIdx.x];
    const int pid = ch.panel, w = p.pw[pid], h = p.ph[pid];
    const int nk = (h - w + kK - 1) / kK, per = (nk + (int)gridDim.y - 1) / (int)gridDim.y;
    const int b0 = min(nk, (int)blockIdx.y * per), b1 = min(nk, b0 + per);
    if (b0 >= b1) return;
    const int64_t prow = p.prow[pid];
    const int tid = threadIdx.x, warp = tid >> 5;

    if (tid == 0) {
        for (int g = 0; g < kSlices; ++g) mbar_init(&done[g], 1);
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(kSlCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    const int r = tid & (kM - 1), part = tid / kM, i = ch.r0 + r;
    const bool row_ok = i < h;
    const int64_t cbi = row_ok ? colbase[prow + i] : 0, rbi = row_ok ? relbase[prow + i] + prow : 0;
    auto columns = [&](int b) {                        // the 64 columns of block b
        if (tid < kK) {
            const int j = w + b * kK + tid;
            const bool in = j < h;
            s_cb[b & 1][tid] = in ? colbase[prow + j] : 0;
            s_rb[b & 1][tid] = in ? relbase[prow + j] + prow : 0;
            s_sc[b & 1][tid] = in ? dexp[p.rows[prow + j]] : 0;
        }
    };
    double x[kQ];
    auto gather = [&](int b) {
#pragma unroll
        for (int q = 0; q < kQ; ++q) {
            const int k = kQ * part + q, j = w + b * kK + k;
            double v = 0.0;
            if (row_ok && j < h)
                v = i >= j ? Z[s_cb[b & 1][k] + p.relmap[s_rb[b & 1][k] + i]] : Z[cbi + p.relmap[rbi + j]];
            x[q] = v;
        }
    };
    columns(b0);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem;
    const uint32_t tlane = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    gather(b0);
    double acc[kQ];
#pragma unroll
    for (int q = 0; q < kQ; ++q) acc[q] = 0.0;
    uint32_t phase = 0;
    for (int b = b0; b < b1; ++b) {
        const int j0 = w + b * kK, ksteps = (min(kK, h - j0) + 15) / 16;
        int32_t ea;
        {
            int sc[kQ], f = kFieldZero;
#pragma unroll
            for (int q = 0; q < kQ; ++q) sc[q] = s_sc[b & 1][kQ * part + q];
#pragma unroll
            for (int q = 0; q < kQ; ++q) f = max(f, exp_field(x[q], sc[q]));
            s_f[part][r] = f;
            __syncthreads();
            f = max(max(s_f[0][r], s_f[1][r]), max(s_f[2][r], s_f[3][r]));
            ea = row_exp(f);
            if (part < ksteps) {
#pragma unroll 1
                for (int q8 = 0; q8 < kQ; q8 += 8) {
                    uint32_t wd[kSlices][4];
                    if (q8 == 0) digits8(x, f, wd, sc);
                    else digits8(x + 8, f, wd, sc + 8);
                    unsigned char *t = sA + r * kRowBytes + (((kQ * part + q8) * 2) ^ ((r & 7) << 4));
#pragma unroll
                    for (int s = 0; s < kSlices; ++s)
                        *reinterpret_cast<uint4 *>(t + s * kABytes) = make_uint4(wd[s][0], wd[s][1], wd[s][2], wd[s][3]);
                }
            }
        }
        {
            const int c = tid & 63, pb = tid >> 6;     // eight entries of Lh's column c
            double y[8];
            int sc[8], f = kFieldZero;
            const double *src = Lh + p.pval[pid] + (int64_t)c * h + j0 + 8 * pb;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                sc[q] = -s_sc[b & 1][8 * pb + q];
                y[q] = c < w && j0 + 8 * pb + q < h ? src[q] : 0.0;
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) f = max(f, exp_field(y[q], sc[q]));
            s_g[pb][c] = f;
            __syncthreads();
#pragma unroll
            for (int q = 0; q < 8; ++q) f = max(f, s_g[q][c]);
            if (pb == 0) s_eb[c] = row_exp(f);
            if (8 * pb < 16 * ksteps) {
                uint32_t wd[kSlices][4];
                digits8(y, f, wd, sc);
                unsigned char *t = sB + c * kRowBytes + ((16 * pb) ^ ((c & 7) << 4));
#pragma unroll
                for (int s = 0; s < kSlices; ++s)
                    *reinterpret_cast<uint4 *>(t + s * kBBytes) = make_uint4(wd[s][0], wd[s][1], wd[s][2], wd[s][3]);
            }
        }
        if (b + 1 < b1) columns(b + 1);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if (warp == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (elect_one()) issue_pairs(tmem, sA, sB, (w + 15) & ~15, ksteps, done);
            __syncwarp();
        }
        if (b + 1 < b1) gather(b + 1);
        // eight columns at a time (registers); columns past w hold stale sums
        if (kQ * part < w) {
#pragma unroll
            for (int q8 = 0; q8 < kQ; q8 += 8) {
                Sum sum[8];
                auto drain = [&](auto gc) {
                    constexpr int G = decltype(gc)::value;
                    if (!mbar_wait(&done[G], phase)) s_fail = 1;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    uint32_t v[8];
                    tmem_read8(tlane + (uint32_t)(G * kBN + kQ * part + q8), v);
#pragma unroll
                    for (int q = 0; q < 8; ++q) add_group<G>(sum[q], __uint_as_float(v[q]));
                };
                drain(std::integral_constant<int, 6>());
                drain(std::integral_constant<int, 5>());
                drain(std::integral_constant<int, 4>());
                drain(std::integral_constant<int, 3>());
                drain(std::integral_constant<int, 2>());
                drain(std::integral_constant<int, 1>());
                drain(std::integral_constant<int, 0>());
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    acc[q8 + q] += finish(sum[q], ea + s_eb[kQ * part + q8 + q], true);
            }
        }
        // (a warp without columns still has to see the block's last product done)
        if (!mbar_wait(&done[0], phase)) s_fail = 1;
        phase ^= 1u;
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (s_fail) break;
    }
    if (row_ok && !s_fail) {
        double *dst = Z + p.pval[pid] + i;
#pragma unroll
        for (int q = 0; q < kQ; ++q) {
            const int c = kQ * part + q;
            if (c >= w) continue;
            if (gridDim.y == 1) dst[(int64_t)c * h] = acc[q];
            else atomicAdd(dst + (int64_t)c * h, acc[q]);
        }
    }
    if (s_fail) mbar_wait(&done[0], phase ^ 1u);   // no MMA in flight when the accumulators are freed
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (tid == 0 && s_fail) atomicExch(err, 1);
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kSlCols));
}

// Z_JJ -= Lh^T Z_RJ over the 64-row blocks blockIdx.y, blockIdx.y + gridDim.y,
// ... of R: both operands are columns of 64 rows cut into slices; Lh's lie
// twice in the A tile, as X does in the TRSM.  The lower triangle is kept and
// added to both triangles of Z_JJ, which holds Linv^T Linv.
__global__ void __launch_bounds__(kTrThreads, 1)
    selinv_diag_sl_kernel(DevPlan p, const int32_t *__restrict__ panels, const int32_t *__restrict__ dexp,
                          const double *__restrict__ Lh, double *__restrict__ Z, int *err)
{
    extern __shared__ unsigned char smraw[];
    unsigned char *base =
        reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~(uintptr_t)1023);
    unsigned char *sA = base, *sB = base + kSlices * kABytes;
    __shared__ __align__(8) uint64_t done[kSlices];
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail;
    __shared__ int s_f[2][8][kTrRows];
    __shared__ int32_t s_e[2][kTrRows];
    const int pid = panels[blockIdx.x], w = p.pw[pid], h = p.ph[pid];
    const int nk = (h - w + kK - 1) / kK;
    if ((int)blockIdx.y >= nk) return;
    const int64_t pv = p.pval[pid];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (tid == 0) {
        for (int g = 0; g < kSlices; ++g) mbar_init(&done[g], 1);
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(kSlCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem;
    const int cs = tid & (kTrRows - 1), ps = tid / kTrRows;          // staging: column and 8-row part
    const int quad = warp & 3;
    const int a = 32 * (quad & 1) + lane, part = 4 * (quad >> 1) + (warp >> 2);
    double acc[kTC];
#pragma unroll
    for (int q = 0; q < kTC; ++q) acc[q] = 0.0;
    uint32_t phase = 0;
    for (int b = blockIdx.y; b < nk; b += gridDim.y) {
        const int j0 = w + b * kK + kTC * ps, ksteps = (min(kK, h - w - b * kK) + 15) / 16;
#pragma unroll 1
        for (int o = 0; o < 2; ++o) {
            const double *src = (o == 0 ? Lh : Z) + pv + (int64_t)cs * h + j0;
            double x[kTC];
            int sc[kTC], f = kFieldZero;
#pragma unroll
            for (int q = 0; q < kTC; ++q) {
                x[q] = cs < w && j0 + q < h ? src[q] : 0.0;
                sc[q] = j0 + q < h ? dexp[p.rows[p.prow[pid] + j0 + q]] : 0;   // row j of Lh divided, of Z times
                if (o == 0) sc[q] = -sc[q];
            }
#pragma unroll
            for (int q = 0; q < kTC; ++q) f = max(f, exp_field(x[q], sc[q]));
            s_f[o][ps][cs] = f;
            __syncthreads();
#pragma unroll
            for (int q = 0; q < 8; ++q) f = max(f, s_f[o][q][cs]);
            if (ps == 0) s_e[o][cs] = row_exp(f);
            if (kTC * ps < 16 * ksteps) {
                uint32_t wd[kSlices][4];
                digits8(x, f, wd, sc);
                unsigned char *t = (o == 0 ? sA : sB) + cs * kRowBytes + ((16 * ps) ^ ((cs & 7) << 4));
                const int step = o == 0 ? kABytes : kBBytes;
#pragma unroll
                for (int s = 0; s < kSlices; ++s) {
                    const uint4 v = make_uint4(wd[s][0], wd[s][1], wd[s][2], wd[s][3]);
                    *reinterpret_cast<uint4 *>(t + s * step) = v;
                    if (o == 0) *reinterpret_cast<uint4 *>(t + s * step + kTrRows * kRowBytes) = v;
                }
            }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if (warp == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (elect_one()) issue_pairs(tmem, sA, sB, (w + 15) & ~15, ksteps, done);
            __syncwarp();
        }
        Sum sum[kTC];
        auto drain = [&](auto gc) {
            constexpr int G = decltype(gc)::value;
            if (!mbar_wait(&done[G], phase)) s_fail = 1;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            uint32_t v[kTC];
            tmem_read8(tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(G * kBN + kTC * part), v);
#pragma unroll
            for (int i = 0; i < kTC; ++i) add_group<G>(sum[i], __uint_as_float(v[i]));
        };
        drain(std::integral_constant<int, 6>());
        drain(std::integral_constant<int, 5>());
        drain(std::integral_constant<int, 4>());
        drain(std::integral_constant<int, 3>());
        drain(std::integral_constant<int, 2>());
        drain(std::integral_constant<int, 1>());
        drain(std::integral_constant<int, 0>());
        phase ^= 1u;
        const int32_t ea = s_e[0][a];
#pragma unroll
        for (int q = 0; q < kTC; ++q) acc[q] += finish(sum[q], ea + s_e[1][kTC * part + q], true);
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (s_fail) break;
    }
    if (!s_fail && a < w) {
#pragma unroll
        for (int q = 0; q < kTC; ++q) {
            const int c = kTC * part + q;
            if (c > a) continue;
            atomicAdd(&Z[pv + a + (int64_t)c * h], acc[q]);
            if (c < a) atomicAdd(&Z[pv + c + (int64_t)a * h], acc[q]);
        }
    }
    if (s_fail) mbar_wait(&done[0], phase ^ 1u);   // no MMA in flight when the accumulators are freed
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (tid == 0 && s_fail) atomicExch(err, 1);
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kSlCols));
}

// Leading exponents of L's diagonal, by column.
__global__ void diag_exp_kernel(DevPlan p, const double *__restrict__ L, int32_t *__restrict__ dexp)
{
    for (int q = blockIdx.x; q < p.npanels; q += gridDim.x) {
        const int w = p.pw[q], h = p.ph[q];
        for (int k = threadIdx.x; k < w; k += blockDim.x)
            dexp[p.pfcol[q] + k] = ((__double2hiint(L[p.pval[q] + k + (int64_t)k * h]) >> 20) & 0x7FF) - 1023;
    }
}

// ---------------------------------------------------------------------------
// Small tasks in FP64 on the CUDA cores, one warp a task: the lower
// trapezoid's entries in turns over the lanes, column by column (neighbouring
// lanes read neighbouring rows), straight from L2.  A 64 x 64 tile of such a
// task is mostly padding: the leaves' tasks have a few hundred multiply-adds.
// 64^3 grid: 0.65 ms for four levels' tasks.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) update_small_kernel(DevPlan p, const DevTask *__restrict__ tasks,
                                                           const int32_t *__restrict__ ids, int count,
                                                           const double *__restrict__ Aop,
                                                           const double *__restrict__ Bop, double *__restrict__ C)
{
    const int wi = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (wi >= count) return;
    const DevTask tk = tasks[ids[wi]];
    const int h = p.ph[tk.src], K = p.pw[tk.src];
    const int M = h - tk.r0, N = tk.r1 - tk.r0, hT = p.ph[tk.tgt];
    const double *A = Aop + p.pval[tk.src] + tk.r0, *B = Bop + p.pval[tk.src] + tk.r0;
    const int32_t *srow = p.rows + p.prow[tk.src] + tk.r0;
    const int32_t *rmap = p.relmap + tk.relmap_off;
    double *Ct = C + p.pval[tk.tgt] - p.pfcol[tk.tgt] * hT;
    int j = 0, rem = lane;
    while (j < N && rem >= M - j) {
        rem -= M - j;
        ++j;
    }
    while (j < N) {
        const int i = j + rem;
        double s = 0.0;
#pragma unroll 4
        for (int k = 0; k < K; ++k) s = fma(A[i + (int64_t)k * h], B[j + (int64_t)k * h], s);
        atomicAdd(Ct + rmap[i] + (int64_t)srow[j] * hT, -s);
        rem += 32;
        while (j < N && rem >= M - j) {
            rem -= M - j;
            ++j;
        }
    }
}

}  // namespace

void launch_update_sl(const void *mapa, const void *mapb, int64_t oprows, int64_t exprows, const DevPlan &p,
                      const SlTile *tiles, int count, const int64_t *colbase, const int64_t *relbase, const int32_t *expa,
                      const int32_t *expb, double *C, int *err, int per_cta, int wmax, cudaStream_t s)
{
    if (count <= 0) return;
    static int nsm = 0;
    if (!nsm) {
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        cudaFuncSetAttribute(update_sl_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSlSmem);
        cudaFuncSetAttribute(update_sl_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSlSmem);
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        nsm = std::max(v, 1);
    }
    int grid = std::min(count, nsm);
    if (per_cta > 0) grid = std::max(grid, (count + per_cta - 1) / per_cta);
    const CUtensorMap &ma = *reinterpret_cast<const CUtensorMap *>(mapa);
    const CUtensorMap &mb = *reinterpret_cast<const CUtensorMap *>(mapb);
    if (wmax > kK)
        update_sl_kernel<true><<<grid, kSlThreads, kSlSmem, s>>>(ma, mb, oprows, exprows, tiles, count, colbase, relbase,
                                                                 p.relmap, expa, expb, C, err);
    else
        update_sl_kernel<false><<<grid, kSlThreads, kSlSmem, s>>>(ma, mb, oprows, exprows, tiles, count, colbase, relbase,
                                                                  p.relmap, expa, expb, C, err);
}

void launch_trsm_sl(const DevPlan &p, const RowChunk *chunks, int count, const double *Dinv, double *X, double *Wout,
                    int mode, const int32_t *rowexp, void *opa, void *opb, int32_t *expa, int32_t *expb,
                    const SlPlace *places, int64_t oprows, int64_t exprows, int *err, cudaStream_t s)
{
    if (count <= 0) return;
    static bool once = false;
    if (!once) {
        cudaFuncSetAttribute(trsm_sl_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTrSmem);
        once = true;
    }
    trsm_sl_kernel<<<count, kTrThreads, kTrSmem, s>>>(p, chunks, Dinv, X, Wout, mode, rowexp, (__half *)opa, (__half *)opb,
                                                      expa, expb, places, oprows, exprows, err);
}

void launch_selinv_sl(const DevPlan &p, const RowChunk *chunks, int count, int nsplit, const int64_t *colbase,
                      const int64_t *relbase, const int32_t *dexp, const double *Lh, double *Z, int *err,
                      cudaStream_t s)
{
    if (count <= 0) return;
    static bool once = false;
    if (!once) {
        cudaFuncSetAttribute(selinv_sl_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTrSmem);
        once = true;
    }
    selinv_sl_kernel<<<dim3(count, nsplit), kTrThreads, kTrSmem, s>>>(p, chunks, colbase, relbase, dexp, Lh, Z, err);
}

void launch_selinv_diag_sl(const DevPlan &p, const int32_t *panels, int count, int nsplit, const int32_t *dexp,
                           const double *Lh, double *Z, int *err, cudaStream_t s)
{
    if (count <= 0) return;
    static bool once = false;
    if (!once) {
        cudaFuncSetAttribute(selinv_diag_sl_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTrSmem);
        once = true;
    }
    selinv_diag_sl_kernel<<<dim3(count, nsplit), kTrThreads, kTrSmem, s>>>(p, panels, dexp, Lh, Z, err);
}

void launch_diag_exp(const DevPlan &p, const double *L, int32_t *dexp, cudaStream_t s)
{
    if (p.npanels > 0) diag_exp_kernel<<<std::min(p.npanels, 152 * 8), 64, 0, s>>>(p, L, dexp);
}

void launch_update_small(const DevPlan &p, const DevTask *tasks, const int32_t *ids, int count, const double *Aop,
                         const double *Bop, double *C, cudaStream_t s)
{
    if (count <= 0) return;
    update_small_kernel<<<(count + 7) / 8, 256, 0, s>>>(p, tasks, ids, count, Aop, Bop, C);
}

}  // namespace spx
