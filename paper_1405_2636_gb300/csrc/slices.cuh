// slices.cuh -- FP64 products on the FP16 tensor cores without rounding
// errors.  (Error-free splitting of a matrix product: Ozaki, Ogita, Oishi,
// Rump, "Error-free transformations of matrix multiplication by using fast
// routines of matrix multiplication and its applications", 2012.)
//
// This part's FP64 unit retires 1.7 multiply-adds a cycle and SM, its FP16
// tensor path 4,096.  So a row of K <= 64 doubles with largest magnitude
// below 2^e is written as 57-bit fixed-point numbers f = x 2^(57 - e),
// rounded to nearest, each cut into seven signed digits
//   f = sum_s d_s 256^(6 - s),  |d_0| <= 512, -128 <= d_s <= 127 (s > 0),
// which FP16 holds exactly.  A product of digits is an integer of at most 18
// bits, and the sum over K of all digit pairs (s, t) with s + t = g stays
// within 2^24 in magnitude (g = 0: 64 x 2^18; g = 6: 64 (2 x 2^16 + 5 x 2^14)),
// so the FP32 accumulators of tcgen05.mma hold the group sums exactly.  Groups
// 0 .. 6 (28 of the 49 digit pairs) are kept; sum_g v_g 256^(6 - g) is put
// together in integers and rounded once to a double.
//
// Error of one dot product: digits below 2^-57 of a row's bound are rounded
// off (entries within a factor 16 of the row's largest lose nothing), and the
// omitted groups come to about 2^-56 of the product of the rows' largest
// entries (digits vary independently), an eighth of FP64's unit roundoff.  So
// the error is relative to the product of the two rows' largest entries, not to
// the sum of the products' magnitudes as that of multiply-adds: where entries
// grow along one operand's rows and fall along the other's (the scales of the
// unknowns that the sum runs over), the caller scales the columns by powers of
// two, up in one and down in the other, before the cut.
// Measured forward errors of solutions against those with FP64 multiply-adds,
// root mean square over 10 to 24 systems of a kind: 0.84 (20^3 diffusion),
// 0.87 (32^3), 1.00 (LDL^T), 1.00 (graph order, 128-wide panels; an eighth
// group, 34 pairs instead of 28, changed nothing).
//
// Integers only from the bits of the input to the bits of the result: on
// this part a conversion to or from a double occupies the FP64 unit.
#pragma once

#include "tc_common.cuh"

#include <cuda_fp16.h>

namespace spx {
namespace sl {

constexpr int kSlices = kSliceCount;
constexpr int kGroups = 7;                // digit pairs (s, t) by s + t, those up to 6
constexpr int kK = 64;                    // columns of one digit block (128 bytes of FP16)
constexpr int32_t kExpBad = 1 << 20;      // row exponent of a row holding an infinity or a NaN

constexpr int kFieldBad = 1 << 16;        // the exponent field of an infinity or a NaN, past every scaled one
constexpr int kFieldZero = -(1 << 14);    // ... of a row of zeros, below every scaled one

// Biased exponent field of |x| (subnormals and zero: 1, so that x = m 2^(field - 1075)).
__device__ __forceinline__ int exp_field(double x)
{
    const int e = (__double2hiint(x) >> 20) & 0x7FF;
    return e == 0x7FF ? kFieldBad : max(e, 1);
}

// The same for x 2^scale; a zero does not count.
__device__ __forceinline__ int exp_field(double x, int scale)
{
    const int hi = __double2hiint(x) & 0x7FFFFFFF;
    if ((hi | __double2loint(x)) == 0) return kFieldZero;
    const int e = hi >> 20;
    return e == 0x7FF ? kFieldBad : (e > 0 ? e : 1) + scale;
}

// Row exponent e (every |x| of the row below 2^e) from the row's largest field.
__device__ __forceinline__ int32_t row_exp(int field) { return field >= kFieldBad ? kExpBad : field - 1022; }

// Fixed-point number of x 2^scale in a row whose largest (scaled) exponent
// field is `field`, with 128 added to each of its six low digits: byte i
// (i < 6) holds digit 6 - i plus 128, the bits above 48 digit 0 (arithmetic).
__device__ __forceinline__ long long fixed_biased(double x, int field, int scale = 0)
{
    const long long b = __double_as_longlong(x);
    const int ef = (int)((b >> 52) & 0x7FF);
    long long m = b & 0xFFFFFFFFFFFFFLL;
    if (ef > 0) m |= 0x10000000000000LL;
    // m 2^(ef + scale - field + 4), at most 2^57: shifted with one bit to spare,
    // then rounded to nearest.  A tie (every other entry that loses one bit) goes
    // up or down by a bit from the middle of the mantissa: one way for all would
    // make the products of L's equal-signed entries too large together.
    const int n = min(max(field - scale - (ef > 0 ? ef : 1), 0), 63);
    const long long M = (m << 5) - ((b >> 40) & 1);
    const long long f = (long long)(((unsigned long long)M >> n) + 1) >> 1;
    const long long sign = b >> 63;
    return (f ^ sign) - sign + 0x808080808080LL;
}

// The seven digits of two numbers (fixed_biased), as half2 words.
__device__ __forceinline__ void digits2(long long f0, long long f1, uint32_t (&w)[kSlices])
{
    const uint32_t l0 = (uint32_t)f0, h0 = (uint32_t)(f0 >> 32), l1 = (uint32_t)f1, h1 = (uint32_t)(f1 >> 32);
    const __half2 c128 = __half2half2(__ushort_as_half(0x6480));   // 1024 + 128
    const __half2 c512 = __half2half2(__ushort_as_half(0x6600));   // 1024 + 512
    // 0x6400 + b is the half 1024 + b for 0 <= b <= 1024
    auto conv = [](uint32_t v, __half2 c) {
        __half2 h = *reinterpret_cast<__half2 *>(&v);
        h = __hsub2(h, c);
        return *reinterpret_cast<uint32_t *>(&h);
    };
    const uint32_t t0 = (uint32_t)(((int)h0 >> 16) + 512), t1 = (uint32_t)(((int)h1 >> 16) + 512);
    w[0] = conv((t0 | (t1 << 16)) + 0x64006400u, c512);
    w[1] = conv((__byte_perm(h0, h1, 0x0501) & 0x00FF00FFu) | 0x64006400u, c128);
    w[2] = conv((__byte_perm(h0, h1, 0x0400) & 0x00FF00FFu) | 0x64006400u, c128);
    w[3] = conv((__byte_perm(l0, l1, 0x0703) & 0x00FF00FFu) | 0x64006400u, c128);
    w[4] = conv((__byte_perm(l0, l1, 0x0602) & 0x00FF00FFu) | 0x64006400u, c128);
    w[5] = conv((__byte_perm(l0, l1, 0x0501) & 0x00FF00FFu) | 0x64006400u, c128);
    w[6] = conv((__byte_perm(l0, l1, 0x0400) & 0x00FF00FFu) | 0x64006400u, c128);
}

// Running sum of the groups from g = 6 down to g = 0: T = hi 2^32 + lo.
struct Sum {
    long long hi;
    uint32_t lo;
};

// Group g's value v joins: groups 6 .. 3 build the low part in hi, which is
// cut into (hi, lo) after group 3; groups 2 .. 0 add to hi.
template <int G>
__device__ __forceinline__ void add_group(Sum &s, float v)
{
    const int q = __float2int_rn(v);
    if constexpr (G == 6) s.hi = q;
    else s.hi += (long long)q * (1 << (8 * ((6 - G) & 3)));
    if constexpr (G == 3) {
        s.lo = (uint32_t)s.hi;
        s.hi >>= 32;
    }
    // keeps the compiler from holding every group's values back to the end
    asm volatile("" : "+l"(s.hi));
}

// (hi 2^32 + lo) 2^(e - 66) rounded to a double, e the sum of the two rows'
// exponents; ties round up in magnitude.  neg: the negated value.
__device__ __forceinline__ double finish(Sum s, int e, bool neg)
{
    const bool minus = s.hi < 0;
    long long hi = s.hi;
    uint32_t lo = s.lo;
    if (minus) {
        hi = ~hi + (lo == 0 ? 1 : 0);
        lo = 0u - lo;
    }
    uint32_t a = (uint32_t)(hi >> 32), b = (uint32_t)hi, c = lo;
    int p = 95 + e - 66 + 1023;
    if (a == 0) {
        a = b;
        b = c;
        c = 0;
        p -= 32;
        if (a == 0) {
            a = b;
            b = 0;
            p -= 32;
            if (a == 0) return e >= kExpBad / 2 ? __longlong_as_double(0x7FF8000000000000LL) : 0.0;
        }
    }
    const int n = __clz(a);
    p -= n;
    const uint32_t mh = __funnelshift_l(b, a, n), ml = __funnelshift_l(c, b, n);
    const unsigned long long m = ((unsigned long long)mh << 32) | ml;
    // m >> 11 holds the leading bit, which adds one to the exponent field
    unsigned long long bits = ((unsigned long long)(unsigned)(p - 1) << 52) + (m >> 11) + ((m >> 10) & 1u);
    if ((unsigned)(p - 1) >= 2046u) {   // outside the normal range
        if (e >= kExpBad / 2) bits = 0x7FF8000000000000ULL;
        else if (p > 0) bits = 0x7FF0000000000000ULL;
        else bits = p < -51 ? 0 : (m >> (12 - p)) + ((m >> (11 - p)) & 1u);
    }
    return __longlong_as_double((long long)(bits | ((unsigned long long)(minus != neg) << 63)));
}

// FP16 operands, FP32 accumulator, both K-major, M = 128, N = 16 .. 64.
__device__ __forceinline__ uint32_t idesc_f16(int n)
{
    return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(tc::kM >> 4) << 24);
}

// 16 or 8 columns of this warp's 32 TMEM lanes.  The values pass through the
// wait, so that nothing uses them before it.
__device__ __forceinline__ void tmem_read16(uint32_t t, uint32_t (&v)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 "
                 "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                   "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]),
                   "=r"(v[15])
                 : "r"(t));
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                   "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]),
                   "+r"(v[15])
                 :
                 : "memory");
}

__device__ __forceinline__ void tmem_read8(uint32_t t, uint32_t (&v)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(t));
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7])
                 :
                 : "memory");
}

}  // namespace sl
}  // namespace spx
