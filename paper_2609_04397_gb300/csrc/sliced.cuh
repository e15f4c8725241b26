// Sliced FP64: block products of FP64 operators on the FP16 tensor cores.
//
// GB300's FP64 pipe does 2 multiply-adds a clock and SM (1.26 TFLOP/s on the
// chip), its tensor cores 950 with mma.sync (m16n8k16, f16 operands, FP32
// accumulators; measured). An FP64 dot product is therefore cut into exact
// small-integer products (the splitting of Ozaki, Ogita, Oishi and Rump,
// "Error-free transformations of matrix multiplication by using fast routines
// of matrix multiplication", 2012):
//
//  * every row of the stored values and every column of X (per structure of a
//    batched operator) gets one power-of-two scale from its largest magnitude,
//    and every element becomes a 56-bit fixed-point integer below it;
//  * that integer is written in base 256 with kSliceDigits = 7 balanced digits
//    -128 .. 127: one byte each, which f16 holds exactly;
//  * products of digits i and j (digit 0 the most significant) are integers up
//    to 2^14 and belong to level i + j, of weight 256^-(i + j). Sums over
//    kSliceFlush steps stay below 2^24 in the levels 0 to 4 whatever the digits,
//    so the FP32 accumulators hold them exactly, in any order (kSliceFlush on the
//    levels below); longer rows carry each level's upper part into the next one up
//    every kSliceFlush steps;
//  * the levels 0 .. 7 (34 of the 49 digit pairs) are added as integers and rounded
//    to FP64 once. The pairs left out are below 2^-61 of (row scale) x (column scale)
//    a term, the rounding of an element to 56 bits below 2^-56.
//
// An FP64 multiply-add chain instead rounds at every step; on panels of entries of
// like size the sliced product is the nearer one to the exact result. The scales
// make its error an absolute one, though: an output whose terms are all far below
// the row's and the column's largest would lose digits. So every output also
// carries an estimate of sum |h x| (the products of the leading digits'
// magnitudes, one more MMA in 35), and an output whose estimate is too low
// (kSliceGuard, slice_guard) is computed with FP64 multiply-adds by the same
// warp, alone or with its pass of 16 columns. What remains is within K 2^-53 of
// sum |h x|, the bound of a K-term multiply-add chain, and the one rounding. Rows
// and columns with Inf, NaN or extreme exponents and panels with mostly tiny
// entries (one-hot or localised columns) take the multiply-adds as well, and lose
// the two passes over X (2 to 6 % at k = 8 to 32 on 50k and 20k atoms).
//
// (The FP8 form of the same scheme, 12 base-32 digits in e4m3, needs no carries
// and is as exact, but mma.sync runs e4m3 operands converted on the f16
// pipe here: 79 products at the f16 rate, 5.5 against 1.4 ms at k = 32 on the
// 50k-atom operator. INT8 mma.sync does 250 multiply-adds a clock and SM.)
#pragma once

#include "internal.cuh"

namespace vbcsr {

// Least sum of |leading digit| products of an output. In units of the last place (2^-55
// of a scale) every element is rounded by up to 1/2, which costs an output up to
// (sum |h| + sum |x|) / 2 <= 2^54 K (1 + sum |h x| / 2^110); the levels left out and the
// FP32 sums past 2^24 in the levels 5 to 7 add less than 2 % of 2^54 K. Leading digits d
// and e stand for magnitudes of at least (d - 0.502) 2^48 and (e - 0.502) 2^48. The least
// sum |h x| for a given estimate and room for K roundings is that of products 1 x 128:
// 0.496 of the estimate times 2^96, and 2^54 K <= K 2^-53 (0.496 G 2^96) from G = 4129 on,
// whatever K is. (At 512 products of K = 764 were off by up to 2300 2^-53 of sum |h x|.)
constexpr float kSliceGuard = 4352.f;
// The same with the sum of the leading digits' magnitudes of the row and of the column over
// the K terms at hand: sum |h| + sum |x| <= (digits + 1.004 K) 2^48, the levels left out
// are below 2^48.4 K, sum |h x| is at least 0.248 of the estimate times 2^96. Panels whose
// column maxima lie far above most entries stay resolved by it (Student's t with 3 degrees of
// freedom, 20k disordered atoms, k = 8: 325 us, 886 by kSliceGuard alone, 546 by multiply-adds).
__device__ __forceinline__ float slice_guard(int digits, int K) {
    return fminf(kSliceGuard, 66.f * ((float)digits / (float)K + 3.7f));
}
// A column with more than 3/8 of its elements below 2^-kSliceTiny of its largest, where the
// leading digit is zero, is not tried: many outputs would not be resolved, and a pass that
// fails costs a fifth of the multiply-adds at k = 8 (columns that fall by 10^3 from end to
// end, 45 % below: tried, 1819 / 667 us at k = 8 on 50k zinc-blende / 20k disordered atoms,
// not tried 2380 / 577). Student's t with 3 degrees of freedom (a fifth below at 10^5 rows) is
// tried and runs 1.6 to 2.3 times as fast as multiply-adds on 20k atoms.
constexpr int kSliceTiny = 8;
constexpr int kSliceLevels = 8;
// 16-column steps between carries: 5 products x 192 columns x 2^14 < 2^24 in level 4. The
// levels 5, 6 and 7 have 6, 7 and 6 products: sums of nearly extreme digits throughout pass
// 2^24 there and lose a unit or two of 2^-54, 2^-62, 2^-70 of the scales' product a step; in
// level 5 (and 6) that takes leading digits near 128 of both (of one) operands, whose sum
// |h x| (sum |h| + sum |x|, see kSliceGuard) is then far above the loss.
constexpr int kSliceFlush = 12;
constexpr int kSliceTile = kSliceDigits * 16;   // bytes of one row of a 16-column value tile
// biased FP64 exponents a row or column maximum may have (the products of two
// stay clear of overflow and of subnormal results)
constexpr int kSliceExpMin = 640, kSliceExpMax = 1400;

// Exponent of a scale from the high word of the largest magnitude, such that
// |v| / 2^(E - 1077) is below 0.991 * 2^55 (the balanced digits reach
// 0.996 * 2^55): a mantissa of 1.98 or more takes the next exponent.
__device__ __forceinline__ int slice_exp(uint32_t hi) { return (int)((hi + 0x51ECu) >> 20); }
// 0 when the maximum is zero; false: this row or column is not sliced
__device__ __forceinline__ bool slice_exp_ok(uint32_t hi) {
    const int e = slice_exp(hi);
    return hi == 0 || (hi < 0x7fe00000u && e >= kSliceExpMin && e <= kSliceExpMax);
}
// high word of |x| as the maximum sees it (1 for a magnitude below its range)
__device__ __forceinline__ uint32_t slice_mag(double x) {
    const uint64_t b = (uint64_t)__double_as_longlong(x) & 0x7fffffffffffffffull;
    const uint32_t hi = (uint32_t)(b >> 32);
    return hi ? hi : ((uint32_t)b ? 1u : 0u);
}

// x at scale exponent E as a fixed-point integer of D = 7 or 8 base-256 digits
// plus 128 in every byte: byte b holds digit (D - 1 - b) + 128. Integer
// arithmetic throughout (the FP64 pipe is the scarce unit).
template <int D = kSliceDigits>
__device__ __forceinline__ uint64_t slice_bytes(double x, int E) {
    constexpr uint64_t kBias = D == 8 ? 0x8080808080808080ull : 0x80808080808080ull;
    constexpr int kTop = D == 8 ? 10 : 2;          // shift of a 53-bit mantissa at the scale's own exponent
    const uint64_t b = (uint64_t)__double_as_longlong(x);
    const int eb = (int)((b >> 52) & 0x7ff);
    uint64_t m = b & 0xfffffffffffffull;
    if (eb) m |= 1ull << 52;
    const int sh = kTop - (E - (eb ? eb : 1));     // value = m * 2^sh units, |.| < 2^(8 D - 1)
    uint64_t v;
    if (sh >= 0) v = m << sh;
    else if (sh > -54) v = (m + (1ull << (-sh - 1))) >> -sh;
    else v = 0;
    return (b >> 63) ? kBias - v : kBias + v;
}

// two biased bytes as the f16 pair of their digits: 0x6400 | byte is 1024 + byte
__device__ __forceinline__ uint32_t slice_half2(uint32_t bytes, uint32_t sel) {
    uint32_t r = __byte_perm(bytes, 0x64646464u, sel);
    asm("sub.f16x2 %0, %0, %1;" : "+r"(r) : "r"(0x64806480u));   // - 1152
    return r;
}

// The digits of four elements (K order) as f16 pairs: f[i][0] digit i of (v0, v1), f[i][1] of (v2, v3)
template <int D>
__device__ __forceinline__ void slice_pairs(const uint2 (&v)[4], uint32_t (&f)[D][2]) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint2 a = v[2 * h], b = v[2 * h + 1];
        const uint32_t p[4] = {__byte_perm(a.x, b.x, 0x5140), __byte_perm(a.x, b.x, 0x7362),
                               __byte_perm(a.y, b.y, 0x5140), __byte_perm(a.y, b.y, 0x7362)};
#pragma unroll
        for (int i = 0; i < D; ++i) {
            const int byte = D - 1 - i;
            f[i][h] = slice_half2(p[byte >> 1], byte & 1 ? 0x4342 : 0x4140);
        }
    }
}

// sum over levels of c[L] * 256^(7 - L), rounded to FP64 once (to nearest, ties
// to even), times 2^e2, in integer arithmetic: with the sum's two halves
// converted and joined on the FP64 pipe (4 of its operations an output, 64
// clocks of an SM for a warp), the pattern-sampled kernel spent 80 % of its time there.
// BOUND22: every |c| is below 2^22 (at most 16 terms a pair); then 62 leading bits
// of the sum fit one 64-bit integer whatever its size, and one conversion (16
// clocks of the otherwise idle FP64 pipe against some 30 instructions) rounds them;
// what is cut off is below 2^-58 of the scales' product.
template <bool BOUND22 = false>
__device__ __forceinline__ double slice_value(const float (&c)[kSliceLevels], int e2) {
    long long p[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (BOUND22) {
            // c + 1.5 * 2^23 holds the integer in its low bits over the constant below (full
            // rate; a float-to-integer conversion runs at an eighth of it); two levels make
            // one 32-bit integer
            constexpr uint32_t kM = 0x4b400000u;
            uint32_t b[4];
#pragma unroll
            for (int L = 0; L < 4; ++L) b[L] = __float_as_uint(__fadd_rn(c[4 * h + L], 12582912.f));
            const int q0 = (int)(b[0] * 256u + (b[1] - kM * 257u)), q1 = (int)(b[2] * 256u + (b[3] - kM * 257u));
            p[h] = (long long)q0 * 65536 + q1;
        } else {
            p[h] = __float2int_rn(c[4 * h]);
#pragma unroll
            for (int L = 1; L < 4; ++L) p[h] = p[h] * 256 + __float2int_rn(c[4 * h + L]);
        }
    }
    if (BOUND22) {
        const long long v = (p[0] << 20) + (p[1] >> 12);   // |p[0]| < 2^42.1
        const uint64_t b = (uint64_t)__double_as_longlong((double)v);
        return v == 0 ? 0.0 : __longlong_as_double((long long)(b + ((uint64_t)(int64_t)(e2 + 12) << 52)));
    }
    // T = s * 2^32 + lo, then its magnitude m * 2^32 + mlo
    const long long s = p[0] + (p[1] >> 32);
    const uint32_t lo = (uint32_t)p[1];
    const bool neg = s < 0;
    uint64_t m = neg ? ~(uint64_t)s + (lo == 0) : (uint64_t)s;
    uint32_t mlo = neg ? 0u - lo : lo;
    int e = 1023 + 63 + 32;
    if (m == 0) {
        m = mlo;
        mlo = 0;
        e -= 32;
    }
    if (m == 0) return 0.0;
    const int sh = __clzll((long long)m);
    e -= sh;
    // top: the leading 64 bits, the rest only counts as a sticky bit
    uint64_t top = m << sh;
    uint32_t rest;
    if (sh < 32) {
        top |= (uint64_t)mlo >> (32 - sh);
        rest = mlo << sh;
    } else {
        top |= (uint64_t)mlo << (sh - 32);
        rest = 0;
    }
    const uint32_t low11 = (uint32_t)top & 0x7ffu;
    const uint64_t mant = top >> 11;
    const uint32_t up = (low11 & 0x400u) && ((low11 & 0x3ffu) | rest | ((uint32_t)mant & 1u));
    // the leading bit of mant adds one to the exponent field; |e2| keeps the result
    // normal (kSliceExpMin .. kSliceExpMax)
    const uint64_t bits = ((uint64_t)(e + e2 - 1) << 52) + mant + up;
    return __longlong_as_double((long long)(bits | (neg ? 1ull << 63 : 0ull)));
}

// Sum over digits of one operand in registers (t[e][d], integers below 2^24) and of
// the other across the four lanes of a group, two a lane (e): sum over d and j =
// 2 t4 + e of t * 256^(12 - d - j), times 2^e2 and in units of 2^40 (the units of
// slice_value), on every lane of the group. Two conversions, a fused multiply-add and
// two additions of the FP64 pipe, which little else uses here; the largest part
// carries the rounding.
__device__ __forceinline__ double slice_value_of_lanes(const float (&t)[2][8], int t4, int e2) {
    long long hi = 0, lo = 0;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        long long p = __float2int_rn(t[e][0]), r = __float2int_rn(t[e][4]);
#pragma unroll
        for (int d = 1; d < 4; ++d) p = p * 256 + __float2int_rn(t[e][d]);
#pragma unroll
        for (int d = 5; d < 7; ++d) r = r * 256 + __float2int_rn(t[e][d]);
        hi = hi * 256 + p;   // below 2^57
        lo = lo * 256 + r;   // below 2^49
    }
    double v = fma((double)hi, 16777216.0, (double)lo);
    v *= t4 == 0 ? 1.0 : t4 == 1 ? 0x1p-16 : t4 == 2 ? 0x1p-32 : 0x1p-48;
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    const uint64_t bits = (uint64_t)__double_as_longlong(v);
    return (bits << 1) == 0 ? 0.0 : __longlong_as_double((long long)(bits + ((uint64_t)(int64_t)e2 << 52)));
}

// Carry the upper part of every level into the one above (exact: integers below 2^24)
__device__ __forceinline__ void slice_carry(float (&acc)[kSliceLevels][4]) {
#pragma unroll
    for (int L = kSliceLevels - 1; L > 0; --L)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            // adding 1.5 * 2^23 rounds to an integer
            const float c = __fadd_rn(__fmaf_rn(acc[L][j], 0.00390625f, 12582912.f), -12582912.f);
            acc[L][j] = __fmaf_rn(c, -256.f, acc[L][j]);
            acc[L - 1][j] += c;
        }
}

__device__ __forceinline__ void mma_f16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

}  // namespace vbcsr
