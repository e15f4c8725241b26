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
//    kSliceFlush columns stay below 2^24 in the levels that matter, so the FP32
//    accumulators hold them exactly, in any order; longer rows carry each
//    level's upper part into the next one up every kSliceFlush columns;
//  * the levels 0 .. 7 (34 digit pairs) are added as integers and rounded to
//    FP64 once. What is dropped is about 2^-58 of (row scale) x (column scale).
//
// An FP64 multiply-add chain instead rounds at every step; on the operators
// and panels of this repository the sliced product is the nearer one to the
// exact result. The scales make its error an absolute one, though: an output
// whose terms are all far below the row's and the column's largest would lose
// digits. So every output also carries an estimate of sum |h x| (the products
// of the leading digits' magnitudes, one more MMA in 35), and the remaining
// columns of an item with an output whose estimate is below kSliceGuard are
// computed with FP64 multiply-adds by the same warp: what remains has an error
// of at most a few dozen 2^-53 of sum |h x|, inside the K 2^-53 of a K-term
// multiply-add chain. Rows and columns with Inf, NaN or extreme exponents and
// panels with mostly tiny entries take the multiply-adds as well.
//
// (The FP8 form of the same scheme, 12 base-32 digits in e4m3, needs no carries
// and is as exact, but mma.sync runs e4m3 operands converted on the f16
// pipe here: 79 products at the f16 rate, 5.5 against 1.1 ms at k = 32 on the
// 50k-atom operator. INT8 mma.sync does 250 multiply-adds a clock and SM.)
#pragma once

#include "internal.cuh"

namespace vbcsr {

constexpr float kSliceGuard = 512.f;   // least sum of |leading digit| products of an output
constexpr int kSliceLevels = 8;
constexpr int kSliceFlush = 12;        // 16-column steps between carries: 5 products x 192 columns x 2^14 < 2^24
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

// x at scale exponent E as a fixed-point integer plus 128 in every byte of the
// low 7: byte b holds digit (6 - b) + 128. Integer arithmetic throughout (the
// FP64 pipe is the scarce unit).
constexpr uint64_t kSliceBias = 0x80808080808080ull;
__device__ __forceinline__ uint64_t slice_bytes(double x, int E) {
    const uint64_t b = (uint64_t)__double_as_longlong(x);
    const int eb = (int)((b >> 52) & 0x7ff);
    uint64_t m = b & 0xfffffffffffffull;
    if (eb) m |= 1ull << 52;
    const int sh = 2 - (E - (eb ? eb : 1));        // value = m * 2^sh units, |.| < 2^55
    uint64_t v;
    if (sh >= 0) v = m << sh;
    else if (sh > -54) v = (m + (1ull << (-sh - 1))) >> -sh;
    else v = 0;
    return (b >> 63) ? kSliceBias - v : kSliceBias + v;
}

// two biased bytes as the f16 pair of their digits: 0x6400 | byte is 1024 + byte
__device__ __forceinline__ uint32_t slice_half2(uint32_t bytes, uint32_t sel) {
    uint32_t r = __byte_perm(bytes, 0x64646464u, sel);
    asm("sub.f16x2 %0, %0, %1;" : "+r"(r) : "r"(0x64806480u));   // - 1152
    return r;
}

// sum over levels of c[L] * 256^(7 - L) (each an integer below 2^24 in FP32),
// rounded to FP64 once, times 2^e2
__device__ __forceinline__ double slice_value(const float (&c)[kSliceLevels], int e2) {
    int i[kSliceLevels];
#pragma unroll
    for (int L = 0; L < kSliceLevels; ++L) i[L] = __float2int_rn(c[L]);
    long long p[2];
#pragma unroll
    for (int h = 0; h < 2; ++h)
        p[h] = ((long long)i[4 * h] << 24) + ((long long)i[4 * h + 1] << 16) +
               (((long long)i[4 * h + 2] << 8) + i[4 * h + 3]);
    // both parts are below 2^53: the fused multiply-add rounds their sum once
    const double r = fma((double)p[0], 4294967296.0, (double)p[1]);
    const uint64_t b = (uint64_t)__double_as_longlong(r);
    // |e2| keeps the result normal (kSliceExpMin .. kSliceExpMax): scale by the exponent field
    return r == 0.0 ? 0.0 : __longlong_as_double((long long)(b + ((uint64_t)(int64_t)e2 << 52)));
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
