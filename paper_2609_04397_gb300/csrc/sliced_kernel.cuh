// The product kernel of the sliced FP64 operators (sliced.cuh): spmm_sliced.cu
// instantiates it for real operators, spmm_sliced_c128.cu for complex ones.
#pragma once

#include "fma_kernel.cuh"
#include "sliced.cuh"

namespace vbcsr {

namespace {

constexpr int kSliceList = (kSliceKMax + 16) * sizeof(int32_t);   // X rows of an item and of one step more
constexpr uint32_t kSliceWary = 2;  // such passes after which the first attempt of a wide kernel is CAREFUL
constexpr int kSliceState = 16;   // bytes that a warp keeps from item to item
// unresolved outputs of a pass computed one by one: at most a quarter of the pass (they take
// about twice the FP64 pipe's time of an item's common multiply-adds, and far more latency)
constexpr int kSliceSingles = 32;
constexpr int kSliceStages = 4;   // value tiles in flight per warp (16 columns, up to 1792 bytes each)

// What a warp keeps from item to item, behind its list: [0] the structure of the last item,
// [1] its passes that run multiply-adds: bit p for the 16 columns of pass p, bit 31 for pass
// 31 and all after it; [2] passes with outputs below kSliceGuard since a CAREFUL one had none
__device__ __forceinline__ volatile uint32_t *slice_state(unsigned char *ring) {
    return reinterpret_cast<volatile uint32_t *>(ring + kSliceStages * 16 * kSliceTile + kSliceList);
}

// the operator's own arithmetic, for what is not sliced
template <int B, bool TRANS, typename T, typename TA>
__device__ __noinline__ void fma_item_fallback(const ProdArgs &a, const WorkItem &w, int kc, int32_t *s_x,
                                               int64_t *s_a, int lane, double &dot) {
    process_item<B, TRANS, T, TA, T, T>(a, w, kc, s_x, s_a, nullptr, lane, dot);
}

// Columns [n0, n1) of item w by FP64 multiply-adds (complex T: two real columns of the
// sliced panels make one)
template <bool TRANS, typename T, typename TA>
__device__ __noinline__ void fma_columns(const ProdArgs &a, int64_t n0, int64_t n1, const WorkItem &w, unsigned char *smem, int lane,
                                         double &dot) {
    ProdArgs b = a;
    constexpr int cw = sizeof(T) / sizeof(double);
    b.k = (n1 - n0) / cw;
    b.ldx = a.ldx / cw;
    b.ldy = a.ldy / cw;
    b.ldz = a.ldz / cw;
    b.ldr = a.ldr / cw;
    b.X = static_cast<const double *>(a.X) + n0;
    b.Y = static_cast<double *>(a.Y) + n0;
    if (a.gamma_nz) b.Z = static_cast<const double *>(a.Z) + n0;
    if (a.item_partials) b.R = static_cast<const double *>(a.R) + n0;
    int kc = 1;
    while (kc < b.k && kc < 32) kc <<= 1;
    int64_t *s_a = reinterpret_cast<int64_t *>(smem);
    int32_t *s_x = reinterpret_cast<int32_t *>(smem + kKMax * sizeof(int64_t));
#define VBCSR_SLICE_CASE(NB) \
    case NB: fma_item_fallback<NB, TRANS, T, TA>(b, w, kc, s_x, s_a, lane, dot); break;
    switch (w.B) {
        VBCSR_SLICE_CASE(1) VBCSR_SLICE_CASE(2) VBCSR_SLICE_CASE(3) VBCSR_SLICE_CASE(4)
        VBCSR_SLICE_CASE(5) VBCSR_SLICE_CASE(6) VBCSR_SLICE_CASE(7) VBCSR_SLICE_CASE(8)
        VBCSR_SLICE_CASE(9) VBCSR_SLICE_CASE(10) VBCSR_SLICE_CASE(11) VBCSR_SLICE_CASE(12)
        VBCSR_SLICE_CASE(13) VBCSR_SLICE_CASE(14) VBCSR_SLICE_CASE(15) VBCSR_SLICE_CASE(16)
        default: break;
    }
#undef VBCSR_SLICE_CASE
}

// Output (row r of the item, real column c) by FP64 multiply-adds: the whole warp, four
// lanes a stored block, so a chain has a few terms a block and at most K / 4. Items that
// need it are small and come last, where their latency shows. Complex T: the real column
// is one component of a complex one.
template <bool TRANS, typename T>
__device__ __noinline__ double slice_one_output(const ProdArgs &a, const WorkItem &w, int r, int64_t c, int lane) {
    constexpr int cw = sizeof(T) / sizeof(double);
    const double *V = static_cast<const double *>(a.values), *X = static_cast<const double *>(a.X) + c;
    double acc = 0.0;
    for (int e = lane >> 2; e < w.nlist; e += 8) {
        const int64_t l = w.lbegin + e;
        const double *v = V + cw * (TRANS ? a.tl.pbase[l] + w.Kp + r : w.vbase + (int64_t)r * w.Kp + a.fl.pcol[l]);
        const int64_t step = TRANS ? cw * (int64_t)a.tl.kp[l] : cw;
        const double *x = X + (int64_t)(TRANS ? a.tl.xrow[l] : a.fl.xrow[l]) * a.ldx;
        const int n = TRANS ? a.tl.bi[l] : a.fl.w[l];
#pragma unroll 4
        for (int t = lane & 3; t < n; t += 4) {
            const double *vt = v + t * step, *xt = x + t * a.ldx;
            acc = fma(vt[0], xt[0], acc);
            // re: - im(v) im(x); im: + im(v) re(x); the adjoint conjugates v
            if (cw == 2) acc = fma(((c & 1) != 0) != TRANS ? vt[1] : -vt[1], xt[c & 1 ? -1 : 1], acc);
        }
    }
    for (int m = 16; m > 0; m >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, m);
    return acc;
}

// Sums of the magnitudes of the leading digits: sum[r] of row r of the item's value tiles,
// sum[16 + c] of column n0 + c of the X rows in s_x (sum in shared memory)
__device__ __noinline__ void slice_digit_sums(const unsigned char *tiles, int B, int K, const uint64_t *xdig, int ldp,
                                              int64_t n0, const int32_t *s_x, int *sum, int lane) {
    const int i = lane & 15, h = lane >> 4;
    unsigned rows = 0, cols = 0;
    if (i < B)
        for (int t = h; 16 * t < K; t += 2) {
            const uint4 v = __ldg(reinterpret_cast<const uint4 *>(tiles + (int64_t)t * B * kSliceTile + 16 * i));
            const uint32_t zero = 0x80808080u;
            rows += __vsadu4(v.x, zero) + __vsadu4(v.y, zero) + __vsadu4(v.z, zero) + __vsadu4(v.w, zero);
        }
    if (n0 + i < ldp)
#pragma unroll 8
        for (int t = h; t < K; t += 2)
            cols += abs((int)(__ldg(xdig + (int64_t)s_x[t] * ldp + n0 + i) >> 48 & 0xff) - 128);
    rows += __shfl_xor_sync(0xffffffffu, rows, 16);
    cols += __shfl_xor_sync(0xffffffffu, cols, 16);
    __syncwarp();
    sum[lane] = (int)(h ? cols : rows);
    __syncwarp();
}

// Whether slice_guard resolves every output of a pass of 16 columns (or the last ones) that has
// some below kSliceGuard, from the leading digits alone: lane % 16 a column, the two halves
// 8 rows each. Complex T: an output whose every term has a part that is zero throughout is an
// exact zero. A small loop: the code of the CAREFUL pass, fetched for one item near the end
// of a launch, took 119,000 clocks (20k zinc-blende atoms, k = 16: 350 us with it for every such
// pass, 334 with this first, 316 with none).
template <typename T>
__device__ __noinline__ bool slice_recheck(const SliceArgs &q, const unsigned char *tiles, int B, int K, int64_t yrow,
                                           int64_t k, int64_t n0, const uint32_t *cmax, const int32_t *s_x, int lane) {
    const int64_t c = n0 + (lane & 15);
    const int r0 = lane >> 4 << 3;
    const uint32_t zero = 0x80808080u;
    unsigned low[8], rows[8], cols = 0;
#pragma unroll
    for (int r = 0; r < 8; ++r) low[r] = rows[r] = 0;
    for (int t = 0; t < K; t += 16, tiles += B * kSliceTile) {
        uint32_t x[4] = {zero, zero, zero, zero};   // leading digits of four X rows a word
        if (c < q.ldp)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                x[i] = 0;
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    x[i] |= (uint32_t)(__ldg(q.xdig + (int64_t)s_x[t + 4 * i + j] * q.ldp + c) >> 48 & 0xff) << (8 * j);
            }
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = __vabsdiffu4(x[i], zero), cols += __dp4a(x[i], 0x01010101u, 0u);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            if (r0 + r >= B) break;
            const uint4 v = __ldg(reinterpret_cast<const uint4 *>(tiles + 16 * (r0 + r)));
            const uint32_t h[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t d = __vabsdiffu4(h[i], zero);
                rows[r] = __dp4a(d, 0x01010101u, rows[r]);
                low[r] = __dp4a(d, x[i], low[r]);
            }
        }
    }
    bool ok = true;
    const bool live = c < k && cmax[c] != 0;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        if (r0 + r >= B) break;
        const int e = q.rexp[yrow + r0 + r];
        bool out = live && e != 0;
        if (sizeof(T) > sizeof(double) && out) {
            const uint32_t *own = q.cown + (cmax - q.cmax);
            const int parts = q.rparts[yrow + r0 + r];
            out = ((parts & 1) && own[c]) || ((parts & 2) && own[c ^ 1]);
        }
        ok &= e >= 0 && (!out || (float)low[r] >= slice_guard((int)(rows[r] + cols), K));
    }
    return __all_sync(0xffffffffu, ok);
}

// One pass of an item: up to 16 columns (WIDE) or up to 8, steps of 16 virtual
// columns. A step's value tile (7 digits x B rows x 16 bytes, contiguous) comes
// through a ring of shared-memory stages by asynchronous copies; the 16 gathered
// X rows (8 bytes a column) are loaded to registers one step ahead. Lane t4 of a
// fragment owns virtual columns 4 t4 .. 4 t4 + 3 of the step (an order the two
// operands share, so it does not matter to the sums): their bytes are one 32-bit
// word of the value tile and four X loads.
//
// WIDE passes put the 16 columns on the M side of the MMA and the rows, NR
// groups of 8, on the N side, so that items of up to 8 rows take half the MMAs
// (and the outputs of a store are 8 consecutive columns); narrow ones put the
// (up to 16) rows on the M side and the 8 columns on the N side. Narrow passes of
// up to 8 rows (PAIR) fill the M side with two digits of the 8 columns, j and
// j + 1: accumulator L then holds level L of the even digits and level L + 1 of
// the odd ones, and 19 MMAs make the 34 digit pairs (35 with the rows on the M
// side, half of it padding). NINTH: items of 9 rows (an sp3d5 basis), the ninth
// alone with its digits as the N side, one more MMA per digit of X (PAIR: per two)
// instead of another group of 8 rows: 44 MMAs a wide step instead of 72, 25 a
// narrow one instead of 36 (50k zinc-blende atoms, k = 32: 1.43 ms against 1.56).
// Returns false, with nothing written, when an output is below kSliceGuard and not `force`.
// Such a pass is made a second time: with force (wide kernels) when the sums that its error
// really depends on resolve it (slice_recheck), else with CAREFUL (code that would cost the
// first one registers): outputs that slice_guard does not resolve are computed by
// slice_one_output, a few of them (kSliceSingles; rows of few entries have one now and
// then: corners of a cluster, 40 to 120 columns; without this the k = 32 product on 50k
// zinc-blende atoms took 1.52 ms, all 16 columns of such items by multiply-adds). It
// returns false when there are more or a row has no scale.
template <bool TRANS, bool WIDE, int NR, bool NINTH, bool CAREFUL, typename T>
__device__ __forceinline__ bool slice_pass(const ProdArgs &a, const SliceArgs &q, const WorkItem &w,
                                           const unsigned char *vsrc, int K, int64_t n0, const uint32_t *cmax,
                                           unsigned char *ring, const int32_t *s_x, int lane, bool force, double &dot) {
    constexpr int S = kSliceStages, kStage = 16 * kSliceTile;
    const int nsteps = (K + 15) >> 4;
    constexpr int NX = WIDE ? 2 : 1, NA = WIDE ? NR : 1;
    constexpr bool PAIR = !WIDE && NR == 1;
    // the ninth row: digit j of X (PAIR: j and j + 1) times all its digits, 2 t4 + e a lane
    constexpr int NJ = NINTH ? (WIDE ? kSliceDigits : 4) : 1;
    float ninth[NJ][4], nlow[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        nlow[r] = 0.f;
#pragma unroll
        for (int j = 0; j < NJ; ++j) ninth[j][r] = 0.f;
    }
    const int g = lane >> 2, t4 = lane & 3;
    float acc[NA][kSliceLevels][4], low[NA][4];
#pragma unroll
    for (int n = 0; n < NA; ++n)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            low[n][j] = 0.f;
#pragma unroll
            for (int L = 0; L < kSliceLevels; ++L) acc[n][L][j] = 0.f;
        }
    if (nsteps > 0) {
        const uint64_t *xd = q.xdig + n0 + g;
        const int tile = w.B * kSliceTile;
        // this lane's 16-byte chunks of a tile: lane, lane + 32, ... below 7 B (at most 4)
        constexpr int kChunks = (16 * kSliceTile / 16 + 31) / 32;
        bool mine[kChunks];
#pragma unroll
        for (int u = 0; u < kChunks; ++u) mine[u] = 16 * (lane + 32 * u) < tile;
        const unsigned char *src = vsrc + 16 * lane;
        auto issue = [&](int s) {   // steps are issued in order
            const bool in = s < nsteps;
            unsigned char *dst = ring + (s % S) * kStage + 16 * lane;
#pragma unroll
            for (int u = 0; u < kChunks; ++u)
                if (in && mine[u]) cp_async16(dst + 512 * u, src + 512 * u);
            src += tile;
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        uint2 x[NX][4];
        auto load_x = [&](int s) {
            const int4 xi = *reinterpret_cast<const int4 *>(s_x + 16 * s + 4 * t4);
            const int row[4] = {xi.x, xi.y, xi.z, xi.w};
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const uint2 *p = reinterpret_cast<const uint2 *>(xd + (int64_t)row[r] * q.ldp);
#pragma unroll
                for (int n = 0; n < NX; ++n) x[n][r] = __ldg(p + 8 * n);
            }
        };
        load_x(0);
#pragma unroll
        for (int s = 0; s < S - 1; ++s) issue(s);
        const int digit = w.B * 16;   // bytes from a digit's plane of a tile to the next
        int carry = kSliceFlush;
        for (int s = 0; s < nsteps; ++s) {
            asm volatile("cp.async.wait_group %0;" ::"n"(S - 2) : "memory");
            __syncwarp();
            issue(s + S - 1);
            uint32_t b[NX][kSliceDigits][2];
#pragma unroll
            for (int n = 0; n < NX; ++n) slice_pairs<kSliceDigits>(x[n], b[n]);
            load_x(s + 1);   // the list has one step past the last
            const unsigned char *st = ring + (s % S) * kStage + g * 16 + t4 * 4;
            if constexpr (NINTH) {
                constexpr uint32_t kAbs = 0x7fff7fffu;
                // digit g of the ninth row (the eighth digit is zero)
                const uint32_t word = g < kSliceDigits ? *reinterpret_cast<const uint32_t *>(
                                                             ring + (s % S) * kStage + g * digit + 128 + t4 * 4)
                                                       : 0x80808080u;
                const uint32_t v0 = slice_half2(word, 0x4140), v1 = slice_half2(word, 0x4342);
#pragma unroll
                for (int j = 0; j < NJ; ++j) {
                    const int a0 = WIDE ? j : 2 * j, a1 = WIDE || j == 3 ? a0 : a0 + 1;
                    const uint32_t cols[4] = {b[0][a0][0], WIDE ? b[NX - 1][a0][0] : j == 3 ? 0u : b[0][a1][0],
                                              b[0][a0][1], WIDE ? b[NX - 1][a0][1] : j == 3 ? 0u : b[0][a1][1]};
                    mma_f16(ninth[j], cols, v0, v1);
                }
                const uint32_t cols[4] = {b[0][0][0] & kAbs, WIDE ? b[NX - 1][0][0] & kAbs : 0u, b[0][0][1] & kAbs,
                                          WIDE ? b[NX - 1][0][1] & kAbs : 0u};
                mma_f16(nlow, cols, v0 & kAbs, v1 & kAbs);
            }
#pragma unroll
            for (int i = 0; i < kSliceDigits; ++i, st += digit) {
                // digit i of rows g (and g + 8)
                uint32_t v[NR][2];
#pragma unroll
                for (int n = 0; n < NR; ++n) {
                    const uint32_t word = *reinterpret_cast<const uint32_t *>(st + 128 * n);
                    v[n][0] = slice_half2(word, 0x4140);
                    v[n][1] = slice_half2(word, 0x4342);
                }
                const uint32_t rows[4] = {v[0][0], v[NR - 1][0], v[0][1], v[NR - 1][1]};   // M side of a narrow pass
#pragma unroll
                for (int j = 0; j < kSliceDigits && i + j < kSliceLevels; ++j) {
                    if (PAIR) {
                        if (j % 2) continue;
                        const int j1 = j + 1 < kSliceDigits ? j + 1 : j;
                        const bool one = j + 1 < kSliceDigits;   // the eighth digit is zero
                        const uint32_t cols[4] = {b[0][j][0], one ? b[0][j1][0] : 0u, b[0][j][1], one ? b[0][j1][1] : 0u};
                        mma_f16(acc[0][i + j], cols, v[0][0], v[0][1]);
                    } else if (WIDE) {
                        const uint32_t cols[4] = {b[0][j][0], b[NX - 1][j][0], b[0][j][1], b[NX - 1][j][1]};
#pragma unroll
                        for (int n = 0; n < NA; ++n) mma_f16(acc[n][i + j], cols, v[n % NR][0], v[n % NR][1]);
                    } else {
                        mma_f16(acc[0][i + j], rows, b[0][j][0], b[0][j][1]);
                    }
                }
                if (i == 0) {   // magnitudes of the leading digits
                    constexpr uint32_t kAbs = 0x7fff7fffu;
                    if (PAIR) {
                        const uint32_t cols[4] = {b[0][0][0] & kAbs, 0u, b[0][0][1] & kAbs, 0u};
                        mma_f16(low[0], cols, v[0][0] & kAbs, v[0][1] & kAbs);
                    } else if (WIDE) {
                        const uint32_t cols[4] = {b[0][0][0] & kAbs, b[NX - 1][0][0] & kAbs, b[0][0][1] & kAbs,
                                                  b[NX - 1][0][1] & kAbs};
#pragma unroll
                        for (int n = 0; n < NA; ++n) mma_f16(low[n], cols, v[n % NR][0] & kAbs, v[n % NR][1] & kAbs);
                    } else {
                        const uint32_t r[4] = {rows[0] & kAbs, rows[1] & kAbs, rows[2] & kAbs, rows[3] & kAbs};
                        mma_f16(low[0], r, b[0][0][0] & kAbs, b[0][0][1] & kAbs);
                    }
                }
            }
            if (--carry == 0) {
                carry = kSliceFlush;
#pragma unroll
                for (int n = 0; n < NA; ++n) slice_carry(acc[n]);
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
    }
    // accumulator j = 2 h + e of tile n: row and column (relative to the item and the pass)
    // (PAIR: row 2 t4 + e, column g; h = 1 holds the odd digits, of one level more)
    auto row_of = [&](int n, int h, int e) { return PAIR ? 2 * t4 + e : WIDE ? 8 * n + 2 * t4 + e : g + 8 * h; };
    auto col_of = [&](int h, int e) { return PAIR ? g : WIDE ? g + 8 * h : 2 * t4 + e; };
    int er[NA][4], ec[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int64_t c = n0 + col_of(j >> 1, j & 1);
        const uint32_t M = c < a.k ? cmax[c] : 0u;
        ec[j] = M ? slice_exp(M) : 0;
#pragma unroll
        for (int n = 0; n < NA; ++n) {
            const int r = row_of(n, j >> 1, j & 1);
            er[n][j] = r < w.B ? q.rexp[w.yrow + r] : 0;
        }
    }
    // every output's terms must be resolved by the fixed point (or be exactly zero)
    bool ok = true;
#pragma unroll
    for (int n = 0; n < NA; ++n)
#pragma unroll
        for (int j = 0; j < 4; ++j) ok &= er[n][j] >= 0 && (er[n][j] == 0 || ec[j] == 0 || low[n][PAIR ? j & 1 : j] >= kSliceGuard);
    const int e9 = NINTH ? q.rexp[w.yrow + 8] : 0;
    if (NINTH) {
        ok &= e9 >= 0;
#pragma unroll
        for (int h = 0; h < NX; ++h)   // lanes t4 = 0 hold digit 0
            ok &= e9 == 0 || ec[2 * h] == 0 || t4 != 0 || nlow[2 * h] >= kSliceGuard;
    }
    if (!CAREFUL && !__all_sync(0xffffffffu, ok || force)) return false;
    uint32_t bad = 0;   // those for slice_one_output: bit 4 n + j, 8 + h for the ninth row's column g + 8 h
    if (CAREFUL) {
        const bool again = !__all_sync(0xffffffffu, ok);
        if (lane == 0) slice_state(ring)[2] = again ? max(slice_state(ring)[2], 1u) : 0u;
        int *sum = reinterpret_cast<int *>(ring);
        slice_digit_sums(vsrc, w.B, K, q.xdig, q.ldp, n0, s_x, sum, lane);
        bool scaled = e9 >= 0;
        // a complex output whose every term has a part that is zero throughout is an exact zero
        auto zero = [&](int r, int c) {
            if (sizeof(T) == sizeof(double)) return false;
            const uint32_t *own = q.cown + (cmax - q.cmax);
            const int parts = q.rparts[w.yrow + r];
            return !((parts & 1) && own[n0 + c]) && !((parts & 2) && own[(n0 + c) ^ 1]);
        };
#pragma unroll
        for (int n = 0; n < NA; ++n)
#pragma unroll
            for (int j = 0; j < (PAIR ? 2 : 4); ++j) {
                scaled &= er[n][j] >= 0;
                const int r = row_of(n, j >> 1, j & 1), c = col_of(j >> 1, j & 1);
                if (er[n][j] != 0 && ec[j] != 0 && low[n][j] < slice_guard(sum[r] + sum[16 + c], K) && !zero(r, c))
                    bad |= 1u << (4 * n + j);
            }
        if (NINTH && t4 == 0)
#pragma unroll
            for (int h = 0; h < NX; ++h)
                if (e9 != 0 && ec[2 * h] != 0 && nlow[2 * h] < slice_guard(sum[8] + sum[16 + g + 8 * h], K) &&
                    !zero(8, g + 8 * h))
                    bad |= 256u << h;
        if (!__all_sync(0xffffffffu, scaled) ||
            __reduce_add_sync(0xffffffffu, __popc(bad)) > min(min(kSliceSingles, K >> 4), w.B * (WIDE ? 4 : 2)))
            return false;
        __syncwarp();   // before the next pass's tiles go where the sums were
    }
    auto store = [&](int64_t row, int64_t c, double o) {
        double *y = static_cast<double *>(a.Y) + row * a.ldy + c;
        if (!q.alpha_pow2) o *= a.alpha;
        if (a.beta_nz) o += a.beta * *y;
        if (a.gamma_nz) o += a.gamma * static_cast<const double *>(a.Z)[row * a.ldz + c];
        *y = o;
        if (a.item_partials) dot += static_cast<const double *>(a.R)[row * a.ldr + c] * o;
    };
    if constexpr (NINTH) {
#pragma unroll
        for (int h = 0; h < NX; ++h) {   // column g + 8 h
            // the digits of X in units of their last, for the lane's digits 2 t4 and 2 t4 + 1 of the row
            float t[2][8];
#pragma unroll
            for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int d = 0; d < kSliceDigits; ++d)
                    t[e][d] = WIDE ? ninth[d % NJ][2 * h + e] : ninth[d / 2 % NJ][2 * (d & 1) + e];
            const double o = slice_value_of_lanes(t, t4, e9 + ec[2 * h] - 2114 + q.alpha_exp);
            if (t4 == 0 && n0 + g + 8 * h < a.k && !(bad & (256u << h))) store(w.yrow + 8, n0 + g + 8 * h, o);
        }
    }
#pragma unroll
    for (int n = 0; n < NA; ++n)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (PAIR && j >= 2) continue;
            const int r = row_of(n, j >> 1, j & 1);
            const int64_t c = n0 + col_of(j >> 1, j & 1);
            if (r >= (NINTH ? 8 : w.B) || c >= a.k || (bad & (1u << (4 * n + j)))) continue;
            const int64_t row = w.yrow + r;
            float lv[kSliceLevels];
#pragma unroll
            for (int L = 0; L < kSliceLevels; ++L)
                lv[L] = acc[n][L][j] + (PAIR && L > 0 ? acc[n][L > 0 ? L - 1 : 0][(j + 2) & 3] : 0.f);
            store(row, c, slice_value(lv, er[n][j] + ec[j] - 2114 + q.alpha_exp));
        }
    if (CAREFUL)
        for (unsigned lanes; (lanes = __ballot_sync(0xffffffffu, bad != 0)) != 0;) {
            const int src = __ffs(lanes) - 1, bit = __ffs(bad) - 1, j = bit & 3;
            const bool last = bit >= 8;
            const int r = __shfl_sync(0xffffffffu, last ? 8 : row_of(bit >> 2, j >> 1, j & 1), src);
            const int c = __shfl_sync(0xffffffffu, last ? g + 8 * j : col_of(j >> 1, j & 1), src);
            double o = slice_one_output<TRANS, T>(a, w, r, n0 + c, lane);
            if (q.alpha_pow2) o *= a.alpha;
            if (lane != src) continue;
            store(w.yrow + r, n0 + c, o);
            bad &= bad - 1;
        }
    return true;
}

template <bool TRANS, bool WIDE, bool CAREFUL, typename T>
__device__ __forceinline__ bool slice_pass_rows(const ProdArgs &a, const SliceArgs &q, const WorkItem &w,
                                                const unsigned char *vsrc, int K, int64_t n0, const uint32_t *cmax,
                                                unsigned char *ring, const int32_t *s_x, int lane, bool force,
                                                double &dot) {
    return w.B <= 8 ? slice_pass<TRANS, WIDE, 1, false, CAREFUL, T>(a, q, w, vsrc, K, n0, cmax, ring, s_x, lane, force, dot)
           : w.B == 9 ? slice_pass<TRANS, WIDE, 1, true, CAREFUL, T>(a, q, w, vsrc, K, n0, cmax, ring, s_x, lane, force, dot)
                      : slice_pass<TRANS, WIDE, 2, false, CAREFUL, T>(a, q, w, vsrc, K, n0, cmax, ring, s_x, lane, force, dot);
}

// A pass with unresolved outputs, or the first attempt at one where the warp's last ones
// had outputs below kSliceGuard (panels of a few large entries; the outputs are the same bits either way)
template <bool TRANS, bool WIDE, typename T>
__device__ __noinline__ bool slice_pass_again(const ProdArgs &a, const SliceArgs &q, const WorkItem &w,
                                              const unsigned char *vsrc, int K, int64_t n0, const uint32_t *cmax,
                                              unsigned char *ring, const int32_t *s_x, int lane, double &dot) {
    return slice_pass_rows<TRANS, WIDE, true, T>(a, q, w, vsrc, K, n0, cmax, ring, s_x, lane, false, dot);
}

// One warp per work item (up to 16 output rows). WIDE: k > 8, passes of 16
// columns with a last one of 8 where that is enough; otherwise one pass of up to 8
// columns.
// Complex operators (T = double2, TA its arithmetic): the kernel sees two real
// columns a complex one and two virtual columns a complex value, re meeting the
// X row x and im the row i x (slice_panel_kernel).
// (The arguments are grid constants: the calls take their addresses, and with a copy on the
// stack the k = 32 product on 50k zinc-blende atoms took 1.48 ms against 1.45.)
template <bool TRANS, bool WIDE, typename T, typename TA>
__global__ void __launch_bounds__(128, WIDE ? 3 : 4) slice_product_kernel(const __grid_constant__ ProdArgs a,
                                                                            const __grid_constant__ SliceArgs q) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int kRing = kSliceStages * 16 * kSliceTile;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char *ring = smem_raw + (size_t)warp * (kRing + kSliceList + kSliceState);
    int32_t *s_x = reinterpret_cast<int32_t *>(ring + kRing);
    volatile uint32_t *state = slice_state(ring);
    if (lane == 0) {
        state[0] = ~0u;
        state[2] = 0;
    }
    __syncwarp();
    double dot = 0.0;

    // the next item is claimed when an item starts (lane 0's value counts)
    auto claim = [&](int64_t from) -> unsigned long long {
        if (!a.queue) return (unsigned long long)(from + (int64_t)gridDim.x * 4);
        return lane == 0 ? atomicAdd(reinterpret_cast<unsigned long long *>(a.queue), 1ull) : 0ull;
    };
    int64_t it = (int64_t)blockIdx.x * 4 + warp;
    if (a.queue) it = (int64_t)__shfl_sync(0xffffffffu, claim(0), 0);
    while (it < a.n_items) {
        const unsigned long long next = claim(it);
        const WorkItem w = a.items[it];
        const SliceItem si = q.sitems[it];
        const uint32_t *cmax = q.cmax + (int64_t)si.strct * q.ldp;
        if ((uint32_t)si.strct != state[0]) {
            // a small structure is not sliced, nor a pass with a column outside the sliced range or
            // mostly tiny (one such column of 32: 5.06 ms at k = 32 on 50k zinc-blende atoms, 8.91
            // with all of them by multiply-adds)
            const uint32_t most = (uint32_t)q.struct_rows[si.strct] / 8 * 3;
            uint32_t plain = q.struct_nnz[si.strct] < q.min_nnz ? ~0u : 0u;
            for (int c0 = 0; c0 < (int)a.k; c0 += 32) {
                const int c = c0 + lane;
                const unsigned m = __ballot_sync(
                    0xffffffffu, c < (int)a.k && (!slice_exp_ok(cmax[c]) || q.ccnt[(int64_t)si.strct * q.ldp + c] > most));
                if (m & 0xffffu) plain |= 1u << min(c0 >> 4, 31);
                if (m >> 16) plain |= 1u << min((c0 >> 4) + 1, 31);
            }
            __syncwarp();
            if (lane == 0) {
                state[0] = (uint32_t)si.strct;
                state[1] = plain;
            }
            __syncwarp();
        }
        uint32_t skip = si.doff < 0 ? ~0u : state[1];   // this item's passes that are not tried
        constexpr int cw = sizeof(T) / sizeof(double);
        const int K = cw * w.K, nsteps = (K + 15) >> 4;
        const unsigned char *vsrc = q.vdig + si.doff;
        if (skip != ~0u && nsteps > 0) {
            // X row of every virtual column (a valid row past the last one: its digits meet zeros)
            __syncwarp();
            for (int e = lane; e < w.nlist; e += 32) {
                const int64_t l = w.lbegin + e;
                const int xr = TRANS ? a.tl.xrow[l] : a.fl.xrow[l];
                const int pc = TRANS ? a.tl.vcol[l] : a.fl.pcol[l];
                const int wd = TRANS ? a.tl.bi[l] : a.fl.w[l];
                for (int t = 0; t < cw * wd; ++t) s_x[cw * pc + t] = cw * xr + t;
                if (e == w.nlist - 1)
                    for (int t = K; t < 16 * nsteps + 16; ++t) s_x[t] = cw * xr;
            }
            __syncwarp();
        }
        if constexpr (!WIDE) {   // one pass
            const bool tried = skip == 0;
            if (!tried || state[2] || !slice_pass_rows<TRANS, false, false, T>(a, q, w, vsrc, K, 0, cmax, ring, s_x, lane, false, dot)) {
                const WorkItem wc = w;   // copies: the calls take addresses, which would keep w and dot in memory
                double dc = dot;
                if (!tried || !slice_pass_again<TRANS, false, T>(a, q, wc, vsrc, K, 0, cmax, ring, s_x, lane, dc))
                    fma_columns<TRANS, T, TA>(a, 0, a.k, wc, ring, lane, dc);
                __syncwarp();
                dot = dc;
            }
        } else {
            int64_t n0 = 0;
            while (n0 < a.k) {
                // sliced up to the next pass that is not tried
                const uint32_t left = skip >> min((int)(n0 >> 4), 31);
                const int64_t stop = left ? min(a.k, n0 + 16 * (int64_t)(__ffs(left) - 1)) : a.k;
                bool ok = n0 >= stop || state[2] < kSliceWary, force = false;
            attempt:
                for (; ok && n0 + 8 < stop; n0 += ok ? 16 : 0)
                    ok = slice_pass_rows<TRANS, true, false, T>(a, q, w, vsrc, K, n0, cmax, ring, s_x, lane, force, dot), force = false;
                if (ok && n0 < stop) {
                    ok = slice_pass_rows<TRANS, false, false, T>(a, q, w, vsrc, K, n0, cmax, ring, s_x, lane, force, dot);
                    n0 += ok ? 8 : 0;
                }
                if (n0 >= a.k) break;
                if (!ok && state[2] < kSliceWary) {
                    __syncwarp();
                    if (lane == 0) state[2] = state[2] + 1;
                    __syncwarp();
                }
                if (!ok && state[2] < kSliceWary && slice_recheck<T>(q, vsrc, w.B, K, w.yrow, a.k, n0, cmax, s_x, lane)) {
                    ok = force = true;
                    goto attempt;
                }
                const WorkItem wc = w;   // copies: the calls take addresses, which would keep w and dot in memory
                double dc = dot;
                const bool wide = n0 + 8 < a.k;
                if (!ok)
                    ok = wide ? slice_pass_again<TRANS, WIDE, T>(a, q, wc, vsrc, K, n0, cmax, ring, s_x, lane, dc)
                              : slice_pass_again<TRANS, false, T>(a, q, wc, vsrc, K, n0, cmax, ring, s_x, lane, dc);
                else
                    ok = false;   // not tried
                int64_t n1 = n0 + (wide ? 16 : 8);
                if (!ok) {
                    // by multiply-adds, with the passes after it that are not tried: after two with
                    // unresolved outputs none of the item's are
                    const uint32_t self = 1u << min((int)(n0 >> 4), 31);
                    if (!(skip & self)) skip = skip == state[1] ? skip | self : ~0u;
                    if (skip == ~0u) n1 = a.k;
                    while (n1 < a.k && (skip >> min((int)(n1 >> 4), 31) & 1u)) n1 += 16;
                    n1 = min(n1, a.k);
                    fma_columns<TRANS, T, TA>(a, n0, n1, wc, ring, lane, dc);
                    __syncwarp();   // before the next pass's tiles go where the multiply-adds kept their lists
                }
                dot = dc;
                n0 = n1;
            }
        }
        if (a.item_partials) {
            // the item's share of the fused dot at the item's index (summed in a fixed order afterwards)
            for (int m = 16; m > 0; m >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, m);
            if (lane == 0) a.item_partials[it] = dot;
            dot = 0.0;
        }
        it = a.queue ? (int64_t)__shfl_sync(0xffffffffu, next, 0) : (int64_t)next;
    }
}

using SliceKernel = void (*)(ProdArgs, SliceArgs);
template <bool TRANS, typename T, typename TA>
SliceKernel slice_kernel(int64_t k) {
    return k <= 8 ? slice_product_kernel<TRANS, false, T, TA> : slice_product_kernel<TRANS, true, T, TA>;
}

template <typename T, typename TA>
const void *slice_kernel_of(bool trans, int64_t k) {
    return (const void *)(trans ? slice_kernel<true, T, TA>(k) : slice_kernel<false, T, TA>(k));
}

constexpr size_t kSliceSmem = 4 * ((size_t)kSliceStages * 16 * kSliceTile + kSliceList + kSliceState);

template <typename T, typename TA>
cudaError_t launch_slice(bool trans, const ProdArgs &a, const SliceArgs &q, cudaStream_t s) {
    const SliceKernel kern = trans ? slice_kernel<true, T, TA>(a.k) : slice_kernel<false, T, TA>(a.k);
    cudaError_t e = cudaFuncSetAttribute((const void *)kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSliceSmem);
    if (e != cudaSuccess) return e;
    kern<<<a.grid, 128, kSliceSmem, s>>>(a, q);
    return cudaGetLastError();
}

}  // namespace

}  // namespace vbcsr
