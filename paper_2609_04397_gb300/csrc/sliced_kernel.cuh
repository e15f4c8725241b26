// The product kernel of the sliced FP64 operators (sliced.cuh): spmm_sliced.cu
// instantiates it for real operators, spmm_sliced_c128.cu for complex ones.
#pragma once

#include "fma_kernel.cuh"
#include "sliced.cuh"

namespace vbcsr {

namespace {

constexpr int kSliceList = (kSliceKMax + 16) * sizeof(int32_t);   // X rows of an item and of one step more
constexpr int kSliceStages = 4;   // value tiles in flight per warp (16 columns, up to 1792 bytes each)

// the operator's own arithmetic, for what is not sliced
template <int B, bool TRANS, typename T, typename TA>
__device__ __noinline__ void fma_item_fallback(const ProdArgs &a, const WorkItem &w, int kc, int32_t *s_x,
                                               int64_t *s_a, int lane, double &dot) {
    process_item<B, TRANS, T, TA, T, T>(a, w, kc, s_x, s_a, nullptr, lane, dot);
}

// Columns [n0, k) of item w by FP64 multiply-adds (complex T: two real columns of the
// sliced panels make one)
template <bool TRANS, typename T, typename TA>
__device__ __noinline__ void fma_columns(const ProdArgs &a, int64_t n0, const WorkItem &w, unsigned char *smem, int lane,
                                         double &dot) {
    ProdArgs b = a;
    constexpr int cw = sizeof(T) / sizeof(double);
    b.k = (a.k - n0) / cw;
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
// Returns false, with nothing written, when an output is not resolved by the
// fixed point.
template <bool TRANS, bool WIDE, int NR, bool NINTH = false>
__device__ __forceinline__ bool slice_pass(const ProdArgs &a, const SliceArgs &q, const WorkItem &w,
                                           const unsigned char *vsrc, int nsteps, int64_t n0, const uint32_t *cmax,
                                           unsigned char *ring, const int32_t *s_x, int lane, double &dot) {
    constexpr int S = kSliceStages, kStage = 16 * kSliceTile;
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
    if (!__all_sync(0xffffffffu, ok)) return false;
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
            if (t4 == 0 && n0 + g + 8 * h < a.k) store(w.yrow + 8, n0 + g + 8 * h, o);
        }
    }
#pragma unroll
    for (int n = 0; n < NA; ++n)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (PAIR && j >= 2) continue;
            const int r = row_of(n, j >> 1, j & 1);
            const int64_t c = n0 + col_of(j >> 1, j & 1);
            if (r >= (NINTH ? 8 : w.B) || c >= a.k) continue;
            const int64_t row = w.yrow + r;
            float lv[kSliceLevels];
#pragma unroll
            for (int L = 0; L < kSliceLevels; ++L)
                lv[L] = acc[n][L][j] + (PAIR && L > 0 ? acc[n][L > 0 ? L - 1 : 0][(j + 2) & 3] : 0.f);
            store(row, c, slice_value(lv, er[n][j] + ec[j] - 2114 + q.alpha_exp));
        }
    return true;
}

// One warp per work item (up to 16 output rows). WIDE: k > 8, passes of 16
// columns with a last one of 8 where that is enough; otherwise one pass of up to 8
// columns.
// Complex operators (T = double2, TA its arithmetic): the kernel sees two real
// columns a complex one and two virtual columns a complex value, re meeting the
// X row x and im the row i x (slice_panel_kernel).
template <bool TRANS, bool WIDE, typename T, typename TA>
__global__ void __launch_bounds__(128, WIDE ? 3 : 4) slice_product_kernel(ProdArgs a, SliceArgs q) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int kRing = kSliceStages * 16 * kSliceTile;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char *ring = smem_raw + (size_t)warp * (kRing + kSliceList);
    int32_t *s_x = reinterpret_cast<int32_t *>(ring + kRing);
    double dot = 0.0;

    // the next item is claimed when an item starts (lane 0's value counts)
    auto claim = [&](int64_t from) -> unsigned long long {
        if (!a.queue) return (unsigned long long)(from + (int64_t)gridDim.x * 4);
        return lane == 0 ? atomicAdd(reinterpret_cast<unsigned long long *>(a.queue), 1ull) : 0ull;
    };
    int last_strct = -1;
    bool last_plain = false;
    int64_t it = (int64_t)blockIdx.x * 4 + warp;
    if (a.queue) it = (int64_t)__shfl_sync(0xffffffffu, claim(0), 0);
    while (it < a.n_items) {
        const unsigned long long next = claim(it);
        const WorkItem w = a.items[it];
        const SliceItem si = q.sitems[it];
        const uint32_t *cmax = q.cmax + (int64_t)si.strct * q.ldp;
        if (si.strct != last_strct) {
            // a small structure, or one with a column outside the sliced range or mostly tiny, is not sliced
            last_strct = si.strct;
            const uint32_t most = (uint32_t)q.struct_rows[si.strct] >> 2;
            bool p = q.struct_nnz[si.strct] < q.min_nnz;
            for (int c = lane; c < (int)a.k; c += 32)
                p |= !slice_exp_ok(cmax[c]) || q.ccnt[(int64_t)si.strct * q.ldp + c] > most;
            last_plain = __any_sync(0xffffffffu, p);
        }
        const bool plain = last_plain || si.doff < 0;
        constexpr int cw = sizeof(T) / sizeof(double);
        const int K = cw * w.K, nsteps = (K + 15) >> 4;
        const unsigned char *vsrc = q.vdig + si.doff;
        int64_t n0 = 0;
        if (!plain && nsteps > 0) {
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
        if (!plain) {
            bool ok = true;
            if constexpr (WIDE)
                for (; ok && n0 + 8 < a.k; n0 += ok ? 16 : 0)
                    ok = w.B <= 8 ? slice_pass<TRANS, true, 1>(a, q, w, vsrc, nsteps, n0, cmax, ring, s_x, lane, dot)
                         : w.B == 9
                             ? slice_pass<TRANS, true, 1, true>(a, q, w, vsrc, nsteps, n0, cmax, ring, s_x, lane, dot)
                             : slice_pass<TRANS, true, 2>(a, q, w, vsrc, nsteps, n0, cmax, ring, s_x, lane, dot);
            if (ok && n0 < a.k) {
                ok = w.B <= 8 ? slice_pass<TRANS, false, 1>(a, q, w, vsrc, nsteps, n0, cmax, ring, s_x, lane, dot)
                     : w.B == 9
                         ? slice_pass<TRANS, false, 1, true>(a, q, w, vsrc, nsteps, n0, cmax, ring, s_x, lane, dot)
                         : slice_pass<TRANS, false, 2>(a, q, w, vsrc, nsteps, n0, cmax, ring, s_x, lane, dot);
                n0 += ok ? 8 : 0;
            }
        }
        if (n0 < a.k) {
            const WorkItem wc = w;   // copies: the call takes addresses, which would keep w and dot in memory
            double dc = dot;
            fma_columns<TRANS, T, TA>(a, n0, wc, ring, lane, dc);
            dot = dc;
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

constexpr size_t kSliceSmem = 4 * ((size_t)kSliceStages * 16 * kSliceTile + kSliceList);

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
