// Sliced FP64 products (sliced.cuh): the digit copies of the values and of X,
// and the tensor-core product kernel of an FP64 operator, forward and adjoint.
#include "fma_kernel.cuh"
#include "sliced.cuh"

namespace vbcsr {

namespace {

// ---------------------------------------------------------------------------
// X: column maxima per structure, then the digits

// A CTA takes `per` consecutive chunks of X rows (each of one structure);
// thread tx of TX takes columns tx, tx + TX, ..., threads ty stride the rows.
struct ColWalk {
    int tx, ty, TX, TY;
    __device__ __forceinline__ ColWalk(int cols) {
        TX = 1;
        while (TX < cols && TX < 32) TX <<= 1;
        TY = blockDim.x / TX;
        tx = threadIdx.x % TX;
        ty = threadIdx.x / TX;
    }
};

// f(row0, rows, structure, last) over the CTA's chunks; `last` marks the end of a
// structure's run of chunks
template <typename F>
__device__ __forceinline__ void over_chunks(const SliceChunk *chunks, int64_t n_chunks, int per, F f) {
    const int64_t q1 = min(n_chunks, ((int64_t)blockIdx.x + 1) * per);
    for (int64_t q = (int64_t)blockIdx.x * per; q < q1; ++q) {
        const SliceChunk c = chunks[q];
        f(c, q + 1 == q1 || chunks[q + 1].strct != c.strct);
    }
}

__global__ void __launch_bounds__(256) slice_colmax_kernel(const SliceChunk *chunks, int64_t n_chunks, int per,
                                                           const double *__restrict__ X, int64_t ldx, int k, int ldp,
                                                           uint32_t *cmax) {
    __shared__ uint32_t red[256];
    const ColWalk w(k);
    for (int c0 = 0; c0 < k; c0 += w.TX) {
        const int col = c0 + w.tx;
        uint32_t m = 0;
        over_chunks(chunks, n_chunks, per, [&](const SliceChunk &c, bool last) {
            if (col < k) {
                const double *x = X + (int64_t)c.row0 * ldx + col;
#pragma unroll 4
                for (int r = w.ty; r < c.nrows; r += w.TY) m = max(m, slice_mag(x[(int64_t)r * ldx]));
            }
            if (!last) return;
            __syncthreads();
            red[threadIdx.x] = m;
            __syncthreads();
            for (int h = w.TY / 2; h > 0; h >>= 1) {
                if (w.ty < h) red[threadIdx.x] = max(red[threadIdx.x], red[threadIdx.x + h * w.TX]);
                __syncthreads();
            }
            if (w.ty == 0 && col < k && red[w.tx]) atomicMax(cmax + (int64_t)c.strct * ldp + col, red[w.tx]);
            m = 0;
        });
    }
}

// X as biased fixed point [rows, ldp] (8 bytes an element, 7 of them digits);
// columns k .. ldp - 1 are zero. ccnt counts the elements below 2^-10 of their
// column's maximum.
__global__ void __launch_bounds__(256) slice_panel_kernel(const SliceChunk *chunks, int64_t n_chunks, int per,
                                                          const double *__restrict__ X, int64_t ldx, int k, int ldp,
                                                          const uint32_t *__restrict__ cmax, uint32_t *ccnt,
                                                          uint64_t *__restrict__ out) {
    __shared__ uint32_t red[256];
    const ColWalk w(ldp);
    for (int c0 = 0; c0 < ldp; c0 += w.TX) {
        const int col = c0 + w.tx;
        uint32_t tiny = 0;
        over_chunks(chunks, n_chunks, per, [&](const SliceChunk &c, bool last) {
            if (col < ldp) {
                const uint32_t M = col < k ? cmax[(int64_t)c.strct * ldp + col] : 0u;
                const bool live = M != 0 && slice_exp_ok(M);
                const int E = slice_exp(M);
                const double *x = X + (int64_t)c.row0 * ldx + (live ? col : 0);
                uint64_t *o = out + (int64_t)c.row0 * ldp + col;
#pragma unroll 4
                for (int r = w.ty; r < c.nrows; r += w.TY) {
                    const double v = live ? x[(int64_t)r * ldx] : 0.0;
                    tiny += live && (slice_mag(v) >> 20) + 10 < (M >> 20);
                    o[(int64_t)r * ldp] = slice_bytes(v, E);
                }
            }
            if (!last) return;
            __syncthreads();
            red[threadIdx.x] = tiny;
            __syncthreads();
            for (int h = w.TY / 2; h > 0; h >>= 1) {
                if (w.ty < h) red[threadIdx.x] += red[threadIdx.x + h * w.TX];
                __syncthreads();
            }
            if (w.ty == 0 && col < k && red[w.tx]) atomicAdd(ccnt + (int64_t)c.strct * ldp + col, red[w.tx]);
            tiny = 0;
        });
    }
}

// ---------------------------------------------------------------------------
// values: one warp per work item; row maxima, then 16-column tiles of digits
// [tile][digit][row][16 columns], two tiles at a time staged in shared memory
// and stored 16 bytes a lane. Forward items are read with the lanes along a row
// of the page; adjoint ones (TRANS), whose rows are the columns of the pages'
// blocks, with BP = 1, 2, 4, 8 or 16 lanes along the item's rows (consecutive in
// the pages) and 32 / BP virtual columns a load: with a virtual column per lane
// every load touched 32 sectors (0.47 ms for 3.8e7 entries, the forward
// form 0.18).

// the digits of element (row p, column t of the two staged tiles)
__device__ __forceinline__ void stage_digits(uint8_t *stage, int B, int p, int t, double v, int E) {
    const uint64_t u = slice_bytes(E > 0 ? v : 0.0, E);
    uint8_t *o = stage + (t >> 4) * B * kSliceTile + p * 16 + (t & 15);
#pragma unroll
    for (int i = 0; i < kSliceDigits; ++i) o[i * B * 16] = (uint8_t)(u >> (8 * (6 - i)));
}

// 16 loads of an adjoint item at once: row q of virtual columns t0 + u * (32 / BP) + lane / BP, u < BP
template <int BP>
__device__ __forceinline__ void adj_columns(const double *panel, const int64_t *s_a, const WorkItem &w, int t0, int lane,
                                            double (&v)[BP]) {
    const int q = lane % BP;
#pragma unroll
    for (int u = 0; u < BP; ++u) {
        const int t = t0 + u * (32 / BP) + lane / BP;
        v[u] = t < w.K && q < w.B ? panel[s_a[t] + q] : 0.0;
    }
}

template <int BP>
__device__ __forceinline__ void adj_item_digits(const double *panel, const int64_t *s_a, const WorkItem &w, uint8_t *dst,
                                                uint8_t *stage, int32_t *rexp, int lane) {
    uint32_t m = 0;
    for (int t0 = 0; t0 < w.K; t0 += 32) {
        double v[BP];
        adj_columns<BP>(panel, s_a, w, t0, lane, v);
#pragma unroll
        for (int u = 0; u < BP; ++u) m = max(m, slice_mag(v[u]));
    }
#pragma unroll
    for (int h = BP; h < 32; h <<= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, h));
    const int E = m == 0 ? 0 : (slice_exp_ok(m) ? slice_exp(m) : -1), q = lane % BP;
    if (lane < w.B) rexp[w.yrow + lane] = E;
    const int nt = (w.K + 15) >> 4;
    for (int c = 0; c < nt; c += 2) {
        double v[BP];
        adj_columns<BP>(panel, s_a, w, 16 * c, lane, v);
        if (q < w.B)
#pragma unroll
            for (int u = 0; u < BP; ++u) stage_digits(stage, w.B, q, u * (32 / BP) + lane / BP, v[u], E);
        __syncwarp();
        uint4 *d = reinterpret_cast<uint4 *>(dst + (int64_t)c * w.B * kSliceTile);
        const int n = min(2, nt - c) * w.B * (kSliceTile / 16);
        for (int e = lane; e < n; e += 32) d[e] = reinterpret_cast<uint4 *>(stage)[e];
        __syncwarp();
    }
}

template <bool TRANS>
__global__ void __launch_bounds__(128) slice_values_kernel(const WorkItem *items, const SliceItem *sitems,
                                                           int64_t n_items, AdjList tl, const double *panel,
                                                           uint8_t *dig, int32_t *rexp) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warps = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint8_t *stage = smem_raw + (size_t)warp * 32 * kSliceTile;
    int64_t *s_a = reinterpret_cast<int64_t *>(smem_raw + (size_t)warps * 32 * kSliceTile) + (size_t)warp * kSliceKMax;
    __shared__ int s_e[4][16];
    for (int64_t it = (int64_t)blockIdx.x * warps + warp; it < n_items; it += (int64_t)gridDim.x * warps) {
        const WorkItem w = items[it];
        const SliceItem si = sitems[it];
        if (si.doff < 0) continue;   // too wide: never sliced
        if constexpr (TRANS) {
            __syncwarp();
            for (int e = lane; e < w.nlist; e += 32) {
                const int64_t l = w.lbegin + e;
                const int64_t pb = tl.pbase[l];
                const int kp = tl.kp[l], bi = tl.bi[l], vc = tl.vcol[l];
                for (int p = 0; p < bi; ++p) s_a[vc + p] = pb + (int64_t)p * kp + w.Kp;
            }
            __syncwarp();
            uint8_t *dst = dig + si.doff;
            if (w.B > 8) adj_item_digits<16>(panel, s_a, w, dst, stage, rexp, lane);
            else if (w.B > 4) adj_item_digits<8>(panel, s_a, w, dst, stage, rexp, lane);
            else if (w.B > 2) adj_item_digits<4>(panel, s_a, w, dst, stage, rexp, lane);
            else adj_item_digits<2>(panel, s_a, w, dst, stage, rexp, lane);
        } else {
            const double *src = panel + w.vbase;
            auto load = [&](int t, double (&v)[16]) {               // column t of the item, all rows at once
                const bool in = t < w.K;
                const double *c = src + (in ? t : 0);
#pragma unroll
                for (int p = 0; p < 16; ++p) v[p] = in && p < w.B ? c[(int64_t)p * w.Kp] : 0.0;
            };
            uint32_t m[16];
#pragma unroll
            for (int p = 0; p < 16; ++p) m[p] = 0;
            for (int t = lane; t < w.K; t += 32) {
                double v[16];
                load(t, v);
#pragma unroll
                for (int p = 0; p < 16; ++p) m[p] = max(m[p], slice_mag(v[p]));
            }
#pragma unroll
            for (int p = 0; p < 16; ++p) {
                const uint32_t r = __reduce_max_sync(0xffffffffu, m[p]);
                const int e = r == 0 ? 0 : (slice_exp_ok(r) ? slice_exp(r) : -1);
                if (lane == p) {
                    s_e[warp][p] = e;
                    if (p < w.B) rexp[w.yrow + p] = e;
                }
            }
            __syncwarp();
            const int nt = (w.K + 15) >> 4;
            for (int c = 0; c < nt; c += 2) {
                double v[16];
                load(16 * c + lane, v);
#pragma unroll
                for (int p = 0; p < 16; ++p) {
                    if (p >= w.B) break;
                    stage_digits(stage, w.B, p, lane, v[p], s_e[warp][p]);
                }
                __syncwarp();
                uint4 *dst = reinterpret_cast<uint4 *>(dig + si.doff + (int64_t)c * w.B * kSliceTile);
                const int n = min(2, nt - c) * w.B * (kSliceTile / 16);
                for (int q = lane; q < n; q += 32) dst[q] = reinterpret_cast<uint4 *>(stage)[q];
                __syncwarp();
            }
        }
    }
}

// ---------------------------------------------------------------------------
// the product

constexpr int kSliceList = (kSliceKMax + 16) * sizeof(int32_t);   // X rows of an item and of one step more
constexpr int kSliceStages = 4;   // value tiles in flight per warp (16 columns, up to 1792 bytes each)

template <int B, bool TRANS>
__device__ __noinline__ void fma_item_fallback(const ProdArgs &a, const WorkItem &w, int kc, int32_t *s_x,
                                               int64_t *s_a, int lane, double &dot) {
    process_item<B, TRANS, double, double, double, double>(a, w, kc, s_x, s_a, nullptr, lane, dot);
}

// Columns [n0, k) of item w by FP64 multiply-adds
template <bool TRANS>
__device__ __noinline__ void fma_columns(const ProdArgs &a, int64_t n0, const WorkItem &w, unsigned char *smem, int lane,
                                         double &dot) {
    ProdArgs b = a;
    b.k = a.k - n0;
    b.X = static_cast<const double *>(a.X) + n0;
    b.Y = static_cast<double *>(a.Y) + n0;
    if (a.gamma_nz) b.Z = static_cast<const double *>(a.Z) + n0;
    if (a.item_partials) b.R = static_cast<const double *>(a.R) + n0;
    int kc = 1;
    while (kc < b.k && kc < 32) kc <<= 1;
    int64_t *s_a = reinterpret_cast<int64_t *>(smem);
    int32_t *s_x = reinterpret_cast<int32_t *>(smem + kKMax * sizeof(int64_t));
#define VBCSR_SLICE_CASE(NB) \
    case NB: fma_item_fallback<NB, TRANS>(b, w, kc, s_x, s_a, lane, dot); break;
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
// (up to 16) rows on the M side and the 8 columns on the N side. Returns false,
// with nothing written, when an output is not resolved by the fixed point.
template <bool TRANS, bool WIDE, int NR>
__device__ __forceinline__ bool slice_pass(const ProdArgs &a, const SliceArgs &q, const WorkItem &w,
                                           const unsigned char *vsrc, int nsteps, int64_t n0, const uint32_t *cmax,
                                           unsigned char *ring, const int32_t *s_x, int lane, double &dot) {
    constexpr int S = kSliceStages, kStage = 16 * kSliceTile;
    constexpr int NX = WIDE ? 2 : 1, NA = WIDE ? NR : 1;
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
                    if (WIDE) {
                        const uint32_t cols[4] = {b[0][j][0], b[NX - 1][j][0], b[0][j][1], b[NX - 1][j][1]};
#pragma unroll
                        for (int n = 0; n < NA; ++n) mma_f16(acc[n][i + j], cols, v[n % NR][0], v[n % NR][1]);
                    } else {
                        mma_f16(acc[0][i + j], rows, b[0][j][0], b[0][j][1]);
                    }
                }
                if (i == 0) {   // magnitudes of the leading digits
                    constexpr uint32_t kAbs = 0x7fff7fffu;
                    if (WIDE) {
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
    auto row_of = [&](int n, int h, int e) { return WIDE ? 8 * n + 2 * t4 + e : g + 8 * h; };
    auto col_of = [&](int h, int e) { return WIDE ? g + 8 * h : 2 * t4 + e; };
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
        for (int j = 0; j < 4; ++j) ok &= er[n][j] >= 0 && (er[n][j] == 0 || ec[j] == 0 || low[n][j] >= kSliceGuard);
    if (!__all_sync(0xffffffffu, ok)) return false;
#pragma unroll
    for (int n = 0; n < NA; ++n)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (!WIDE && NR == 1 && j >= 2) continue;
            const int r = row_of(n, j >> 1, j & 1);
            const int64_t c = n0 + col_of(j >> 1, j & 1);
            if (r >= w.B || c >= a.k) continue;
            const int64_t row = w.yrow + r;
            float lv[kSliceLevels];
#pragma unroll
            for (int L = 0; L < kSliceLevels; ++L) lv[L] = acc[n][L][j];
            double o = slice_value(lv, er[n][j] + ec[j] - 2114 + q.alpha_exp);
            double *y = static_cast<double *>(a.Y) + row * a.ldy + c;
            if (!q.alpha_pow2) o *= a.alpha;
            if (a.beta_nz) o += a.beta * *y;
            if (a.gamma_nz) o += a.gamma * static_cast<const double *>(a.Z)[row * a.ldz + c];
            *y = o;
            if (a.item_partials) dot += static_cast<const double *>(a.R)[row * a.ldr + c] * o;
        }
    return true;
}

// Products of KC <= kSliceThin columns: the digits of X, not its columns, are the
// N side (8 of them a tile, 7 used, one tile a column), so an MMA forms digit i of
// the values times all digits of a column at once: 7 KC MMAs a step instead of 35.
// Every digit pair has an accumulator of its own, so nothing is dropped and the
// sums over up to kSliceKMax columns are exact without carries. X is [rows, KC].
// Bound by reading the value tiles (7 bytes an entry) and cutting them into f16
// pairs. 50k atoms, k = 1 / 2 / 3: 0.32 / 0.43 / 0.56 ms, multiply-adds 0.37 / 0.73 / 1.26.
template <bool TRANS, int KC, int NR>
__device__ __forceinline__ bool slice_thin(const ProdArgs &a, const SliceArgs &q, const WorkItem &w,
                                           const unsigned char *vsrc, int nsteps, const uint32_t *cmax,
                                           unsigned char *ring, const int32_t *s_x, int lane, double &dot) {
    constexpr int S = kSliceStages, kStage = 16 * kSliceTile;
    const int g = lane >> 2, t4 = lane & 3;
    float acc[kSliceDigits][KC][4], low[KC][4];
#pragma unroll
    for (int n = 0; n < KC; ++n)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            low[n][j] = 0.f;
#pragma unroll
            for (int i = 0; i < kSliceDigits; ++i) acc[i][n][j] = 0.f;
        }
    if (nsteps > 0) {
        const int tile = w.B * kSliceTile;
        constexpr int kChunks = (16 * kSliceTile / 16 + 31) / 32;
        bool mine[kChunks];
#pragma unroll
        for (int u = 0; u < kChunks; ++u) mine[u] = 16 * (lane + 32 * u) < tile;
        const unsigned char *src = vsrc + 16 * lane;
        auto issue = [&](int s) {
            const bool in = s < nsteps;
            unsigned char *dst = ring + (s % S) * kStage + 16 * lane;
#pragma unroll
            for (int u = 0; u < kChunks; ++u)
                if (in && mine[u]) cp_async16(dst + 512 * u, src + 512 * u);
            src += tile;
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        // digit g of the lane's four virtual columns: byte 6 - g (the eighth digit is zero)
        const uint8_t *xd = reinterpret_cast<const uint8_t *>(q.xdig) + (g < 7 ? 6 - g : 0);
        uint32_t x[KC][4];
        auto load_x = [&](int s) {
            const int4 xi = *reinterpret_cast<const int4 *>(s_x + 16 * s + 4 * t4);
            const int row[4] = {xi.x, xi.y, xi.z, xi.w};
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int n = 0; n < KC; ++n) x[n][r] = __ldg(xd + ((int64_t)row[r] * KC + n) * 8);
        };
        load_x(0);
#pragma unroll
        for (int s = 0; s < S - 1; ++s) issue(s);
        const int digit = w.B * 16;
        for (int s = 0; s < nsteps; ++s) {
            asm volatile("cp.async.wait_group %0;" ::"n"(S - 2) : "memory");
            __syncwarp();
            issue(s + S - 1);
            uint32_t b[KC][2];
#pragma unroll
            for (int n = 0; n < KC; ++n)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    // 0x6400 | byte is 1024 + byte in f16; less 1152
                    uint32_t p = (x[n][2 * h] + (x[n][2 * h + 1] << 16)) | 0x64006400u;
                    asm("sub.f16x2 %0, %0, %1;" : "+r"(p) : "r"(0x64806480u));
                    b[n][h] = g < 7 ? p : 0u;
                }
            load_x(s + 1);
            const unsigned char *st = ring + (s % S) * kStage + g * 16 + t4 * 4;
#pragma unroll
            for (int i = 0; i < kSliceDigits; ++i, st += digit) {
                uint32_t v[NR][2];
#pragma unroll
                for (int n = 0; n < NR; ++n) {
                    const uint32_t word = *reinterpret_cast<const uint32_t *>(st + 128 * n);
                    v[n][0] = slice_half2(word, 0x4140);
                    v[n][1] = slice_half2(word, 0x4342);
                }
                const uint32_t rows[4] = {v[0][0], v[NR - 1][0], v[0][1], v[NR - 1][1]};
#pragma unroll
                for (int n = 0; n < KC; ++n) mma_f16(acc[i][n], rows, b[n][0], b[n][1]);
                if (i == 0) {   // magnitudes of the leading digits (column 0 of the tile)
                    constexpr uint32_t kAbs = 0x7fff7fffu;
                    const uint32_t r[4] = {rows[0] & kAbs, rows[1] & kAbs, rows[2] & kAbs, rows[3] & kAbs};
#pragma unroll
                    for (int n = 0; n < KC; ++n) mma_f16(low[n], r, b[n][0] & kAbs, b[n][1] & kAbs);
                }
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
    }
    // accumulator 2 h + e: row g + 8 h, digit 2 t4 + e of X. Lanes t4 = 0 hold digit 0 and write.
    int er[2], ec[KC];
    bool ok = true;
#pragma unroll
    for (int h = 0; h < 2; ++h) er[h] = g + 8 * h < w.B ? q.rexp[w.yrow + g + 8 * h] : 0;
#pragma unroll
    for (int n = 0; n < KC; ++n) {
        const uint32_t M = cmax[n];
        ec[n] = M ? slice_exp(M) : 0;
#pragma unroll
        for (int h = 0; h < 2; ++h)
            ok &= er[h] >= 0 && (er[h] == 0 || ec[n] == 0 || t4 != 0 || low[n][2 * h] >= kSliceGuard);
    }
    if (!__all_sync(0xffffffffu, ok)) return false;
#pragma unroll
    for (int h = 0; h < NR; ++h) {
        const int r = g + 8 * h;
#pragma unroll
        for (int n = 0; n < KC; ++n) {
            // sum over the digits of the values, in units of their last: hi * 2^24 + lo, for the
            // lane's two digits of X together (hi below 2^57, lo below 2^49)
            long long hi = 0, lo = 0;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                long long p = __float2int_rn(acc[0][n][2 * h + e]), t = __float2int_rn(acc[4][n][2 * h + e]);
#pragma unroll
                for (int i = 1; i < 4; ++i) p = p * 256 + __float2int_rn(acc[i][n][2 * h + e]);
#pragma unroll
                for (int i = 5; i < 7; ++i) t = t * 256 + __float2int_rn(acc[i][n][2 * h + e]);
                hi = hi * 256 + p;
                lo = lo * 256 + t;
            }
            // a pair of digits weighs 2^-16 of the one before
            double d = fma((double)hi, 16777216.0, (double)lo);
            d *= t4 == 0 ? 1.0 : t4 == 1 ? 0x1p-16 : t4 == 2 ? 0x1p-32 : 0x1p-48;
            d += __shfl_xor_sync(0xffffffffu, d, 2);
            d += __shfl_xor_sync(0xffffffffu, d, 1);
            if (t4 == 0 && r < w.B) {
                // digits 0 and 1 of X in units of 256^5: the same exponent as the level sums of a pass
                const uint64_t bits = (uint64_t)__double_as_longlong(d);
                const int e2 = er[h] + ec[n] - 2114 + q.alpha_exp;
                double o = (bits << 1) == 0 ? 0.0 : __longlong_as_double((long long)(bits + ((uint64_t)(int64_t)e2 << 52)));
                const int64_t row = w.yrow + r;
                double *y = static_cast<double *>(a.Y) + row * a.ldy + n;
                if (!q.alpha_pow2) o *= a.alpha;
                if (a.beta_nz) o += a.beta * *y;
                if (a.gamma_nz) o += a.gamma * static_cast<const double *>(a.Z)[row * a.ldz + n];
                *y = o;
                if (a.item_partials) dot += static_cast<const double *>(a.R)[row * a.ldr + n] * o;
            }
        }
    }
    return true;
}

// One warp per work item (up to 16 output rows). FORM 0: k > 8, passes of 16
// columns with a last one of 8 where that is enough; 8: one pass of up to 8
// columns; 1 .. kSliceThin: that many columns.
template <bool TRANS, int FORM>
__global__ void __launch_bounds__(128, FORM == 0 || FORM == 3 ? 3 : FORM == 1 ? 5 : 4) slice_product_kernel(ProdArgs a, SliceArgs q) {
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
            bool p = q.struct_nnz[si.strct] * a.k < slice_min_work(a.k);
            for (int c = lane; c < (int)a.k; c += 32)
                p |= !slice_exp_ok(cmax[c]) || q.ccnt[(int64_t)si.strct * q.ldp + c] > most;
            last_plain = __any_sync(0xffffffffu, p);
        }
        const bool plain = last_plain || si.doff < 0;
        const int nsteps = (w.K + 15) >> 4;
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
                for (int t = 0; t < wd; ++t) s_x[pc + t] = xr + t;
                if (e == w.nlist - 1)
                    for (int t = w.K; t < 16 * nsteps + 16; ++t) s_x[t] = xr;
            }
            __syncwarp();
        }
        if (!plain) {
            bool ok = true;
            if constexpr (FORM == 0)
                for (; ok && n0 + 8 < a.k; n0 += ok ? 16 : 0)
                    ok = w.B <= 8 ? slice_pass<TRANS, true, 1>(a, q, w, vsrc, nsteps, n0, cmax, ring, s_x, lane, dot)
                                  : slice_pass<TRANS, true, 2>(a, q, w, vsrc, nsteps, n0, cmax, ring, s_x, lane, dot);
            if constexpr (FORM == 0 || FORM == 8) {
                if (ok && n0 < a.k) {
                    ok = w.B <= 8
                             ? slice_pass<TRANS, false, 1>(a, q, w, vsrc, nsteps, n0, cmax, ring, s_x, lane, dot)
                             : slice_pass<TRANS, false, 2>(a, q, w, vsrc, nsteps, n0, cmax, ring, s_x, lane, dot);
                    n0 += ok ? 8 : 0;
                }
            } else {
                ok = w.B <= 8 ? slice_thin<TRANS, FORM, 1>(a, q, w, vsrc, nsteps, cmax, ring, s_x, lane, dot)
                              : slice_thin<TRANS, FORM, 2>(a, q, w, vsrc, nsteps, cmax, ring, s_x, lane, dot);
                n0 = ok ? FORM : 0;
            }
        }
        if (n0 < a.k) {
            const WorkItem wc = w;   // copies: the call takes addresses, which would keep w and dot in memory
            double dc = dot;
            fma_columns<TRANS>(a, n0, wc, ring, lane, dc);
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

}  // namespace

size_t slice_smem_bytes() { return 4 * ((size_t)kSliceStages * 16 * kSliceTile + kSliceList); }

int slice_ldp(int64_t k) { return k <= kSliceThin ? (int)k : (int)((k + 7) / 8 * 8); }

using SliceKernel = void (*)(ProdArgs, SliceArgs);
template <bool TRANS>
static SliceKernel slice_kernel(int64_t k) {
    switch (k) {
        case 1: return slice_product_kernel<TRANS, 1>;
        case 2: return slice_product_kernel<TRANS, 2>;
        case 3: return slice_product_kernel<TRANS, 3>;
        default: return k <= 8 ? slice_product_kernel<TRANS, 8> : slice_product_kernel<TRANS, 0>;
    }
}

const void *slice_kernel_ptr(bool trans, int64_t k) {
    return (const void *)(trans ? slice_kernel<true>(k) : slice_kernel<false>(k));
}

cudaError_t launch_slice_product(bool trans, const ProdArgs &a, const SliceArgs &q, cudaStream_t s) {
    const size_t smem = slice_smem_bytes();
    const SliceKernel kern = trans ? slice_kernel<true>(a.k) : slice_kernel<false>(a.k);
    cudaError_t e = cudaFuncSetAttribute((const void *)kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<a.grid, 128, smem, s>>>(a, q);
    return cudaGetLastError();
}

cudaError_t launch_slice_panel(const SliceChunk *chunks, int64_t n_chunks, const double *X, int64_t ldx, int k, int ldp,
                               uint32_t *cmax, uint32_t *ccnt, uint64_t *out, cudaStream_t s) {
    if (n_chunks == 0) return cudaSuccess;
    // about 2048 elements a CTA: several chunks of narrow panels
    const int per = k >= 8 ? 1 : 8 / k;
    const unsigned grid = (unsigned)((n_chunks + per - 1) / per);
    slice_colmax_kernel<<<grid, 256, 0, s>>>(chunks, n_chunks, per, X, ldx, k, ldp, cmax);
    slice_panel_kernel<<<grid, 256, 0, s>>>(chunks, n_chunks, per, X, ldx, k, ldp, cmax, ccnt, out);
    return cudaGetLastError();
}

cudaError_t launch_slice_values(bool trans, const WorkItem *items, const SliceItem *sitems, int64_t n_items,
                                const AdjList &tl, const double *panel, uint8_t *dig, int32_t *rexp, cudaStream_t s) {
    if (n_items == 0) return cudaSuccess;
    const int warps = 4;
    const size_t smem = (size_t)warps * (32 * kSliceTile + (trans ? kSliceKMax * sizeof(int64_t) : 0));
    const void *kern = trans ? (const void *)slice_values_kernel<true> : (const void *)slice_values_kernel<false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int64_t need = (n_items + warps - 1) / warps;
    const int grid = (int)(need < 65535 ? need : 65535);
    if (trans) slice_values_kernel<true><<<grid, warps * 32, smem, s>>>(items, sitems, n_items, tl, panel, dig, rexp);
    else slice_values_kernel<false><<<grid, warps * 32, smem, s>>>(items, sitems, n_items, tl, panel, dig, rexp);
    return cudaGetLastError();
}

}  // namespace vbcsr
