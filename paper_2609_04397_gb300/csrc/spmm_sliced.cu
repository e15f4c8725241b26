// Sliced FP64 products (sliced.cuh): the digit copies of the values and of X,
// and the tensor-core product kernel of an FP64 operator, forward and adjoint.
#include "fma_kernel.cuh"
#include "sliced.cuh"

namespace vbcsr {

namespace {

// ---------------------------------------------------------------------------
// X: column maxima per structure, then the digits

// One CTA per chunk of X rows (rows of one structure); thread tx of TX takes
// columns tx, tx + TX, ..., threads ty stride the rows.
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

__global__ void __launch_bounds__(256) slice_colmax_kernel(const SliceChunk *chunks, int64_t n_chunks, const double *X,
                                                           int64_t ldx, int k, int ldp, uint32_t *cmax) {
    __shared__ uint32_t red[256];
    const ColWalk w(k);
    for (int64_t q = blockIdx.x; q < n_chunks; q += gridDim.x) {
        const SliceChunk c = chunks[q];
        for (int c0 = 0; c0 < k; c0 += w.TX) {
            const int col = c0 + w.tx;
            uint32_t m = 0;
            if (col < k)
                for (int r = w.ty; r < c.nrows; r += w.TY) m = max(m, slice_mag(X[(int64_t)(c.row0 + r) * ldx + col]));
            __syncthreads();
            red[threadIdx.x] = m;
            __syncthreads();
            for (int h = w.TY / 2; h > 0; h >>= 1) {
                if (w.ty < h) red[threadIdx.x] = max(red[threadIdx.x], red[threadIdx.x + h * w.TX]);
                __syncthreads();
            }
            if (w.ty == 0 && col < k && red[w.tx]) atomicMax(cmax + (int64_t)c.strct * ldp + col, red[w.tx]);
        }
    }
}

// X as biased fixed point [rows, ldp] (8 bytes an element, 7 of them digits);
// columns k .. ldp - 1 are zero. ccnt counts the elements below 2^-10 of their
// column's maximum.
__global__ void __launch_bounds__(256) slice_panel_kernel(const SliceChunk *chunks, int64_t n_chunks, const double *X,
                                                          int64_t ldx, int k, int ldp, const uint32_t *cmax,
                                                          uint32_t *ccnt, uint64_t *out) {
    __shared__ uint32_t red[256];
    const ColWalk w(ldp);
    for (int64_t q = blockIdx.x; q < n_chunks; q += gridDim.x) {
        const SliceChunk c = chunks[q];
        for (int c0 = 0; c0 < ldp; c0 += w.TX) {
            const int col = c0 + w.tx;
            uint32_t tiny = 0;
            if (col < ldp) {
                const uint32_t M = col < k ? cmax[(int64_t)c.strct * ldp + col] : 0u;
                const bool live = M != 0 && slice_exp_ok(M);
                const int E = slice_exp(M);
                for (int r = w.ty; r < c.nrows; r += w.TY) {
                    const double x = live ? X[(int64_t)(c.row0 + r) * ldx + col] : 0.0;
                    tiny += (slice_mag(x) >> 20) + 10 < (M >> 20);
                    out[(int64_t)(c.row0 + r) * ldp + col] = slice_bytes(x, E);
                }
                if (!live) tiny = 0;
            }
            __syncthreads();
            red[threadIdx.x] = tiny;
            __syncthreads();
            for (int h = w.TY / 2; h > 0; h >>= 1) {
                if (w.ty < h) red[threadIdx.x] += red[threadIdx.x + h * w.TX];
                __syncthreads();
            }
            if (w.ty == 0 && col < k && red[w.tx]) atomicAdd(ccnt + (int64_t)c.strct * ldp + col, red[w.tx]);
        }
    }
}

// ---------------------------------------------------------------------------
// values: one warp per work item; row maxima, then 16-column tiles of digits
// [tile][digit][row][16 columns], two tiles at a time staged in shared memory
// and stored 16 bytes a lane

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
        if (TRANS) {
            __syncwarp();
            for (int e = lane; e < w.nlist; e += 32) {
                const int64_t l = w.lbegin + e;
                const int64_t pb = tl.pbase[l];
                const int kp = tl.kp[l], bi = tl.bi[l], vc = tl.vcol[l];
                for (int p = 0; p < bi; ++p) s_a[vc + p] = pb + (int64_t)p * kp + w.Kp;
            }
            __syncwarp();
        }
        const double *src = TRANS ? panel : panel + w.vbase;
        const int64_t ps = TRANS ? 1 : w.Kp;                    // from a row to the next
        auto load = [&](int t, double (&v)[16]) {               // column t of the item, all rows at once
            const bool in = t < w.K;
            const double *c = src + (in ? (TRANS ? s_a[t] : t) : 0);
#pragma unroll
            for (int p = 0; p < 16; ++p) v[p] = in && p < w.B ? c[p * ps] : 0.0;
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
            uint8_t *o = stage + (lane >> 4) * w.B * kSliceTile + (lane & 15);
#pragma unroll
            for (int p = 0; p < 16; ++p) {
                if (p >= w.B) break;
                const int E = s_e[warp][p];
                const uint64_t u = slice_bytes(E > 0 ? v[p] : 0.0, E);
#pragma unroll
                for (int i = 0; i < kSliceDigits; ++i) o[(i * w.B + p) * 16] = (uint8_t)(u >> (8 * (6 - i)));
            }
            __syncwarp();
            uint4 *dst = reinterpret_cast<uint4 *>(dig + si.doff + (int64_t)c * w.B * kSliceTile);
            const int n = min(2, nt - c) * w.B * (kSliceTile / 16);
            for (int q = lane; q < n; q += 32) dst[q] = reinterpret_cast<uint4 *>(stage)[q];
            __syncwarp();
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

// One warp per work item (up to 16 output rows); KWIDE: k > 8, passes of 16
// columns with a last one of 8 where that is enough.
template <bool TRANS, bool KWIDE>
__global__ void __launch_bounds__(128, KWIDE ? 3 : 4) slice_product_kernel(ProdArgs a, SliceArgs q) {
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
            bool p = q.struct_nnz[si.strct] * a.k < kSliceMinWork;
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
            if (KWIDE)
                for (; ok && n0 + 8 < a.k; n0 += ok ? 16 : 0)
                    ok = w.B <= 8 ? slice_pass<TRANS, true, 1>(a, q, w, vsrc, nsteps, n0, cmax, ring, s_x, lane, dot)
                                  : slice_pass<TRANS, true, 2>(a, q, w, vsrc, nsteps, n0, cmax, ring, s_x, lane, dot);
            if (ok && n0 < a.k) {
                ok = w.B <= 8 ? slice_pass<TRANS, false, 1>(a, q, w, vsrc, nsteps, n0, cmax, ring, s_x, lane, dot)
                              : slice_pass<TRANS, false, 2>(a, q, w, vsrc, nsteps, n0, cmax, ring, s_x, lane, dot);
                n0 += ok ? 8 : 0;
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

const void *slice_kernel_ptr(bool trans, int64_t k) {
    if (trans) return k <= 8 ? (const void *)slice_product_kernel<true, false> : (const void *)slice_product_kernel<true, true>;
    return k <= 8 ? (const void *)slice_product_kernel<false, false> : (const void *)slice_product_kernel<false, true>;
}

cudaError_t launch_slice_product(bool trans, const ProdArgs &a, const SliceArgs &q, cudaStream_t s) {
    const size_t smem = slice_smem_bytes();
    const void *kern = slice_kernel_ptr(trans, a.k);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (trans) {
        if (a.k <= 8) slice_product_kernel<true, false><<<a.grid, 128, smem, s>>>(a, q);
        else slice_product_kernel<true, true><<<a.grid, 128, smem, s>>>(a, q);
    } else {
        if (a.k <= 8) slice_product_kernel<false, false><<<a.grid, 128, smem, s>>>(a, q);
        else slice_product_kernel<false, true><<<a.grid, 128, smem, s>>>(a, q);
    }
    return cudaGetLastError();
}

cudaError_t launch_slice_panel(const SliceChunk *chunks, int64_t n_chunks, const double *X, int64_t ldx, int k, int ldp,
                               uint32_t *cmax, uint32_t *ccnt, uint64_t *out, cudaStream_t s) {
    if (n_chunks == 0) return cudaSuccess;
    const int grid = (int)(n_chunks < 65535 ? n_chunks : 65535);
    slice_colmax_kernel<<<grid, 256, 0, s>>>(chunks, n_chunks, X, ldx, k, ldp, cmax);
    slice_panel_kernel<<<grid, 256, 0, s>>>(chunks, n_chunks, X, ldx, k, ldp, cmax, ccnt, out);
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
