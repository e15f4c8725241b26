// Sliced FP64 products (sliced.cuh): the digit copies of the values and of X,
// and the tensor-core product kernel of an FP64 operator, forward and adjoint.
#include "sliced_kernel.cuh"

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

// CPLX: X holds (re, im) pairs as two columns, which share a scale
template <bool CPLX>
__global__ void __launch_bounds__(256) slice_colmax_kernel(const SliceChunk *chunks, int64_t n_chunks, int per,
                                                           const double *__restrict__ X, int64_t ldx, int k, int ldp,
                                                           uint32_t *cmax, uint32_t *cown) {
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
            if (w.ty == 0 && col < k && red[w.tx]) {
                atomicMax(cmax + (int64_t)c.strct * ldp + col, red[w.tx]);
                if (CPLX) {
                    atomicMax(cmax + (int64_t)c.strct * ldp + (col ^ 1), red[w.tx]);
                    cown[(int64_t)c.strct * ldp + col] = 1;   // a part that is not all zero
                }
            }
            m = 0;
        });
    }
}

// X as biased fixed point [rows, ldp] (8 bytes an element, 7 of them digits);
// columns k .. ldp - 1 are zero. ccnt counts the elements below 2^-kSliceTiny
// of their column's maximum (CPLX: of which both parts are: a real panel's zero imaginary
// parts are not resolved worse for it). CPLX: two rows for a row of X, x = (re, im) and
// i x = (-im, re).
template <bool CPLX>
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
                uint64_t *o = out + (int64_t)c.row0 * ldp * (CPLX ? 2 : 1) + col;
#pragma unroll 4
                for (int r = w.ty; r < c.nrows; r += w.TY) {
                    const double v = live ? x[(int64_t)r * ldx] : 0.0;
                    uint32_t mag = slice_mag(v);
                    if (CPLX) {
                        // i x: -im in the real column, re in the imaginary one (the neighbour's value)
                        o[2 * (int64_t)r * ldp] = slice_bytes(v, E);
                        const double u = live ? x[(int64_t)r * ldx + (col & 1 ? -1 : 1)] : 0.0;
                        mag = max(mag, slice_mag(u));
                        o[(2 * (int64_t)r + 1) * ldp] = slice_bytes(col & 1 ? u : -u, E);
                    } else {
                        o[(int64_t)r * ldp] = slice_bytes(v, E);
                    }
                    tiny += live && (mag >> 20) + kSliceTiny < (M >> 20);
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
// blocks, with BP = 2, 4, 8 or 16 lanes along the item's rows (consecutive in
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
template <int BP, bool CPLX>
__device__ __forceinline__ void adj_columns(const double *panel, const int64_t *s_a, const WorkItem &w, int t0, int lane,
                                            double (&v)[BP]) {
    const int q = lane % BP;
#pragma unroll
    for (int u = 0; u < BP; ++u) {
        const int t = t0 + u * (32 / BP) + lane / BP;
        if (CPLX)   // (re, -im) of the conjugate are two virtual columns
            v[u] = t < 2 * w.K && q < w.B ? (t & 1 ? -1.0 : 1.0) * panel[2 * (s_a[t >> 1] + q) + (t & 1)] : 0.0;
        else
            v[u] = t < w.K && q < w.B ? panel[s_a[t] + q] : 0.0;
    }
}

template <int BP, bool CPLX>
__device__ __forceinline__ void adj_item_digits(const double *panel, const int64_t *s_a, const WorkItem &w, uint8_t *dst,
                                                uint8_t *stage, int32_t *rexp, int32_t *rparts, int lane) {
    const int K = CPLX ? 2 * w.K : w.K;
    uint32_t m = 0;
    for (int t0 = 0; t0 < K; t0 += 32) {
        double v[BP];
        adj_columns<BP, CPLX>(panel, s_a, w, t0, lane, v);
#pragma unroll
        for (int u = 0; u < BP; ++u) m = max(m, slice_mag(v[u]));
    }
#pragma unroll
    for (int h = 2 * BP; h < 32; h <<= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, h));
    // lanes BP apart hold neighbouring virtual columns (CPLX: the two parts of a value)
    const uint32_t other = __shfl_xor_sync(0xffffffffu, m, BP);
    if (CPLX && lane < w.B) rparts[w.yrow + lane] = (m != 0) | (other != 0) << 1;
    m = max(m, other);
    const int E = m == 0 ? 0 : (slice_exp_ok(m) ? slice_exp(m) : -1), q = lane % BP;
    if (lane < w.B) rexp[w.yrow + lane] = E;
    const int nt = (K + 15) >> 4;
    for (int c = 0; c < nt; c += 2) {
        double v[BP];
        adj_columns<BP, CPLX>(panel, s_a, w, 16 * c, lane, v);
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

// CPLX: a complex value is two virtual columns, (re, im) forward (as they lie in
// the pages) and (re, -im) adjoint
template <bool TRANS, bool CPLX>
__global__ void __launch_bounds__(128) slice_values_kernel(const WorkItem *items, const SliceItem *sitems,
                                                           int64_t n_items, AdjList tl, const double *panel,
                                                           uint8_t *dig, int32_t *rexp, int32_t *rparts) {
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
            if (w.B > 8) adj_item_digits<16, CPLX>(panel, s_a, w, dst, stage, rexp, rparts, lane);
            else if (w.B > 4) adj_item_digits<8, CPLX>(panel, s_a, w, dst, stage, rexp, rparts, lane);
            else if (w.B > 2) adj_item_digits<4, CPLX>(panel, s_a, w, dst, stage, rexp, rparts, lane);
            else adj_item_digits<2, CPLX>(panel, s_a, w, dst, stage, rexp, rparts, lane);
        } else {
            constexpr int cw = CPLX ? 2 : 1;
            const int K = cw * w.K;
            const double *src = panel + cw * w.vbase;
            auto load = [&](int t, double (&v)[16]) {               // column t of the item, all rows at once
                const bool in = t < K;
                const double *c = src + (in ? t : 0);
#pragma unroll
                for (int p = 0; p < 16; ++p) v[p] = in && p < w.B ? c[(int64_t)p * cw * w.Kp] : 0.0;
            };
            uint32_t m[16];
#pragma unroll
            for (int p = 0; p < 16; ++p) m[p] = 0;
            for (int t = lane; t < K; t += 32) {
                double v[16];
                load(t, v);
#pragma unroll
                for (int p = 0; p < 16; ++p) m[p] = max(m[p], slice_mag(v[p]));
            }
#pragma unroll
            for (int p = 0; p < 16; ++p) {
                const uint32_t r = __reduce_max_sync(0xffffffffu, m[p]);
                if (CPLX) {   // even lanes hold the real parts
                    const unsigned any = __ballot_sync(0xffffffffu, m[p] != 0);
                    if (lane == p && p < w.B)
                        rparts[w.yrow + p] = ((any & 0x55555555u) != 0) | ((any & 0xaaaaaaaau) != 0) << 1;
                }
                const int e = r == 0 ? 0 : (slice_exp_ok(r) ? slice_exp(r) : -1);
                if (lane == p) {
                    s_e[warp][p] = e;
                    if (p < w.B) rexp[w.yrow + p] = e;
                }
            }
            __syncwarp();
            const int nt = (K + 15) >> 4;
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

}  // namespace

int slice_ldp(int64_t k) { return (int)((k + 7) / 8 * 8); }

size_t slice_smem_bytes() { return kSliceSmem; }

const void *slice_kernel_ptr(bool trans, int64_t k) { return slice_kernel_of<double, double>(trans, k); }

cudaError_t launch_slice_product(bool trans, const ProdArgs &a, const SliceArgs &q, cudaStream_t s) {
    return launch_slice<double, double>(trans, a, q, s);
}

cudaError_t launch_slice_panel(bool cplx, const SliceChunk *chunks, int64_t n_chunks, const double *X, int64_t ldx, int k,
                               int ldp, uint32_t *cmax, uint32_t *ccnt, uint32_t *cown, uint64_t *out, cudaStream_t s) {
    if (n_chunks == 0) return cudaSuccess;
    // about 2048 elements a CTA: several chunks of narrow panels
    const int per = k >= 8 ? 1 : 8 / k;
    const unsigned grid = (unsigned)((n_chunks + per - 1) / per);
    if (cplx) {
        slice_colmax_kernel<true><<<grid, 256, 0, s>>>(chunks, n_chunks, per, X, ldx, k, ldp, cmax, cown);
        slice_panel_kernel<true><<<grid, 256, 0, s>>>(chunks, n_chunks, per, X, ldx, k, ldp, cmax, ccnt, out);
    } else {
        slice_colmax_kernel<false><<<grid, 256, 0, s>>>(chunks, n_chunks, per, X, ldx, k, ldp, cmax, cown);
        slice_panel_kernel<false><<<grid, 256, 0, s>>>(chunks, n_chunks, per, X, ldx, k, ldp, cmax, ccnt, out);
    }
    return cudaGetLastError();
}

template <bool TRANS, bool CPLX>
static cudaError_t values_launch(const WorkItem *items, const SliceItem *sitems, int64_t n_items, const AdjList &tl,
                                 const double *panel, uint8_t *dig, int32_t *rexp, int32_t *rparts, cudaStream_t s) {
    const int warps = 4;
    const size_t smem = (size_t)warps * (32 * kSliceTile + (TRANS ? kSliceKMax * sizeof(int64_t) : 0));
    cudaError_t e = cudaFuncSetAttribute((const void *)slice_values_kernel<TRANS, CPLX>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int64_t need = (n_items + warps - 1) / warps;
    slice_values_kernel<TRANS, CPLX><<<(unsigned)(need < 65535 ? need : 65535), warps * 32, smem, s>>>(
        items, sitems, n_items, tl, panel, dig, rexp, rparts);
    return cudaGetLastError();
}

cudaError_t launch_slice_values(bool cplx, bool trans, const WorkItem *items, const SliceItem *sitems, int64_t n_items,
                                const AdjList &tl, const double *panel, uint8_t *dig, int32_t *rexp, int32_t *rparts,
                                cudaStream_t s) {
    if (n_items == 0) return cudaSuccess;
    if (cplx)
        return trans ? values_launch<true, true>(items, sitems, n_items, tl, panel, dig, rexp, rparts, s)
                     : values_launch<false, true>(items, sitems, n_items, tl, panel, dig, rexp, rparts, s);
    return trans ? values_launch<true, false>(items, sitems, n_items, tl, panel, dig, rexp, rparts, s)
                 : values_launch<false, false>(items, sitems, n_items, tl, panel, dig, rexp, rparts, s);
}

}  // namespace vbcsr
