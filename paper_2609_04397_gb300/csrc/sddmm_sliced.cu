// Sliced FP64 pattern-sampled product (sliced.cuh): D_ij = alpha A_i B_j^T + beta D_ij
// on the stored blocks, the contraction running over the k panel columns.
//
// Here every row of A and of B has a scale of its own (the contraction runs
// along the rows), so the operands keep 8 base-256 digits: one 64-bit word an
// element, 36 digit pairs in the levels 0 .. 7. What is dropped is about 2^-60
// of (row scale of A) x (row scale of B), which leaves room for rows whose
// large columns do not meet: an output is sliced as long as its leading
// digits' products reach kSddmmGuard.
//
// The FP64 multiply-adds it replaces bound the earlier kernel at every k (1.09
// ms for 3.8e7 entries at k = 16, 0.88 of the FP64 pipe).
#include "sliced.cuh"

namespace vbcsr {

namespace {

constexpr int kSdDigits = 8;
// Least sum of |leading digit| products of an output. In units of the last place (2^-63
// of a scale) a column's term is off by up to 2^62 (the rounding of an operand) and
// 2^64.8 (7 pairs of level 8 left out), and a one-step sum (k <= 16) by another 2^68 cut
// off in slice_value: 2^65.2 k + 2^68 together. An estimate G means sum |a b| of at least
// 0.248 G 2^112 (a leading digit d of a magnitude of (d - 0.502) 2^56 or more), and the
// error is within k 2^-53 of it, the bound of a k-term chain, from G = 296 + 2060 / k on:
// 640 at kSddmmMinCols. (At 16, sums of 18 columns were off by up to 160 2^-53. Rows of
// six normal entries reach 704 but for one output in 10^5.)
constexpr float kSddmmGuard = 704.f;

// Fixed-point rows of A (blockIdx.y = 0) and B (1): G lanes a row, kp columns
// (a multiple of 16; columns past k are zero). exps: scale exponent of a row,
// 0 when the row is zero, -1 when it is outside the sliced range.
__global__ void __launch_bounds__(256) slice_rows_kernel(int64_t rows_a, int64_t rows_b, int k, int kp, int G, const double *A,
                                                         int64_t lda, const double *B, int64_t ldb, uint64_t *fa,
                                                         uint64_t *fb, int32_t *ea, int32_t *eb) {
    const bool second = blockIdx.y != 0;
    const double *P = second ? B : A;
    const int64_t ld = second ? ldb : lda, rows = second ? rows_b : rows_a;
    uint64_t *out = second ? fb : fa;
    int32_t *ex = second ? eb : ea;
    const int per = blockDim.x / G, c0 = threadIdx.x % G;
    // a warp's rows end together: the loop bound is rounded up to whole blocks
    for (int64_t r0 = (int64_t)blockIdx.x * per; r0 < rows; r0 += (int64_t)gridDim.x * per) {
        const int64_t r = r0 + threadIdx.x / G;
        const bool in = r < rows;
        uint32_t m = 0;
        if (in)
            for (int c = c0; c < k; c += G) m = max(m, slice_mag(P[r * ld + c]));
        for (int h = G / 2; h > 0; h >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, h));
        const int E = slice_exp(m);
        const bool live = m != 0 && slice_exp_ok(m);
        if (!in) continue;
        if (c0 == 0) ex[r] = m == 0 ? 0 : (live ? E : -1);
        for (int c = c0; c < kp; c += G)
            out[r * kp + c] = slice_bytes<kSdDigits>(live && c < k ? P[r * ld + c] : 0.0, E);
    }
}

// The 16 virtual columns from t of an item by FP64 multiply-adds
__device__ __noinline__ void sddmm_columns(const SddmmArgs &a, const WorkItem &w, int tn, const int32_t *s_x,
                                           const int64_t *s_u, const int32_t *s_w, int t, int lane) {
    const double *A = static_cast<const double *>(a.A), *B = static_cast<const double *>(a.B);
    double *D = static_cast<double *>(a.D);
    for (int e = lane; e < 16 * w.B; e += 32) {
        const int p = e >> 4, v = t + (e & 15);
        if (v >= tn) continue;
        const double *ar = A + (w.yrow + p) * a.lda, *br = B + (int64_t)s_x[v] * a.ldb;
        double acc = 0.0;
        for (int64_t c = 0; c < a.k; ++c) acc = fma(a.alpha == 1.0 ? ar[c] : a.alpha * ar[c], br[c], acc);
        double *d = D + s_u[v] + (int64_t)p * s_w[v];
        *d = a.beta != 0.0 ? fma(a.beta, *d, acc) : acc;
    }
}

struct SdSliced {
    const uint64_t *fa, *fb;     // fixed-point rows, kp words each
    const int32_t *ea, *eb;      // their scale exponents
    int kp, alpha_one, beta_nz;
};

// One item of up to 8 NR rows, tiles of 16 virtual columns: the gathered rows of
// B are the M side of the MMA (16), the item's rows its N side (8 a tile, so an
// item of up to 8 rows computes one half), 16 panel columns per MMA. Operands are
// loaded as 64-bit words, four consecutive columns a lane (32 bytes), and cut
// into f16 digit pairs in registers. ONE (k <= 16): the digits of the item's rows
// stay in registers for the whole item. The rows of B are loaded one step ahead.
template <int NR, bool ONE>
__device__ __forceinline__ void sddmm_item_sliced(const SddmmArgs &a, const SdSliced &q, const WorkItem &w, int64_t r0,
                                                  int32_t *s_x, int64_t *s_u, int32_t *s_w, int lane) {
    const int g = lane >> 2, t4 = lane & 3, kp = q.kp, nck = kp >> 4;
    double *D = static_cast<double *>(a.D);
    auto load4 = [&](const uint64_t *p, uint2 (&v)[4]) {
        const uint4 x = __ldg(reinterpret_cast<const uint4 *>(p)), y = __ldg(reinterpret_cast<const uint4 *>(p) + 1);
        v[0] = make_uint2(x.x, x.y);
        v[1] = make_uint2(x.z, x.w);
        v[2] = make_uint2(y.x, y.y);
        v[3] = make_uint2(y.z, y.w);
    };
    uint32_t fR[NR][kSdDigits][2];
    auto load_rows = [&](int ck) {
#pragma unroll
        for (int n = 0; n < NR; ++n) {
            // a row past the item's last reads row 0: those outputs are not written
            const int p = 8 * n + g;
            uint2 v[4];
            load4(q.fa + (w.yrow + (p < w.B ? p : 0)) * kp + 16 * ck + 4 * t4, v);
            slice_pairs<kSdDigits>(v, fR[n]);
        }
    };
    // scale exponents of rows 8 n + 2 t4 + e (0 past the last)
    int er[NR][2];
#pragma unroll
    for (int n = 0; n < NR; ++n)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int p = 8 * n + 2 * t4 + e;
            er[n][e] = p < w.B ? q.ea[w.yrow + p] : 0;
        }
    if (ONE) load_rows(0);
    for (int t0 = 0; t0 < w.K; t0 += kKMax) {
        const int tn = min(kKMax, w.K - t0);
        __syncwarp();
        for (int e = lane; e < w.nlist; e += 32) {
            const int64_t l = w.lbegin + e;
            const int xr = a.fl_xrow[l], pc = a.fl_pcol[l], wd = a.fl_w[l];
            const int64_t u = a.fl_uoff[l] + r0 * wd;
            const int lo = max(pc, t0), hi = min(pc + wd, t0 + tn);
            for (int t = lo; t < hi; ++t) {
                s_x[t - t0] = xr + (t - pc);
                s_u[t - t0] = u + (t - pc);
                s_w[t - t0] = wd;
            }
        }
        __syncwarp();
        uint2 x[2][4];
        auto load_b = [&](int t, int ck) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int v = min(t + 8 * h + g, tn - 1);   // past the last column: not written
                load4(q.fb + (int64_t)s_x[v] * kp + 16 * ck + 4 * t4, x[h]);
            }
        };
        load_b(0, 0);
        for (int t = 0; t < tn; t += 16) {
            float acc[NR][kSliceLevels][4], low[NR][4];
#pragma unroll
            for (int n = 0; n < NR; ++n)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    low[n][j] = 0.f;
#pragma unroll
                    for (int L = 0; L < kSliceLevels; ++L) acc[n][L][j] = 0.f;
                }
            int flush = kSliceFlush;
            for (int ck = 0; ck < (ONE ? 1 : nck); ++ck) {
                if (!ONE) load_rows(ck);
                uint32_t b[2][kSdDigits][2];
#pragma unroll
                for (int h = 0; h < 2; ++h) slice_pairs<kSdDigits>(x[h], b[h]);
                if (!ONE && ck + 1 < nck) load_b(t, ck + 1);
                else if (t + 16 < tn) load_b(t + 16, 0);
#pragma unroll
                for (int i = 0; i < kSdDigits; ++i) {
                    uint32_t f[4] = {b[0][i][0], b[1][i][0], b[0][i][1], b[1][i][1]};
#pragma unroll
                    for (int j = 0; j < kSdDigits - i; ++j)
#pragma unroll
                        for (int n = 0; n < NR; ++n) mma_f16(acc[n][i + j], f, fR[n][j][0], fR[n][j][1]);
                    if (i == 0) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) f[j] &= 0x7fff7fffu;
#pragma unroll
                        for (int n = 0; n < NR; ++n)
                            mma_f16(low[n], f, fR[n][0][0] & 0x7fff7fffu, fR[n][0][1] & 0x7fff7fffu);
                    }
                }
                if (!ONE && --flush == 0) {
                    flush = kSliceFlush;
#pragma unroll
                    for (int n = 0; n < NR; ++n) slice_carry(acc[n]);
                }
            }
            // virtual columns t + g, t + 8 + g: a zero row of either side gives an exact zero
            // unless the other one is not finite
            int ev[2];
            bool ok = true;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int v = t + 8 * h + g;
                ev[h] = v < tn ? q.eb[s_x[v]] : 0;
                if (v < tn)
#pragma unroll
                    for (int n = 0; n < NR; ++n)
#pragma unroll
                        for (int e = 0; e < 2; ++e)
                            ok &= ev[h] >= 0 && er[n][e] >= 0 &&
                                  (ev[h] == 0 || er[n][e] == 0 || low[n][2 * h + e] >= kSddmmGuard);
            }
            if (!__all_sync(0xffffffffu, ok)) {
                sddmm_columns(a, w, tn, s_x, s_u, s_w, t, lane);
                continue;
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int v = t + 8 * h + g;
                if (v >= tn) continue;
                double *d = D + s_u[v];
                const int wd = s_w[v];
#pragma unroll
                for (int n = 0; n < NR; ++n)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int p = 8 * n + 2 * t4 + e;
                        if (p >= w.B) continue;
                        float lv[kSliceLevels];
#pragma unroll
                        for (int L = 0; L < kSliceLevels; ++L) lv[L] = acc[n][L][2 * h + e];
                        double o = slice_value<ONE>(lv, ev[h] + er[n][e] - 2114);
                        if (!q.alpha_one) o *= a.alpha;
                        double *dp = d + (int64_t)p * wd;
                        *dp = q.beta_nz ? fma(a.beta, *dp, o) : o;
                    }
            }
        }
    }
}

template <bool ONE>
__global__ void __launch_bounds__(128, 3) slice_sddmm_kernel(SddmmArgs a, SdSliced q) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int64_t *s_u = reinterpret_cast<int64_t *>(smem_raw) + (size_t)warp * kKMax;
    int32_t *s_x = reinterpret_cast<int32_t *>(smem_raw + 4 * kKMax * sizeof(int64_t)) + (size_t)warp * 2 * kKMax;
    for (;;) {
        unsigned long long t = 0;
        if (lane == 0) t = atomicAdd(reinterpret_cast<unsigned long long *>(a.queue), 1ull);
        const int64_t it = (int64_t)__shfl_sync(0xffffffffu, t, 0);
        if (it >= a.n_items) break;
        const WorkItem w = a.items[it];
        if (w.nlist == 0) continue;
        const int64_t r0 = (w.vbase - a.fl_pbase[w.lbegin]) / w.Kp;   // first row inside the block row
        if (w.B <= 8) sddmm_item_sliced<1, ONE>(a, q, w, r0, s_x, s_u, s_x + kKMax, lane);
        else sddmm_item_sliced<2, ONE>(a, q, w, r0, s_x, s_u, s_x + kKMax, lane);
    }
}

}  // namespace

cudaError_t launch_sddmm_sliced(const SddmmArgs &a, int64_t rows_a, int64_t rows_b, uint64_t *fa, uint64_t *fb, int32_t *ea,
                                int32_t *eb, cudaStream_t s) {
    if (a.n_items == 0) return cudaSuccess;
    const int k = (int)a.k, kp = (k + 15) / 16 * 16;
    int G = 1;
    while (G < k && G < 32) G <<= 1;
    const int64_t per = 256 / G, most = rows_a > rows_b ? rows_a : rows_b;
    const int64_t need = (most + per - 1) / per;
    slice_rows_kernel<<<dim3((unsigned)(need < 16384 ? need : 16384), 2), 256, 0, s>>>(
        rows_a, rows_b, k, kp, G, (const double *)a.A, a.lda, (const double *)a.B, a.ldb, fa, fb, ea, eb);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const size_t smem = 4 * kKMax * (sizeof(int64_t) + 2 * sizeof(int32_t));
    const bool one = kp == 16;
    const void *kern = one ? (const void *)slice_sddmm_kernel<true> : (const void *)slice_sddmm_kernel<false>;
    const SdSliced q = {fa, fb, ea, eb, kp, a.alpha == 1.0, a.beta != 0.0};
    const int cap = max_resident_ctas(kern, 128, smem);
    if (cap < 0) return cudaGetLastError();
    if ((e = cudaMemsetAsync(a.queue, 0, sizeof(long long), s)) != cudaSuccess) return e;
    const int64_t ctas = (a.n_items + 3) / 4;
    const int grid = (int)(ctas < cap ? ctas : cap);
    if (one) slice_sddmm_kernel<true><<<grid, 128, smem, s>>>(a, q);
    else slice_sddmm_kernel<false><<<grid, 128, smem, s>>>(a, q);
    return cudaGetLastError();
}

}  // namespace vbcsr
