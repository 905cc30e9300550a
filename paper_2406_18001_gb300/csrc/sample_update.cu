// sample_update.cu -- the small kernels of one outer s-step: index sampling
// (Algorithms 2 and 4, "choose i uniformly at random"), operand packing and
// norms, the scatter update of alpha and the cached gradient, and the
// convergence reductions (Section 5.1's duality gap and residual).
#include "dcd_internal.cuh"

#include <cuda_fp16.h>

namespace dcd {

// ----------------------------------------------------------- sampling -----
// DCD: one thread per iteration.  out[j] = floor(u * m / 2^64), u the
// SplitMix64 draw (seed, stream 0, counter first + j).
__global__ void sample_dcd_kernel(uint64_t seed, const uint64_t *ctr_dev, uint64_t first_host, int64_t m,
                                  int64_t count, int32_t *out, uint64_t *ctr_next)
{
    uint64_t first = (ctr_dev ? *ctr_dev : 0) + first_host;
    if (ctr_next && blockIdx.x == 0 && threadIdx.x == 0) *ctr_next = first + (uint64_t)count;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < count; j += (int64_t)gridDim.x * blockDim.x)
        out[j] = (int32_t)below(sm64_draw(seed, 0, first + (uint64_t)j), (uint64_t)m);
}

// BDCD: one warp per block.  Floyd's algorithm (Bentley & Floyd 1987): for
// q = 0..b-1, J = m-b+q, r uniform in [0, J] from draw (seed, t+1, q); take r
// unless it was already taken, else take J.  The warp tests membership of r
// against the q indices taken so far in parallel.
__global__ void sample_bdcd_kernel(uint64_t seed, const uint64_t *ctr_dev, uint64_t first_host, int64_t m,
                                   int b, int64_t nblocks, int32_t *out, uint64_t *ctr_next)
{
    extern __shared__ int32_t sblk[];  // b indices per warp
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (warp >= nblocks) return;
    const uint64_t t0 = (ctr_dev ? *ctr_dev : 0) + first_host;
    if (ctr_next && warp == 0 && lane == 0) *ctr_next = t0 + (uint64_t)nblocks;
    const uint64_t t = t0 + (uint64_t)warp;
    int32_t *blk = sblk + (threadIdx.x >> 5) * b;
    for (int q = 0; q < b; ++q) {
        const int64_t J = m - b + q;
        const int64_t r = (int64_t)below(sm64_draw(seed, t + 1, (uint64_t)q), (uint64_t)(J + 1));
        bool hit = false;
        for (int p = lane; p < q; p += 32) hit |= (blk[p] == (int32_t)r);
        const unsigned any = __ballot_sync(0xffffffffu, hit);
        if (lane == 0) blk[q] = (int32_t)(any ? J : r);
        __syncwarp();
    }
    for (int q = lane; q < b; q += 32) out[warp * b + q] = blk[q];
}

cudaError_t launch_sample(int method, uint64_t seed, const uint64_t *ctr_dev, uint64_t first_host, int64_t m,
                          int b, int64_t count, int32_t *out, int *err, cudaStream_t st, uint64_t *ctr_next)
{
    (void)err;
    if (count <= 0) return cudaSuccess;
    if (method == 0) {
        int threads = 128;
        int64_t blocks = (count + threads - 1) / threads;
        if (blocks > 4096) blocks = 4096;
        sample_dcd_kernel<<<(unsigned)blocks, threads, 0, st>>>(seed, ctr_dev, first_host, m, count, out, ctr_next);
    } else {
        int threads = 128;  // 4 warps = 4 blocks per CTA
        int64_t blocks = (count * 32 + threads - 1) / threads;
        sample_bdcd_kernel<<<(unsigned)blocks, threads, sizeof(int32_t) * 4 * b, st>>>(seed, ctr_dev, first_host, m,
                                                                                       b, count, out, ctr_next);
    }
    return cudaGetLastError();
}

// ------------------------------------------------------------ packing -----
// Nearest e4m3 code of x (ties to even), saturating at +-448.
__device__ __forceinline__ uint32_t e4m3_code(float x)
{
    uint16_t pair;
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(pair) : "f"(0.f), "f"(x));  // x -> low byte
    return pair & 0xFFu;
}

// Element `off` of a dense source as FP32; an FP8 source is scale * value(q)
// rounded once.
__device__ __forceinline__ float load_as_f32(const void *src, int dtype, int64_t off, float scale = 0.f)
{
    switch (dtype) {
    case DCD_F64: return (float)((const double *)src)[off];
    case DCD_F32: return ((const float *)src)[off];
    case DCD_BF16: return __bfloat162float(((const __nv_bfloat16 *)src)[off]);
    case DCD_FP8E4M3: return (float)((double)scale * (double)e4m3_value(((const uint8_t *)src)[off]));
    default: return 0.f;
    }
}

// dst row r (n_pad doubles, zero padded) = src row rows[r] (or r) in FP64; an FP8 source is
// dequantised with its row scales (exactly).  Row indices outside [0, m) produce a zero row and
// set DEV_BAD_INDEX.
__global__ void pack_rows_kernel(const void *src, int dtype, int64_t ld, int64_t m, int64_t n, const int32_t *rows,
                                 double *dst, int64_t n_pad, int64_t count, int *err, const float *src_scale)
{
    const int64_t total = count * n_pad;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = e / n_pad, c = e - r * n_pad;
        const int64_t sr = rows ? (int64_t)rows[r] : r;
        const bool inb = sr >= 0 && sr < m;
        if (!inb && c == 0) set_error(err, DEV_BAD_INDEX);
        const float rsc = (dtype == DCD_FP8E4M3 && inb) ? src_scale[sr] : 0.f;
        double v = 0.0;
        if (c < n && inb)
            v = (dtype == DCD_F64)       ? ((const double *)src)[sr * ld + c]
                : (dtype == DCD_FP8E4M3) ? (double)rsc * (double)e4m3_value(((const uint8_t *)src)[sr * ld + c])
                                         : (double)load_as_f32(src, dtype, sr * ld + c);
        dst[e] = v;
    }
}

cudaError_t launch_pack_rows(const void *src, int dtype, int64_t ld, int64_t m, int64_t n, const int32_t *rows,
                             double *dst, int64_t n_pad, int64_t count, int *err, cudaStream_t st,
                             const float *src_scale)
{
    if (dtype == DCD_FP8E4M3 && !src_scale) return cudaErrorInvalidValue;
    if (count <= 0) return cudaSuccess;
    int64_t total = count * n_pad;
    int64_t blocks = (total + 255) / 256;
    if (blocks > 152 * 32) blocks = 152 * 32;
    pack_rows_kernel<<<(unsigned)blocks, 256, 0, st>>>(src, dtype, ld, m, n, rows, dst, n_pad, count, err, src_scale);
    return cudaGetLastError();
}

// Per-row FP8 storage (one warp per row): the row is rounded to FP32,
// scale = fl32(max|a| / 448), code = e4m3(fl32(a / scale)) with IEEE FP32
// division; a row of zeros gets scale 0 and zero codes.  An FP8 source is
// copied with its scale.  Columns n..ldq-1 of the destination are zero.
// ------------------------------------------------ literal-order step --
// The paper's printed order (Algorithms 2 and 4) keeps the m x sb block U_k /
// Q_k in memory and forms U_j^T alpha_sk from it.  literal_partial_kernel:
// block b sums rows [b R, (b+1) R) of (y_i) Q[i][c] alpha_i for every column
// c (consecutive threads read consecutive columns of a row), in row order.
template <typename QT>
__global__ void literal_partial_kernel(const QT *Q, int64_t ldq, int64_t m, int64_t ncols, const double *alpha,
                                       const double *y, int64_t rows_per_block, double *partials)
{
    const int64_t r0 = blockIdx.x * rows_per_block, r1 = min(m, r0 + rows_per_block);
    for (int64_t c = threadIdx.x; c < ncols; c += blockDim.x) {
        double acc = 0.0;
        for (int64_t i = r0; i < r1; ++i) {
            const double a = y ? y[i] * alpha[i] : alpha[i];
            acc = fma((double)Q[i * ldq + c], a, acc);
        }
        partials[blockIdx.x * ncols + c] = acc;
    }
}

// u_p = sum of the partials in block order, then the gradient value of the
// step's coordinate i = S[p] written at position i of a full-length array g
// (repeats write the same value):
//   K-SVM: g_i = y_i u_p - 1 + omega alpha_i        (u = U_k^T alpha)
//   K-RR:  g_i = u_p / lambda + m alpha_i - y_i
__global__ void literal_grad_kernel(const double *partials, int64_t nblk, int64_t ncols, const int32_t *S,
                                    int problem, const double *y, const double *alpha, double inv_lambda,
                                    double diag, double *g)
{
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= ncols) return;
    double u = 0.0;
    for (int64_t b = 0; b < nblk; ++b) u += partials[b * ncols + p];
    const int32_t i = S[p];
    g[i] = problem == 0 ? fma(y[i], u, -1.0) + diag * alpha[i] : u * inv_lambda + diag * alpha[i] - y[i];
}

// G_k = V_k^T U_k: row r of the Gram is row S[r] of the stored block
template <typename QT>
__global__ void literal_gram_kernel(const QT *Q, int64_t ldq, const int32_t *S, int64_t ncols, QT *Kss,
                                    int64_t ldk)
{
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= ncols * ncols) return;
    const int64_t r = e / ncols, c = e - r * ncols;
    Kss[r * ldk + c] = Q[(int64_t)S[r] * ldq + c];
}

cudaError_t launch_literal_terms(const void *Q, int q_f64, int64_t ldq, int64_t m, int64_t ncols, const int32_t *S,
                                 int problem, const double *y, const double *alpha, double inv_lambda, double diag,
                                 double *partials, int64_t max_blocks, double *g, void *Kss, int64_t ldk,
                                 cudaStream_t st)
{
    if (ncols <= 0) return cudaSuccess;
    int64_t nblk = max_blocks < 1 ? 1 : max_blocks;
    const int64_t rpb = (m + nblk - 1) / nblk;
    nblk = (m + rpb - 1) / rpb;
    const int thr = ncols >= 256 ? 256 : (int)((ncols + 31) / 32 * 32);
    const double *ys = problem == 0 ? y : nullptr;
    if (q_f64)
        literal_partial_kernel<double><<<(unsigned)nblk, thr, 0, st>>>((const double *)Q, ldq, m, ncols, alpha, ys,
                                                                     rpb, partials);
    else
        literal_partial_kernel<float><<<(unsigned)nblk, thr, 0, st>>>((const float *)Q, ldq, m, ncols, alpha, ys, rpb,
                                                                    partials);
    literal_grad_kernel<<<(unsigned)((ncols + 255) / 256), 256, 0, st>>>(partials, nblk, ncols, S, problem, y, alpha,
                                                                       inv_lambda, diag, g);
    const unsigned gb = (unsigned)((ncols * ncols + 255) / 256);
    if (q_f64)
        literal_gram_kernel<double><<<gb, 256, 0, st>>>((const double *)Q, ldq, S, ncols, (double *)Kss, ldk);
    else
        literal_gram_kernel<float><<<gb, 256, 0, st>>>((const float *)Q, ldq, S, ncols, (float *)Kss, ldk);
    return cudaGetLastError();
}

__global__ void quantize_rows_kernel(const void *src, int dtype, int64_t ld, int64_t m, int64_t n,
                                     const int32_t *rows, const float *src_scale, uint8_t *dst, int64_t ldq,
                                     float *dst_scale, int64_t count, int *err)
{
    const int lane = threadIdx.x & 31;
    const int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (r >= count) return;
    const int64_t sr = rows ? (int64_t)rows[r] : r;
    uint8_t *d = dst + r * ldq;
    if (sr < 0 || sr >= m) {
        if (lane == 0) {
            set_error(err, DEV_BAD_INDEX);
            dst_scale[r] = 0.f;
        }
        for (int64_t c = lane; c < ldq; c += 32) d[c] = 0;
        return;
    }
    bool bad = false;
    float scale;
    if (dtype == DCD_FP8E4M3) {
        const uint8_t *s = (const uint8_t *)src + sr * ld;
        for (int64_t c = lane; c < ldq; c += 32) {
            const uint8_t v = c < n ? s[c] : 0;
            bad |= (v & 0x7F) == 0x7F;
            d[c] = v;
        }
        scale = src_scale[sr];
        bad |= !(scale >= 0.f && scale <= 3.4028234e38f);
    } else {
        float amax = 0.f;
        for (int64_t c = lane; c < n; c += 32) {
            const float v = load_as_f32(src, dtype, sr * ld + c);
            bad |= !(fabsf(v) <= 3.4028234e38f);
            amax = fmaxf(amax, fabsf(v));
        }
        for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
        scale = __fdiv_rn(amax, 448.f);
        for (int64_t c = lane; c < ldq; c += 32) {
            uint32_t code = 0;
            if (c < n && scale > 0.f) code = e4m3_code(__fdiv_rn(load_as_f32(src, dtype, sr * ld + c), scale));
            d[c] = (uint8_t)code;
        }
    }
    if (__any_sync(0xffffffffu, bad) && lane == 0) set_error(err, DEV_BAD_VALUE);
    if (lane == 0) dst_scale[r] = scale;
}

cudaError_t launch_quantize_rows(const void *src, int dtype, int64_t ld, int64_t m, int64_t n, const int32_t *rows,
                                 const float *src_scale, uint8_t *dst, int64_t ldq, float *dst_scale, int64_t count,
                                 int *err, cudaStream_t st)
{
    if (count <= 0) return cudaSuccess;
    if (ldq < n || (dtype == DCD_FP8E4M3 && !src_scale)) return cudaErrorInvalidValue;
    const int64_t blocks = (count * 32 + 255) / 256;
    quantize_rows_kernel<<<(unsigned)blocks, 256, 0, st>>>(src, dtype, ld, m, n, rows, src_scale, dst, ldq, dst_scale,
                                                           count, err);
    return cudaGetLastError();
}

// Number of labels that are not exactly +1 or -1.
__global__ void label_check_kernel(const double *y, int64_t m, int *bad)
{
    int local = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x)
        local += !(y[i] == 1.0 || y[i] == -1.0);
    for (int o = 16; o > 0; o >>= 1) local += __shfl_xor_sync(0xffffffffu, local, o);
    if ((threadIdx.x & 31) == 0 && local) atomicAdd(bad, local);
}

cudaError_t launch_label_check(const double *y, int64_t m, int *bad, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(bad, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    int64_t blocks = (m + 255) / 256;
    if (blocks > 1024) blocks = 1024;
    label_check_kernel<<<(unsigned)blocks, 256, 0, st>>>(y, m, bad);
    return cudaGetLastError();
}

__global__ void f64_to_f32_kernel(const double *src, int64_t count, float *dst)
{
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < count; j += (int64_t)gridDim.x * blockDim.x)
        dst[j] = (float)src[j];
}

cudaError_t launch_f64_to_f32(const double *src, int64_t count, float *dst, cudaStream_t st)
{
    if (count <= 0) return cudaSuccess;
    int64_t blocks = (count + 255) / 256;
    if (blocks > 1024) blocks = 1024;
    f64_to_f32_kernel<<<(unsigned)blocks, 256, 0, st>>>(src, count, dst);
    return cudaGetLastError();
}

// h[r] = gamma * log2(e) * ||x_r||^2 of an FP8 row, the dequantised norm rscale[r]^2 * sum
// value(q)^2, for the RBF expansion ||a||^2 + ||b||^2 - 2 a.b (Section 5.2); 0 for the other
// kernels.  One warp per row: FP32 sums of a lane's columns, combined in FP64, fixed order.
// (pack.cu forms the other operands' terms as it packs them.)
__global__ void row_terms_fp8_kernel(const uint8_t *packed, int64_t n_pad, int64_t m, double scale, float *h,
                                     const float *rscale)
{
    const int lane = threadIdx.x & 31;
    const int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (r >= m) return;
    float sf = 0.f;
    for (int64_t c = lane; c < n_pad; c += 32) {
        const float v = e4m3_value(packed[r * n_pad + c]);
        sf = fmaf(v, v, sf);
    }
    double s = sf;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    s *= (double)rscale[r] * (double)rscale[r];
    if (lane == 0) h[r] = (float)(scale * s);
}

cudaError_t launch_row_terms_fp8(const void *packed, int64_t n_pad, int64_t m, const KernelParams &kp, float *h,
                                 cudaStream_t st, const float *rscale)
{
    if (!rscale) return cudaErrorInvalidValue;
    if (m <= 0) return cudaSuccess;
    const double scale = (kp.kind == DCD_RBF) ? kp.gamma * 1.4426950408889634 : 0.0;
    const int64_t blocks = (m * 32 + 255) / 256;
    row_terms_fp8_kernel<<<(unsigned)blocks, 256, 0, st>>>((const uint8_t *)packed, n_pad, m, scale, h, rscale);
    return cudaGetLastError();
}

// dst row j = src row idx[j] (whole packed rows, 16-byte vectors; row_bytes
// is a multiple of 128), and d0[j] = f0[idx[j]], d1[j] = f1[idx[j]] where
// given.  Indices outside [0, m) give a zero row (and zero values) and set
// DEV_BAD_INDEX.  With link: link[j] = the first position q of the previous
// step with prev[q] == idx[j], or -1 (where the update's part of the gradient
// at a row that the next step samples is found).
// A warp per row, its loads in flight together: latency-bound, the index, then the row.  The links are a
// scan of prev by the same warp (int4 loads, L2 hits) while the row is on its way: a kernel of its own
// took 6 us, which the CTAs of the Gram waited for (their SMs), after 5 us of a gather element by element.
constexpr int GATHER_WARPS = 8;

__global__ void __launch_bounds__(GATHER_WARPS * 32)
    gather_rows_kernel(const uint4 *src, int64_t row_vec, const int32_t *idx, int64_t count, int64_t m, uint4 *dst,
                       int *err, const float *f0, float *d0, const float *f1, float *d1, const float *f2, float *d2,
                       const int32_t *prev, int cprev, int32_t *link)
{
    const int lane = threadIdx.x & 31;
    for (int64_t j = (int64_t)blockIdx.x * GATHER_WARPS + (threadIdx.x >> 5); j < count;
         j += (int64_t)gridDim.x * GATHER_WARPS) {
        const int32_t r = idx[j];
        const bool bad = r < 0 || r >= m;
        if (bad && lane == 0) set_error(err, DEV_BAD_INDEX);
        const uint4 *s = src + (bad ? 0 : r) * row_vec;
        uint4 *d = dst + j * row_vec;
        for (int64_t c0 = 0; c0 < row_vec; c0 += 128) {
            uint4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int64_t c = c0 + 32 * u + lane;
                if (c < row_vec) v[u] = bad ? make_uint4(0, 0, 0, 0) : s[c];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int64_t c = c0 + 32 * u + lane;
                if (c < row_vec) d[c] = v[u];
            }
        }
        if (lane == 0 && d0) d0[j] = bad ? 0.f : f0[r];
        if (lane == 1 && d1) d1[j] = bad ? 0.f : f1[r];
        if (lane == 2 && d2) d2[j] = bad ? 0.f : f2[r];
        if (link) {
            int first = INT32_MAX;
            const int4 *p4 = (const int4 *)prev;
#pragma unroll 8
            for (int q = lane; q < cprev / 4; q += 32) {
                const int4 v = p4[q];
                const int at = v.x == r ? 0 : v.y == r ? 1 : v.z == r ? 2 : v.w == r ? 3 : -1;
                if (at >= 0) first = min(first, 4 * q + at);
            }
            for (int q = (cprev & ~3) + lane; q < cprev; q += 32)
                if (prev[q] == r) first = min(first, q);
            first = __reduce_min_sync(0xffffffffu, first);
            if (lane == 0) link[j] = first == INT32_MAX ? -1 : first;
        }
    }
}

cudaError_t launch_gather_rows(const void *src, int64_t row_bytes, const int32_t *idx, int64_t count, int64_t m,
                               void *dst, int *err, cudaStream_t st, const float *f0, float *d0, const float *f1,
                               float *d1, const float *f2, float *d2, const int32_t *prev, int64_t cprev, int32_t *link)
{
    if (count <= 0) return cudaSuccess;
    if ((d0 && !f0) || (d1 && !f1) || (d2 && !f2)) return cudaErrorInvalidValue;
    if (link && (!prev || cprev > INT32_MAX || ((uintptr_t)prev & 15) != 0)) return cudaErrorInvalidValue;
    int64_t blocks = (count + GATHER_WARPS - 1) / GATHER_WARPS;
    if (blocks > 152 * 8) blocks = 152 * 8;
    gather_rows_kernel<<<(unsigned)blocks, GATHER_WARPS * 32, 0, st>>>((const uint4 *)src, row_bytes / 16, idx, count, m,
                                                                       (uint4 *)dst, err, f0, d0, f1, d1, f2, d2, prev,
                                                                       (int)cprev, link);
    return cudaGetLastError();
}

__global__ void fill_f64_kernel(double *p, double v, int64_t count)
{
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < count; j += (int64_t)gridDim.x * blockDim.x)
        p[j] = v;
}

cudaError_t launch_fill_f64(double *p, double v, int64_t count, cudaStream_t st)
{
    if (count <= 0) return cudaSuccess;
    int64_t blocks = (count + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    fill_f64_kernel<<<(unsigned)blocks, 256, 0, st>>>(p, v, count);
    return cudaGetLastError();
}

// ------------------------------------------------------ gradient init -----
// The diagonal and constant parts of the cached gradient:
//   K-SVM (problem 0): g = -1 + omega * alpha     (+ Q alpha added by the block kernel)
//   K-RR  (problem 1): g = m * alpha - y          (+ K alpha / lambda added likewise)
__global__ void init_grad_kernel(int problem, const double *y, const double *alpha, double diag, int64_t m, double *g)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        double a = alpha[i];
        g[i] = (problem == 0) ? (-1.0 + diag * a) : (diag * a - y[i]);
    }
}

cudaError_t launch_init_grad(int problem, const double *y, const double *alpha, double diag, int64_t m, double *g,
                             cudaStream_t st)
{
    int64_t blocks = (m + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    init_grad_kernel<<<(unsigned)blocks, 256, 0, st>>>(problem, y, alpha, diag, m, g);
    return cudaGetLastError();
}

// Coefficients of the initial gradient pass for a nonzero alpha_0:
// w[j] = y[c] * alpha[c] (K-SVM, y given) or alpha[c] * scale (K-RR, 1/lambda).
__global__ void coef_kernel(const double *y, const double *alpha, const int32_t *cols, int64_t count, double scale,
                            double *w)
{
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < count; j += (int64_t)gridDim.x * blockDim.x) {
        int32_t c = cols[j];
        w[j] = y ? y[c] * alpha[c] : alpha[c] * scale;
    }
}

cudaError_t launch_coef(const double *y, const double *alpha, const int32_t *cols, int64_t count, double scale,
                        double *w, cudaStream_t st)
{
    if (count <= 0) return cudaSuccess;
    int64_t blocks = (count + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    coef_kernel<<<(unsigned)blocks, 256, 0, st>>>(y, alpha, cols, count, scale, w);
    return cudaGetLastError();
}

__global__ void nnz_kernel(const double *alpha, int64_t m, int *count)
{
    int local = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x)
        local += (alpha[i] != 0.0);
    for (int o = 16; o > 0; o >>= 1) local += __shfl_xor_sync(0xffffffffu, local, o);
    if ((threadIdx.x & 31) == 0 && local) atomicAdd(count, local);
}

cudaError_t launch_nnz_count(const double *alpha, int64_t m, int *count, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(count, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    int64_t blocks = (m + 255) / 256;
    if (blocks > 1024) blocks = 1024;
    nnz_kernel<<<(unsigned)blocks, 256, 0, st>>>(alpha, m, count);
    return cudaGetLastError();
}

// --------------------------------------------------------- alpha update ---
// alpha_{sk+s} = alpha_sk + sum_t V_t delta_t (Algorithms 2 and 4) and the
// diagonal part of the gradient update, g[S_j] += diag * delta_j (omega for
// K-SVM-L2, m for K-RR).  Repeated indices are merged deterministically: a
// position with no earlier occurrence of its index is a run head and adds the
// deltas of its index's occurrences in position order.  One warp per
// position, S staged in shared memory: the warp compares 128 positions per
// step (4 per lane, ballot), so a position costs cnt / 128 steps.
// cnt <= 8192.  Also advances the stream counter.
constexpr int UPD_MAX = 8192;
constexpr int UPD_WARPS = 8;

__global__ void __launch_bounds__(UPD_WARPS * 32)
    update_kernel(const int32_t *S, const double *delta, int cnt, double diag, double *alpha, double *g,
                  uint64_t *ctr, uint64_t ctr_advance, int64_t m, int *err)
{
    __shared__ __align__(16) int32_t sS[UPD_MAX];
    // a kernel launched as this one's programmatic dependent may start; it waits for this grid to
    // finish before it touches alpha or g (a no-op without one)
    if (threadIdx.x == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int c4 = (cnt + 3) & ~3;
    for (int q = threadIdx.x; q < c4; q += blockDim.x) sS[q] = q < cnt ? S[q] : -1;
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x == 0 && ctr) *ctr += ctr_advance;
    const int lane = threadIdx.x & 31;
    const int nw = gridDim.x * UPD_WARPS;
    const int4 *s4 = (const int4 *)sS;
    for (int p = blockIdx.x * UPD_WARPS + (threadIdx.x >> 5); p < cnt; p += nw) {  // warp-uniform
        const int32_t key = sS[p];
        if (key < 0 || key >= m) {
            if (lane == 0) set_error(err, DEV_BAD_INDEX);
            continue;
        }
        // head: no earlier position holds key (128 positions per step, 4 per lane)
        bool head = true;
        for (int q0 = 0; q0 < p && head; q0 += 128) {
            const int q = q0 + 4 * lane;
            bool hit = false;
            if (q < p) {
                const int4 w = s4[q >> 2];
                hit = (w.x == key) || (q + 1 < p && w.y == key) || (q + 2 < p && w.z == key) ||
                      (q + 3 < p && w.w == key);
            }
            head = !__any_sync(0xffffffffu, hit);
        }
        if (!head) continue;
        // occurrences at positions >= p, in position order (every lane the same sum)
        double sum = 0.0;
        for (int q0 = p & ~3; q0 < c4; q0 += 128) {
            const int q = q0 + 4 * lane;
            unsigned mk = 0;
            if (q < c4) {
                const int4 w = s4[q >> 2];
                mk = (w.x == key ? 1u : 0u) | (w.y == key ? 2u : 0u) | (w.z == key ? 4u : 0u) | (w.w == key ? 8u : 0u);
                if (q < p) mk &= ~((1u << (p - q)) - 1u);  // only the group holding p starts below p
            }
            unsigned lanes = __ballot_sync(0xffffffffu, mk != 0);
            while (lanes) {  // rare: lanes in order, each lane's hits in order
                const int l = __ffs(lanes) - 1;
                unsigned ml = __shfl_sync(0xffffffffu, mk, l);
                const int ql = q0 + 4 * l;
                while (ml) {
                    sum += delta[ql + __ffs(ml) - 1];
                    ml &= ml - 1;
                }
                lanes &= lanes - 1;
            }
        }
        if (lane == 0) {
            alpha[key] += sum;
            g[key] += diag * sum;
        }
    }
}

// ------------------------------------------------- deferred gradient --
// The deferred K-SVM step.  snapshot: alpha and g at the next step's coordinates, taken before
// this step's block and update write them.
__global__ void dcd_snapshot_kernel(const int32_t *S, int64_t cnt, int64_t m, const double *alpha, const double *g,
                                    double *alpha_out, double *g_out)
{
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= cnt) return;
    const int64_t i = S[p];
    const bool ok = i >= 0 && i < m;
    alpha_out[p] = ok ? alpha[i] : 0.0;
    g_out[p] = ok ? g[i] : 0.0;
}

cudaError_t launch_dcd_snapshot(const int32_t *S, int64_t cnt, int64_t m, const double *alpha, const double *g,
                                double *alpha_out, double *g_out, cudaStream_t st)
{
    if (cnt <= 0) return cudaSuccess;
    dcd_snapshot_kernel<<<(unsigned)((cnt + 127) / 128), 128, 0, st>>>(S, cnt, m, alpha, g, alpha_out, g_out);
    return cudaGetLastError();
}

// The pending parts of the next step's alpha and g at its coordinates p (rows S[p]) from this
// step (coordinates Sc, steps theta, coefficients w = y theta):
//   g_add[p] = y[S[p]] (sum_j Kx[p][j] w[j]) + diag * (sum of theta over this step's positions
//              holding row S[p], in position order), alpha_add[p] = that sum.
// One warp per p; the lanes' partial sums over j are combined by a fixed butterfly.
template <typename KT>
__global__ void dcd_pending_kernel(const int32_t *S, int cnt, const double *y, const KT *Kx, int64_t ldx,
                                   const int32_t *Sc, const double *theta, const double *w, int cc, double diag,
                                   double *alpha_add, double *g_add)
{
    const int lane = threadIdx.x & 31;
    const int p = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (p >= cnt) return;  // warp-uniform
    const int32_t key = S[p];
    double dot = 0.0;
    for (int j = lane; j < cc; j += 32) dot = fma((double)Kx[(int64_t)p * ldx + j], w[j], dot);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
    double sum = 0.0;
    bool any = false;
    for (int q0 = 0; q0 < cc; q0 += 32) {
        unsigned hit = __ballot_sync(0xffffffffu, q0 + lane < cc && Sc[q0 + lane] == key);
        any = any || hit != 0u;
        while (hit) {  // in position order
            sum += theta[q0 + __ffs(hit) - 1];
            hit &= hit - 1u;
        }
    }
    if (lane == 0) {
        double v = y[key] * dot;
        if (any) v += diag * sum;
        g_add[p] = v;
        alpha_add[p] = any ? sum : 0.0;
    }
}

cudaError_t launch_dcd_pending(const int32_t *S, int64_t cnt, const double *y, const void *Kx, bool kx_f64,
                               int64_t ldx, const int32_t *Sc, const double *theta, const double *w, int64_t cc,
                               double diag, double *alpha_add, double *g_add, cudaStream_t st)
{
    if (cnt <= 0) return cudaSuccess;
    const unsigned blocks = (unsigned)((cnt + 3) / 4);
    if (kx_f64)
        dcd_pending_kernel<double><<<blocks, 128, 0, st>>>(S, (int)cnt, y, (const double *)Kx, ldx, Sc, theta, w,
                                                           (int)cc, diag, alpha_add, g_add);
    else
        dcd_pending_kernel<float><<<blocks, 128, 0, st>>>(S, (int)cnt, y, (const float *)Kx, ldx, Sc, theta, w,
                                                          (int)cc, diag, alpha_add, g_add);
    return cudaGetLastError();
}

cudaError_t launch_update(const int32_t *S, const double *delta, int64_t cnt, double diag, double *alpha, double *g,
                          uint64_t *ctr, uint64_t ctr_advance, int64_t m, int *err, cudaStream_t st, bool pdl,
                          int prio)
{
    if (cnt <= 0) return cudaSuccess;
    if (cnt > UPD_MAX) return cudaErrorInvalidValue;
    int64_t blocks = (cnt + UPD_WARPS - 1) / UPD_WARPS;
    if (blocks > 152) blocks = 152;
    if (!pdl && !prio) {
        update_kernel<<<(unsigned)blocks, UPD_WARPS * 32, 0, st>>>(S, delta, (int)cnt, diag, alpha, g, ctr,
                                                                   ctr_advance, m, err);
        return cudaGetLastError();
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks, 1, 1);
    cfg.blockDim = dim3(UPD_WARPS * 32, 1, 1);
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    unsigned na = 0;
    if (pdl) {
        at[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[na++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (prio) {
        at[na].id = cudaLaunchAttributePriority;
        at[na++].val.priority = prio;
    }
    cfg.attrs = at;
    cfg.numAttrs = na;
    return cudaLaunchKernelEx(&cfg, update_kernel, S, delta, (int)cnt, diag, alpha, g, ctr, ctr_advance, m, err);
}

// -------------------------------------------------------- convergence ----
// Partial sums over a fixed partition of [0, m), then one block combines the
// partials in index order, so the result is reproducible.
//   K-RR:  r[0] = ||g||^2
//   K-SVM: with (Q a)_i = g_i + 1 - omega a_i:
//          r[0] = a^T Q a, r[1] = sum a, r[2] = ||a||^2, r[3] = sum max(0, 1-(Qa)_i)^p
constexpr int CHECK_BLOCKS = 256;
constexpr int CHECK_THREADS = 256;

__global__ void check_partial_kernel(int problem, const double *g, const double *alpha, int64_t m, double C, int loss,
                                     double *partials)
{
    __shared__ double red[4][CHECK_THREADS];
    double s0 = 0, s1 = 0, s2 = 0, s3 = 0;
    const double omega = (loss == 2) ? 1.0 / (2.0 * C) : 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        double gi = g[i];
        if (problem == 1) {
            s0 += gi * gi;
        } else {
            double a = alpha[i];
            double qa = gi + 1.0 - omega * a;
            double xi = fmax(0.0, 1.0 - qa);
            s0 += a * qa;
            s1 += a;
            s2 += a * a;
            s3 += (loss == 1) ? xi : xi * xi;
        }
    }
    red[0][threadIdx.x] = s0;
    red[1][threadIdx.x] = s1;
    red[2][threadIdx.x] = s2;
    red[3][threadIdx.x] = s3;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w)
            for (int q = 0; q < 4; ++q) red[q][threadIdx.x] += red[q][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x < 4) partials[blockIdx.x * 4 + threadIdx.x] = red[threadIdx.x][0];
}

// one warp per quantity: each lane sums a fixed strided subset of the
// partials, then a fixed shuffle tree (FP64 adds have a 64-cycle latency, so
// a serial loop over the partials would dominate the check)
__global__ void check_final_kernel(const double *partials, int nblocks, double *result)
{
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (w >= 4) return;
    double s0 = 0.0, s1 = 0.0;
    int b = lane;
    for (; b + 32 < nblocks; b += 64) {
        s0 += partials[b * 4 + w];
        s1 += partials[(b + 32) * 4 + w];
    }
    if (b < nblocks) s0 += partials[b * 4 + w];
    double s = s0 + s1;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) result[w] = s;
}

cudaError_t launch_check(int problem, const double *g, const double *alpha, const double *y, int64_t m, double C,
                         int loss, double *partials, double *result, cudaStream_t st)
{
    (void)y;
    check_partial_kernel<<<CHECK_BLOCKS, CHECK_THREADS, 0, st>>>(problem, g, alpha, m, C, loss, partials);
    check_final_kernel<<<1, 128, 0, st>>>(partials, CHECK_BLOCKS, result);
    return cudaGetLastError();
}

}  // namespace dcd
