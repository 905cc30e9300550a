// pack.cu -- the packed operands of the tensor-core kernel block and their RBF row terms.
//
// One pass per operand: a warp per row (or four) reads the row's values, writes the operand's planes and sums
// the row's squared norm from the rounded values it has just formed (the norm of the row the MMAs
// see).  HBM-bound: each value is read once and each plane written once (a second read where every
// row's scale hangs on the matrix's largest magnitude, fp16).  Loads go eight columns a lane ahead
// of the conversions; lanes own columns lane, lane + 32, ... and sum them in that order.  Measured
// at 50000 x 512 FP32 (102 MB): fp16 packed and its terms 34 us and the largest magnitude 18 (227
// together when the magnitude, the pack and the terms were kernels with scalar loads, one atomic per row
// and FP64 sums), sliced 20000 x 512 30 us (714).
#include "dcd_internal.cuh"

#include <cuda_fp16.h>

namespace dcd {

namespace {

// Element `off` of a dense source of type DT: as FP32 (an FP8 source is scale * value(q) rounded
// once), or as FP64.
template <int DT>
__device__ __forceinline__ float src_f32(const void *src, int64_t off, float scale)
{
    if (DT == DCD_F64) return (float)((const double *)src)[off];
    if (DT == DCD_F32) return ((const float *)src)[off];
    if (DT == DCD_BF16) return __bfloat162float(((const __nv_bfloat16 *)src)[off]);
    return (float)((double)scale * (double)e4m3_value(((const uint8_t *)src)[off]));
}

template <int DT>
__device__ __forceinline__ double src_f64(const void *src, int64_t off, float scale)
{
    if (DT == DCD_F64) return ((const double *)src)[off];
    if (DT == DCD_FP8E4M3) return (double)scale * (double)e4m3_value(((const uint8_t *)src)[off]);
    return (double)src_f32<DT>(src, off, scale);
}

// The type the sliced form cuts in: FP32 sources exactly in FP32, the others in FP64.
template <int DT> struct SliceT { typedef double type; };
template <> struct SliceT<DCD_F32> { typedef float type; };
template <> struct SliceT<DCD_BF16> { typedef float type; };

__device__ __forceinline__ float pow2f(int k) { return __int_as_float((k + 127) << 23); }

// v 2^k exactly (or 0 where it is far below the slices), |k| < 254, in two steps within the range
__device__ __forceinline__ float scale_slices(float v, int k) { return v * pow2f(k / 2) * pow2f(k - k / 2); }
__device__ __forceinline__ double scale_slices(double v, int k) { return ldexp(v, k); }
__device__ __forceinline__ int exponent_of(float v)
{
    int e;
    frexpf(v, &e);
    return e;
}
__device__ __forceinline__ int exponent_of(double v)
{
    int e;
    frexp(v, &e);
    return e;
}

constexpr int PK_U = 8;  // columns a lane loads ahead

// Row r of the destination = source row rows[r] (or r), in the operand kind KIND, zero past column n:
//   BF16, TF32 rounded; BF16X3, TF32X3 split in hi and lo planes; FP16 scaled by the power of two
//   *gbits fixes (sc[r] = the scale: 2^(e - 15), the matrix's largest magnitude in [2^(e-1), 2^e), e
//   >= -110 so that it stays a normal number); SLICED four planes of integers in [-64, 64] of the row
//   scaled by sc[r] = 2^e, its own largest magnitude in [2^(e-1), 2^e):
//   s0 = rint(64 u), s_p = rint(128 r), each step exact (power-of-two scalings and differences).
// h[r] = hscale ||x_r||^2 of the packed row (BF16, TF32, BF16X3: FP32 sums of a lane's columns,
// combined in FP64; TF32X3: FP64; FP16: exact squares in double-single sums; SLICED: exact integer
// sums of the plane products the block keeps), as the pair h + h_lo where h_lo is given.  Split rows
// take the norm the three MMAs reproduce, sum hi (hi + 2 lo).  A row index outside [0, m) gives a
// zero row and DEV_BAD_INDEX; SLICED: an infinite value sets DEV_BAD_VALUE.
template <int KIND, int DT, int R>
__global__ void __launch_bounds__(256) pack_terms_kernel(const void *__restrict__ src, int64_t ld, int64_t m, int64_t n,
                                                         const int32_t *__restrict__ rows, void *__restrict__ dst,
                                                         int64_t n_pad, int64_t count, double hscale, float *h,
                                                         float *h_lo, float *sc, const unsigned *gbits,
                                                         const float *src_scale, int *err)
{
    typedef typename SliceT<DT>::type ST;
    const int lane = threadIdx.x & 31;
    const int64_t r0 = ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5) * R;
    if (r0 >= count) return;
    double part[R];  // the lane's share of each row's squared norm
    float scr = 1.f;
    double sd = 0.0;
    int S0 = 0, S1 = 0, S2 = 0, S3 = 0;
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int64_t r = r0 + i;
        part[i] = 0.0;
        if (r >= count) continue;  // warp-uniform
        const int64_t sr = rows ? (int64_t)rows[r] : r;
        const bool inb = sr >= 0 && sr < m;
        if (!inb && lane == 0) set_error(err, DEV_BAD_INDEX);
        const float rsc = (DT == DCD_FP8E4M3 && inb) ? src_scale[sr] : 0.f;
        const int64_t off = sr * ld;
        float fscale = 1.f;
        int e = 0;
        if (KIND == PACK_FP16) {
            const float mx = __uint_as_float(*gbits);
            if (mx > 0.f && isfinite(mx)) frexpf(mx, &e);
            e = max(e, -110);
            fscale = pow2f(15 - e);
            scr = pow2f(e - 15);
            if (lane == 0) sc[r] = scr;
        }
        if (KIND == PACK_SLICED) {
            ST mx = 0;
            for (int64_t c0 = lane; c0 < n; c0 += 32 * PK_U) {
#pragma unroll
                for (int u = 0; u < PK_U; ++u) {
                    const int64_t c = c0 + 32 * u;
                    if (c < n && inb) {
                        const ST v = sizeof(ST) == 4 ? (ST)src_f32<DT>(src, off + c, rsc) : (ST)src_f64<DT>(src, off + c, rsc);
                        const ST av = v < 0 ? -v : v;
                        mx = av > mx ? av : mx;
                    }
                }
            }
            for (int o = 16; o > 0; o >>= 1) {
                const ST w = __shfl_xor_sync(0xffffffffu, mx, o);
                mx = w > mx ? w : mx;
            }
            if (mx > 0 && isfinite(mx)) e = exponent_of(mx);
            else if (!(mx == 0) && lane == 0) set_error(err, DEV_BAD_VALUE);
            scr = ldexpf(1.f, e);
            if (lane == 0) sc[r] = scr;
        }
        float sf = 0.f, cf = 0.f;
        sd = 0.0;
        for (int64_t c0 = lane; c0 < n_pad; c0 += 32 * PK_U) {
            float v[PK_U];
            ST w[PK_U];
#pragma unroll
            for (int u = 0; u < PK_U; ++u) {
                const int64_t c = c0 + 32 * u;
                const bool in = c < n && inb;
                if (KIND == PACK_SLICED)
                    w[u] = !in ? (ST)0
                           : sizeof(ST) == 4 ? (ST)src_f32<DT>(src, off + c, rsc) : (ST)src_f64<DT>(src, off + c, rsc);
                else
                    v[u] = in ? src_f32<DT>(src, off + c, rsc) : 0.f;
            }
#pragma unroll
            for (int u = 0; u < PK_U; ++u) {
                const int64_t c = c0 + 32 * u;
                if (c >= n_pad) break;
                if (KIND == PACK_BF16X3) {  // v - hi is exact in fp32
                    const __nv_bfloat16 hi = __float2bfloat16_rn(v[u]);
                    const __nv_bfloat16 lo = __float2bfloat16_rn(v[u] - __bfloat162float(hi));
                    __nv_bfloat16 *d = (__nv_bfloat16 *)dst + r * 2 * n_pad;
                    d[c] = hi;
                    d[n_pad + c] = lo;
                    const float fh = __bfloat162float(hi), fl = __bfloat162float(lo);
                    sf = fmaf(fh, fh + 2.f * fl, sf);
                } else if (KIND == PACK_TF32X3) {  // both planes on the tf32 grid
                    uint32_t th, tl;
                    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(th) : "f"(v[u]));
                    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(tl) : "f"(v[u] - __uint_as_float(th)));
                    float *d = (float *)dst + r * 2 * n_pad;
                    d[c] = __uint_as_float(th);
                    d[n_pad + c] = __uint_as_float(tl);
                    const double fh = __uint_as_float(th), fl = __uint_as_float(tl);
                    sd = fma(fh, fh + 2.0 * fl, sd);
                } else if (KIND == PACK_TF32) {
                    // the tf32 grid (10-bit mantissa, nearest, ties away), so that the tensor core sees
                    // exactly the stored value and the row norms match
                    uint32_t t;
                    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(t) : "f"(v[u]));
                    ((float *)dst)[r * n_pad + c] = __uint_as_float(t);
                    sf = fmaf(__uint_as_float(t), __uint_as_float(t), sf);
                } else if (KIND == PACK_FP16) {
                    const __half q = __float2half_rn(v[u] * fscale);  // a power of two: exact, or rounded once
                    ((__half *)dst)[r * n_pad + c] = q;
                    const float f = __half2float(q), p = f * f;  // 22 bits: exact
                    const float t = sf + p, z = t - sf;          // TwoSum
                    cf += (sf - (t - z)) + (p - z);
                    sf = t;
                } else if (KIND == PACK_SLICED) {
                    ST x = scale_slices(w[u], 6 - e);
                    const ST d0 = rint(x);
                    x = (x - d0) * (ST)128;
                    const ST d1 = rint(x);
                    x = (x - d1) * (ST)128;
                    const ST d2 = rint(x);
                    x = (x - d2) * (ST)128;
                    const ST d3 = rint(x);
                    __nv_bfloat16 *d = (__nv_bfloat16 *)dst + r * 4 * n_pad;
                    d[c] = __float2bfloat16_rn((float)d0);
                    d[n_pad + c] = __float2bfloat16_rn((float)d1);
                    d[2 * n_pad + c] = __float2bfloat16_rn((float)d2);
                    d[3 * n_pad + c] = __float2bfloat16_rn((float)d3);
                    const int i0 = (int)d0, i1 = (int)d1, i2 = (int)d2, i3 = (int)d3;
                    S0 += i0 * i0;
                    S1 += 2 * i0 * i1;
                    S2 += 2 * i0 * i2 + i1 * i1;
                    S3 += 2 * (i0 * i3 + i1 * i2);
                } else {
                    const __nv_bfloat16 q = __float2bfloat16_rn(v[u]);
                    ((__nv_bfloat16 *)dst)[r * n_pad + c] = q;
                    sf = fmaf(__bfloat162float(q), __bfloat162float(q), sf);
                }
            }
        }
        part[i] = KIND == PACK_FP16 ? (double)sf + (double)cf : KIND == PACK_TF32X3 ? sd : (double)sf;
    }
    int own = 0;  // the row that this lane holds the sum of
    if (KIND == PACK_SLICED) {
        // a.a = sc^2 2^-12 (S0 + 2^-7 S1 + 2^-14 S2 + 2^-21 S3)
        for (int o = 16; o > 0; o >>= 1) {
            S0 += __shfl_xor_sync(0xffffffffu, S0, o);
            S1 += __shfl_xor_sync(0xffffffffu, S1, o);
            S2 += __shfl_xor_sync(0xffffffffu, S2, o);
            S3 += __shfl_xor_sync(0xffffffffu, S3, o);
        }
        if (lane) return;
        const double s = scr;
        sd = hscale * (s * s) * 0x1p-12 * ((double)S0 + 0x1p-7 * (double)S1 + 0x1p-14 * (double)S2 + 0x1p-21 * (double)S3);
    } else {
        // the butterfly over the lanes, a step of which halves the rows a lane holds as long as it holds
        // several: the same additions, R rows' at once
        int left = R;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            if (left > 1) {
                left >>= 1;
                const bool up = (lane & o) != 0;
                if (up) own += left;
#pragma unroll
                for (int i = 0; i < R / 2; ++i)
                    if (i < left) {
                        const double keep = up ? part[i + left] : part[i], send = up ? part[i] : part[i + left];
                        part[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                    }
            } else {
                part[0] += __shfl_xor_sync(0xffffffffu, part[0], o);
            }
        }
        if ((lane & (32 / R - 1)) || r0 + own >= count) return;
        sd = KIND == PACK_FP16 ? hscale * part[0] * (double)scr * (double)scr : hscale * part[0];
    }
    const float vh = (float)sd;
    h[r0 + own] = vh;
    if ((KIND == PACK_SLICED || KIND == PACK_TF32X3) && h_lo) h_lo[r0 + own] = (float)(sd - (double)vh);
}


// The largest magnitude of the first `count` rows of a dense source, folded into *bits (the FP32 bit
// pattern, which orders like the value for non-negative floats) by one atomicMax per CTA; a value
// that is not finite sets DEV_BAD_VALUE.  Warps stride over the rows; VEC: 16-byte loads (FP32 rows
// that start on 16-byte boundaries).
template <int DT, bool VEC>
__global__ void __launch_bounds__(256) absmax_rows_kernel(const void *__restrict__ src, int64_t ld, int64_t n,
                                                          int64_t count, unsigned *bits, int *err,
                                                          const float *src_scale)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t nw = (int64_t)gridDim.x * 8;
    unsigned mx = 0;  // |v| as bits: infinities and NaNs are the patterns from 0x7f800000
    for (int64_t r = blockIdx.x * 8 + warp; r < count; r += nw) {
        if (VEC) {
            const float4 *p = (const float4 *)((const float *)src + r * ld);
            const int64_t n4 = n >> 2;
#pragma unroll 4
            for (int64_t c = lane; c < n4; c += 32) {
                const float4 v = p[c];
                mx = max(mx, max(max(__float_as_uint(v.x) & 0x7fffffffu, __float_as_uint(v.y) & 0x7fffffffu),
                                 max(__float_as_uint(v.z) & 0x7fffffffu, __float_as_uint(v.w) & 0x7fffffffu)));
            }
            for (int64_t c = (n4 << 2) + lane; c < n; c += 32)
                mx = max(mx, __float_as_uint(((const float *)src)[r * ld + c]) & 0x7fffffffu);
        } else {
            const float rsc = DT == DCD_FP8E4M3 ? src_scale[r] : 0.f;
#pragma unroll 4
            for (int64_t c = lane; c < n; c += 32)
                mx = max(mx, __float_as_uint(src_f32<DT>(src, r * ld + c, rsc)) & 0x7fffffffu);
        }
    }
    __shared__ unsigned red[8];
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) red[warp] = mx;
    __syncthreads();
    if (threadIdx.x) return;
    for (int w = 0; w < 8; ++w) mx = max(mx, red[w]);
    if (mx >= 0x7f800000u) set_error(err, DEV_BAD_VALUE);
    else atomicMax(bits, mx);
}

// Rows a warp takes: four where that still leaves every SM some fifty warps, so that the FP64 sums of
// a row's terms (one FP64 instruction holds a scheduler for 64 cycles, and a row has twelve) are made
// for four rows at once.  fp16, 50000 x 512 FP32: 44 -> 34 us (23 at the memory's rate).
constexpr int64_t PACK_ROWS4 = 32768;

template <int KIND>
cudaError_t launch_dt(const void *src, int dtype, int64_t ld, int64_t m, int64_t n, const int32_t *rows, void *dst,
                      int64_t n_pad, int64_t count, double hscale, float *h, float *h_lo, float *sc,
                      const unsigned *gbits, const float *src_scale, int *err, cudaStream_t st)
{
    constexpr int R4 = KIND == PACK_FP16 || KIND == PACK_BF16 || KIND == PACK_BF16X3 ? 4 : 1;
    const bool four = R4 == 4 && count >= PACK_ROWS4;
    auto kfn = dtype == DCD_F64    ? (four ? pack_terms_kernel<KIND, DCD_F64, R4> : pack_terms_kernel<KIND, DCD_F64, 1>)
               : dtype == DCD_F32  ? (four ? pack_terms_kernel<KIND, DCD_F32, R4> : pack_terms_kernel<KIND, DCD_F32, 1>)
               : dtype == DCD_BF16 ? (four ? pack_terms_kernel<KIND, DCD_BF16, R4> : pack_terms_kernel<KIND, DCD_BF16, 1>)
                                   : (four ? pack_terms_kernel<KIND, DCD_FP8E4M3, R4>
                                           : pack_terms_kernel<KIND, DCD_FP8E4M3, 1>);
    const int64_t per = 8 * (four ? R4 : 1);
    kfn<<<(unsigned)((count + per - 1) / per), 256, 0, st>>>(src, ld, m, n, rows, dst, n_pad, count, hscale, h, h_lo, sc,
                                                             gbits, src_scale, err);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_pack_terms(const void *src, int dtype, int64_t ld, int64_t m, int64_t n, const int32_t *rows,
                              void *dst, int kind, int64_t n_pad, int64_t count, const KernelParams &kp, float *h,
                              int *err, cudaStream_t st, const float *src_scale, float *sc, const unsigned *gbits,
                              float *h_lo)
{
    if (count <= 0) return cudaSuccess;
    if (n_pad < n || n_pad % k_block_elems(kind) || (dtype == DCD_FP8E4M3 && !src_scale)) return cudaErrorInvalidValue;
    if ((kind == PACK_FP16 && (!sc || !gbits)) || (kind == PACK_SLICED && !sc)) return cudaErrorInvalidValue;
    if (h_lo && kind != PACK_TF32X3 && kind != PACK_SLICED) return cudaErrorInvalidValue;
    const double hs = kp.kind == DCD_RBF ? kp.gamma * 1.4426950408889634 : 0.0;
    switch (kind) {
    case PACK_BF16: return launch_dt<PACK_BF16>(src, dtype, ld, m, n, rows, dst, n_pad, count, hs, h, h_lo, sc, gbits, src_scale, err, st);
    case PACK_TF32: return launch_dt<PACK_TF32>(src, dtype, ld, m, n, rows, dst, n_pad, count, hs, h, h_lo, sc, gbits, src_scale, err, st);
    case PACK_BF16X3: return launch_dt<PACK_BF16X3>(src, dtype, ld, m, n, rows, dst, n_pad, count, hs, h, h_lo, sc, gbits, src_scale, err, st);
    case PACK_TF32X3: return launch_dt<PACK_TF32X3>(src, dtype, ld, m, n, rows, dst, n_pad, count, hs, h, h_lo, sc, gbits, src_scale, err, st);
    case PACK_FP16: return launch_dt<PACK_FP16>(src, dtype, ld, m, n, rows, dst, n_pad, count, hs, h, h_lo, sc, gbits, src_scale, err, st);
    case PACK_SLICED: return launch_dt<PACK_SLICED>(src, dtype, ld, m, n, rows, dst, n_pad, count, hs, h, h_lo, sc, gbits, src_scale, err, st);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_absmax_rows(const void *src, int dtype, int64_t ld, int64_t n, int64_t count, unsigned *bits,
                               int *err, cudaStream_t st, const float *src_scale)
{
    if (count <= 0) return cudaSuccess;
    if (dtype == DCD_FP8E4M3 && !src_scale) return cudaErrorInvalidValue;
    const int64_t want = (count + 7) / 8;
    const unsigned blocks = (unsigned)(want < 152 * 8 ? want : 152 * 8);
    if (dtype == DCD_F32 && ((uintptr_t)src & 15) == 0 && ld % 4 == 0)
        absmax_rows_kernel<DCD_F32, true><<<blocks, 256, 0, st>>>(src, ld, n, count, bits, err, src_scale);
    else if (dtype == DCD_F32)
        absmax_rows_kernel<DCD_F32, false><<<blocks, 256, 0, st>>>(src, ld, n, count, bits, err, src_scale);
    else if (dtype == DCD_F64)
        absmax_rows_kernel<DCD_F64, false><<<blocks, 256, 0, st>>>(src, ld, n, count, bits, err, src_scale);
    else if (dtype == DCD_BF16)
        absmax_rows_kernel<DCD_BF16, false><<<blocks, 256, 0, st>>>(src, ld, n, count, bits, err, src_scale);
    else
        absmax_rows_kernel<DCD_FP8E4M3, false><<<blocks, 256, 0, st>>>(src, ld, n, count, bits, err, src_scale);
    return cudaGetLastError();
}

}  // namespace dcd
