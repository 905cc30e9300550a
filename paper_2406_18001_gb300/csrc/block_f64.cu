// block_f64.cu -- the FP64 form's kernel block on the tensor cores, from exact slice products.
//
// GB300's FP64 pipe issues about 1.6 lane operations per clock per SM (a warp instruction every
// 20 cycles), so a block of direct differences (block_simt.cu: two FP64 operations per feature
// and entry) takes 4.7 ms for 6000 x 256 entries at n = 512.  Here each row is scaled by a power
// of two 2^e (max |a| < 2^e) and cut into eight slices, integers s_p in [-64, 64] exact in bf16,
//     a = 2^e (s_0 2^-6 + s_1 2^-13 + ... + s_7 2^-55) to within 2^(e-56)
// (the Ozaki splitting scheme: Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 2012), and the 36
// slice products with p + q <= 7 are summed by tcgen05 kind::f16 into eight FP32 accumulators by
// g = p + q.  Every sum is an exact integer: at most (g + 1) n 2^12 <= 2^24 for n <= 512.  The
// epilogue joins the eight in integer arithmetic and FP64, so that
//     a_i.a_j = 2^(e_i + e_j - 61) (I_hi 2^28 + I_lo),  I_hi, I_lo exact 64-bit integers,
// is rounded once.  What is left out (p + q >= 8, the ninth slice) is at most 9 2^-56 2^(e_i + e_j) a
// feature that is nonzero in both rows, about a tenth of that on average and of either sign: relative
// to the rows' largest magnitudes, not to sum_k |a_ik a_jk| as the rounding of an FP64 sum is.  The two
// are alike while the features that make up a product are not all tiny beside others; where a large
// feature of one row meets a zero of the other they are not (features of 1 beside one of 1e9: 1e-7
// relative).  So the linear and polynomial kernels take the form only if every row of the matrix has
// its magnitude spread over its features, or if the four last slices are zero in all of them (whole
// numbers up to 2^27, bits: nothing is left out); see f64s_row_flags.  Where the first holds,
// sum_k |a_ik a_jk| >= n 2^-11 2^(e_i + e_j) for every two rows, and the part left out stays below
// 2^-45 / sqrt(n) of it (n roundings of like size, of either sign).  The RBF exponent comes from the
// expansion gamma |a_i|^2 + gamma |a_j|^2 - 2 gamma a_i.a_j with norms from compensated FP64 sums: its
// absolute error is some 2^-53 gamma (|a_i|^2 + |a_j|^2), so the form is used where gamma |a|^2 <=
// F64S_HMAX for every row (pack_f64s reports the largest) and the direct differences serve elsewhere.
// What the slices leave out of 2 gamma a_i.a_j, about 2 gamma sqrt(n) 2^-56 2^(e_i + e_j), is less than
// that for rows whose magnitude is spread over their features; where one feature holds it and n is
// large it is more (one feature of 2.05, 511 of 1e-3, gamma |a|^2 = 7.9: 4.3e-14 in a kernel value), so
// gamma 4^e sqrt(n) / 2 has the same limit: at most four times 2^-53 is left out.
//
// What bounds it: the FP64 pipe, with 16 operations an entry instead of 2 n: two integer-to-double
// differences, a sum of the terms and two FMAs for the exponent, ten for exp, one for the
// contraction.  The tiles are 128 rows x 32 columns, one CTA each, persistent: eight accumulators
// of 32 columns fill half of tensor memory, so one unit's epilogue (43 k cycles) runs beside the
// next one's MMAs (18 k at n = 512).  For slice p of the rows one MMA per 16 features multiplies
// the stacked column slices 0..7-p (N = 32 (8 - p)) into accumulators p..7: the row slice is read
// from shared memory once for all its products.
//   warp 0      TMA producer: per 64-feature k-block the column slices (8 x 4 KB, two buffers)
//               and the eight row slices (16 KB each, a slot per slice)
//   warp 1      tensor-memory allocator and MMA issuer
//   warps 2..9  epilogue: a thread per row, two warps per lane quarter (16 columns each)
// Row sums of a tile over its column chunks go to scratch; the last warp to arrive at the tile
// (one atomic per warp) adds them in chunk order and updates g.
//
// Measured (K-RR, m = 6000, n = 512, sb = 256): block 4753 -> 92 us, Gram 4722 -> 34 us;
// the solve's alpha after 64 block updates is 3.3e-15 from 64-bit arithmetic (direct block 7.2e-15).
#include "dcd_internal.cuh"
#include "f64_math.cuh"
#include "tc_ptx.cuh"

namespace dcd {

namespace {

constexpr int FM = 128;            // rows per tile
constexpr int FN = 32;             // columns per tile
constexpr int NSL = 8;             // slices
constexpr int A_SLICE = FM * 128;  // a k-block (64 features) of one row slice: 16 KB
constexpr int B_SLICE = FN * 128;  // of one column slice: 4 KB
constexpr int B_STK = NSL * B_SLICE;
constexpr int COL_WORDS = 16 * 6;  // staged column terms of an epilogue warp: w, h (FP64), exponent, data row
constexpr int F64S_SMEM = 1024 + NSL * A_SLICE + 2 * B_STK + 256 + 64 * 8 + 8 * 2 * COL_WORDS * 4;
constexpr int F64S_THREADS = 320;
constexpr int F64S_COLS = 1024;    // columns per launch (bounds the scratch of the row sums)

struct F64Args {
    const int32_t *row_id, *col_id;  // data-matrix rows of the block's rows / columns (null: the number)
    const int32_t *ex;               // per data row: exponent e
    const double *h;                 // per data row: gamma |a|^2 (RBF)
    const double *w, *rs;            // apply
    double *g, *out;
    int64_t ldo, nrows, m;
    int ncols, ntiles, nchunks, kblocks;
    int64_t n_pad;
    double two_gamma, coef0;
    int degree;
    double *part;                    // [chunk][half][tile rows] row sums
    unsigned *cnt;                   // per tile, zero between launches
    int *err;
};

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}

__device__ __forceinline__ void tmem_wait8(uint32_t (&r)[8])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7])
                 :
                 : "memory");
}

// v 2^k for a normal or zero v whose result is normal (an integer add to the exponent field)
// (|k| <= 461 here: a value of 2^-500 or more stays normal)
__device__ __forceinline__ double scale2(double v, int k)
{
    const int hi = __double2hiint(v);
    return v == 0.0 ? 0.0 : __hiloint2double(hi + (k << 20), __double2loint(v));
}

// an integer |i| < 2^51 as a double: 1.5 2^52 + i built in the bit pattern, less 1.5 2^52
__device__ __forceinline__ double int_to_double(long long i)
{
    return __longlong_as_double(0x4338000000000000LL + i) - 6755399441055744.0;
}

template <int KIND>
__global__ void __launch_bounds__(F64S_THREADS, 1)
    block_f64s_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, F64Args a)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *sA = smem, *sB = smem + NSL * A_SLICE;
    uint64_t *bars = (uint64_t *)(sB + 2 * B_STK);
    uint64_t *fullA = bars, *emptyA = bars + NSL, *fullB = bars + 2 * NSL, *emptyB = fullB + 2, *tfull = emptyB + 2,
             *tempty = tfull + 2, *drain = tempty + 2;
    uint32_t *tmem_holder = (uint32_t *)(drain + 1);
    volatile int *abort_flag = (volatile int *)(tmem_holder + 1);
    double *tab = (double *)(sB + 2 * B_STK + 256);
    double *colterms = tab + 64;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < NSL; ++s) {
            mbar_init(&fullA[s], 1);
            mbar_init(&emptyA[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&fullB[b], 1);
            mbar_init(&emptyB[b], 1);
            mbar_init(&tfull[b], 1);
            mbar_init(&tempty[b], 8);
        }
        mbar_init(drain, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (KIND == DCD_RBF && threadIdx.x >= 64 && threadIdx.x < 128) tab[threadIdx.x - 64] = exp_tab_entry(threadIdx.x - 64);
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_holder)),
                     "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem_base = *tmem_holder;
    const int nunits = a.ntiles * a.nchunks;

    if (warp == 0) {
        // -------------------------------------------------------- producer --
        const uint32_t leader = elect_one();
        uint32_t kt = 0;          // k-blocks copied so far,
        uint32_t nb = 0, na = 0;  // and the column stacks (0 or 1) and row slices of the current one
        bool ok = true;
        for (int u = blockIdx.x; ok && u < nunits; u += gridDim.x) {
            const int ya = (u / a.nchunks) * FM, yb = (u % a.nchunks) * FN;
            for (int kb = 0; ok && kb < a.kblocks; ++kb, ++kt) {
                const uint32_t bs = kt & 1, bp = (kt >> 1) & 1;
                nb = na = 0;
                if (!(ok = mbar_wait_warp(&emptyB[bs], bp ^ 1, abort_flag, a.err))) break;
                nb = 1;
                if (leader) {
                    mbar_expect_tx(&fullB[bs], B_STK);
#pragma unroll
                    for (int p = 0; p < NSL; ++p)
                        tma_load_2d(sB + bs * B_STK + p * B_SLICE, &tmB, &fullB[bs], (int)(p * a.n_pad) + kb * 64, yb);
                }
                __syncwarp();
                for (int p = 0; p < NSL; ++p) {
                    if (!(ok = mbar_wait_warp(&emptyA[p], (kt & 1) ^ 1, abort_flag, a.err))) break;
                    if (leader) {
                        mbar_expect_tx(&fullA[p], A_SLICE);
                        tma_load_2d(sA + p * A_SLICE, &tmA, &fullA[p], (int)(p * a.n_pad) + kb * 64, ya);
                    }
                    __syncwarp();
                    ++na;
                }
                if (!ok) break;
            }
        }
        if (!ok && leader) {  // let every slot's last copy land before the CTA exits (bounded)
            for (uint32_t p = 0; p < NSL; ++p) {
                const uint32_t n = kt + (p < na ? 1 : 0);
                if (n) mbar_drain(&fullA[p], (n - 1) & 1);
            }
            for (uint32_t b = 0; b < 2; ++b) {
                const uint32_t n = (kt + nb + 1 - b) >> 1;
                if (n) mbar_drain(&fullB[b], (n - 1) & 1);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------------------- MMA --
        const uint32_t leader = elect_one();
        const uint32_t a0 = sw128_lo(su32(sA)), b0 = sw128_lo(su32(sB));
        uint32_t kt = 0, acc_it = 0;
        bool ok = true, issued = false;
        for (int u = blockIdx.x; ok && u < nunits; u += gridDim.x, ++acc_it) {
            const uint32_t buf = acc_it & 1, aph = (acc_it >> 1) & 1;
            if (!(ok = mbar_wait_warp(&tempty[buf], aph ^ 1, abort_flag, a.err))) break;
            fence_after();
            const uint32_t dtm = tmem_base + buf * (NSL * FN);
            for (int kb = 0; ok && kb < a.kblocks; ++kb, ++kt) {
                const uint32_t bs = kt & 1, bp = (kt >> 1) & 1;
                if (!(ok = mbar_wait_warp(&fullB[bs], bp, abort_flag, a.err))) break;
                const uint32_t bb = b0 + bs * (B_STK >> 4);
#pragma unroll
                for (int p = 0; p < NSL; ++p) {
                    if (!(ok = mbar_wait_warp(&fullA[p], kt & 1, abort_flag, a.err))) break;
                    fence_after();
                    if (leader) {
#pragma unroll
                        for (int k = 0; k < 4; ++k)  // row slice p times column slices 0..7-p into accumulators p..7
                            mma<0>(dtm + (uint32_t)(p * FN), a0 + p * (A_SLICE >> 4) + 2 * k, bb + 2 * k,
                                   make_idesc(1, FN * (NSL - p), FM), (kb > 0 || k > 0 || p > 0) ? 1u : 0u);
                        mma_commit(&emptyA[p]);
                    }
                    issued = true;
                    __syncwarp();
                }
                if (!ok) break;
                if (leader) mma_commit(&emptyB[bs]);
                __syncwarp();
            }
            if (!ok) break;
            if (leader) mma_commit(&tfull[buf]);
            __syncwarp();
        }
        if (issued && leader) {  // every MMA done before the CTA tears down (bounded)
            mma_commit(drain);
            mbar_drain(drain, 0);
        }
        __syncwarp();
    } else {
        // -------------------------------------------------------- epilogue --
        const int quarter = warp & 3, half = (warp - 2) >> 2;
        const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
        double *ct = colterms + (warp - 2) * COL_WORDS;  // two buffers of COL_WORDS / 2 doubles
        // the unit's column and row terms, loaded one unit ahead
        double n_w = 0.0, n_h = 0.0, r_h = 0.0;
        int n_e = 0, r_e = 0, n_id = -1, r_id = -2;  // no column and no row are no sample's own pair
        auto load_terms = [&](int u) {
            const int64_t c = (int64_t)(u % a.nchunks) * FN + half * 16 + (lane & 15);
            n_w = n_h = r_h = 0.0;
            n_e = r_e = 0;
            n_id = -1;
            r_id = -2;
            if (c < a.ncols) {
                const int64_t id = a.col_id ? a.col_id[c] : c;
                n_id = (int)id;
                if (id >= 0 && id < a.m) {
                    n_e = a.ex[id];
                    if (KIND == DCD_RBF) n_h = a.h[id];
                }
                if (a.w) n_w = a.w[c];
            }
            const int64_t r = (int64_t)(u / a.nchunks) * FM + quarter * 32 + lane;
            if (r < a.nrows) {
                const int64_t id = a.row_id ? a.row_id[r] : r;
                r_id = (int)id;
                if (id >= 0 && id < a.m) {
                    r_e = a.ex[id];
                    if (KIND == DCD_RBF) r_h = a.h[id];
                }
            }
        };
        if ((int)blockIdx.x < nunits) load_terms(blockIdx.x);
        uint32_t acc_it = 0;
        for (int u = blockIdx.x; u < nunits; u += gridDim.x, ++acc_it) {
            const int tile = u / a.nchunks, nc = u % a.nchunks;
            const uint32_t buf = acc_it & 1, aph = (acc_it >> 1) & 1;
            double *cb = ct + buf * (COL_WORDS / 2);
            if (lane < 16) {
                cb[lane] = n_w;
                cb[16 + lane] = n_h;
                ((int *)(cb + 32))[lane] = n_e;
                ((int *)(cb + 40))[lane] = n_id;
            }
            const double hr = r_h;
            const int er = r_e - 61, rid = r_id;
            if (u + (int)gridDim.x < nunits) load_terms(u + gridDim.x);
            __syncwarp();
            if (!mbar_wait_warp(&tfull[buf], aph, abort_flag, a.err)) break;
            fence_after();
            const int64_t row = (int64_t)tile * FM + quarter * 32 + lane;
            const double rf = scale2(a.two_gamma, er);  // RBF: 2 gamma 2^(e_i - 61)
            double part = 0.0;
#pragma unroll 1
            for (int hh = 0; hh < 2; ++hh) {
                const int c0 = half * 16 + hh * 8;
                if (nc * FN + c0 >= a.ncols) break;  // no column left (uniform)
                uint32_t G[NSL][8];
                const uint32_t tb = tmem_base + lane_addr + buf * (NSL * FN) + (uint32_t)c0;
#pragma unroll
                for (int g = 0; g < NSL; ++g) tmem_ld8(tb + (uint32_t)(g * FN), G[g]);
#pragma unroll
                for (int g = 0; g < NSL; ++g) tmem_wait8(G[g]);
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    int s[NSL];
#pragma unroll
                    for (int g = 0; g < NSL; ++g) s[g] = __float2int_rn(__uint_as_float(G[g][q]));
                    const long long ih = (long long)(s[0] * 128 + s[1]) * 16384 + (s[2] * 128 + s[3]);
                    const long long il = (long long)(s[4] * 128 + s[5]) * 16384 + (s[6] * 128 + s[7]);
                    const double d = fma(int_to_double(ih), 268435456.0, int_to_double(il));
                    const int j = hh * 8 + q;
                    const double ds = scale2(d, ((const int *)(cb + 32))[j]);  // a_i.a_j 2^(61 - e_i)
                    double kv;
                    if (KIND == DCD_RBF) {
                        double x = fma(rf, ds, -(hr + cb[16 + j]));
                        // -gamma d^2 <= 0, and 0 of a row against itself
                        x = __double2hiint(x) < 0 && ((const int *)(cb + 40))[j] != rid ? x : 0.0;
                        kv = exp_tab(x, tab);
                    } else {
                        const double dot = scale2(ds, er);
                        if (KIND == DCD_LINEAR) {
                            kv = dot;
                        } else {
                            const double t = a.coef0 + dot;
                            kv = t;
                            for (int e = 1; e < a.degree; ++e) kv *= t;
                        }
                    }
                    if (a.out) {
                        const int64_t col = (int64_t)nc * FN + c0 + q;
                        if (row < a.nrows && col < a.ncols) a.out[row * a.ldo + col] = kv;
                    } else {
                        part = fma(kv, cb[j], part);
                    }
                }
            }
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[buf]);
            if (a.out) continue;
            const int64_t prow = (int64_t)a.ntiles * FM;
            a.part[(int64_t)(nc * 2 + half) * prow + row] = part;
            __threadfence();
            __syncwarp();
            unsigned old = 0;
            if (lane == 0) old = atomicAdd(&a.cnt[tile], 1u);
            old = __shfl_sync(0xffffffffu, old, 0);
            if (old == (unsigned)(8 * a.nchunks - 1)) {  // the tile's last warp: its rows' sums in chunk order
                __threadfence();
                for (int q = 0; q < 4; ++q) {
                    const int64_t r = (int64_t)tile * FM + q * 32 + lane;
                    if (r >= a.nrows) continue;
                    double t = 0.0;
                    for (int k = 0; k < 2 * a.nchunks; ++k) t += __ldcg(a.part + (int64_t)k * prow + r);
                    a.g[r] += (a.rs ? a.rs[r] : 1.0) * t;
                }
                if (lane == 0) a.cnt[tile] = 0u;
            }
        }
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
}

// What one value v != 0 of a row with max |a| in [2^(e-1), 2^e) adds to the row's rule: min(|v| 2^-e, 2^-4)
// in units of 2^-25 (x = v 2^(55-e) rounded), and whether v is no multiple of 2^(e-27) (its last four
// slices are not all zero).
// A row's magnitude is spread over its features if the mean of min(|a_k| 2^-e, 2^-4) is at least 9/16 of
// 2^-4.  With t the truncated values of one such row and u those of another, sum t u >= 2^-4 (sum t + sum
// u) - n 2^-8 >= n 2^-11.  Normal, uniform and +-1 features pass from some 16 features on (a normal row's
// mean is 0.9 of 2^-4, 0.8 where its largest value is beyond 4 sigma; 9/16 is 7 and 4 deviations below
// at n = 30).
__device__ __forceinline__ void f64s_row_flags(double v, long long x, int e, long long &mid, bool &lng)
{
    const long long ax = x < 0 ? -x : x;
    mid += (ax < (1LL << 51) ? ax : 1LL << 51) >> 30;
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const int be = (int)(b >> 52) & 2047;
    const unsigned long long mant = (b & 0xfffffffffffffULL) | (be ? 1ULL << 52 : 0ULL);
    if (mant) lng |= (be ? be : 1) - 1075 + __ffsll((long long)mant) - 1 < e - 27;
}

// The eight slices of each row of a dense FP64 matrix (a warp per row, two features per lane), its
// exponent and gamma times its squared norm (compensated sum: TwoProd and TwoSum).  The scaled
// value is rounded once to a 56-bit integer whose signed base-128 digits are the slices.
// stat[0]: F64S_BAD when a value is not finite or an exponent leaves [-400, 400], F64S_UNEVEN when a row's
// magnitude is not spread over its features, F64S_LONG when a row has a value in its last four slices (a
// row of zeros sets neither); stat[1]: the largest gamma |a|^2 and, with the slices, gamma 4^e sqrt(n) / 2
// (bit pattern of a non-negative double).  dst (and ex) null: norms only.
__global__ void pack_f64s_kernel(const double *__restrict__ A, int64_t lda, int64_t m, int64_t n, double gamma,
                                 __nv_bfloat162 *dst, int64_t n_pad, int32_t *ex, double *h, unsigned long long *stat)
{
    const int lane = threadIdx.x & 31;
    const int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (r >= m) return;
    const double *ar = A + r * lda;
    double mx = 0.0, s = 0.0, c = 0.0;
    bool bad = false;
    for (int64_t k = lane; k < n; k += 32) {
        const double v = ar[k];
        bad |= !isfinite(v);
        mx = fmax(mx, fabs(v));
        const double p = v * v, pe = fma(v, v, -p);
        const double t = s + p, z = t - s;
        c += ((s - (t - z)) + (p - z)) + pe;
        s = t;
    }
    for (int o = 16; o > 0; o >>= 1) {
        mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const double s2 = __shfl_xor_sync(0xffffffffu, s, o), c2 = __shfl_xor_sync(0xffffffffu, c, o);
        const double t = s + s2, z = t - s;
        c += ((s - (t - z)) + (s2 - z)) + c2;
        s = t;
    }
    bad = __any_sync(0xffffffffu, bad);
    int e = 0;
    if (!bad && mx > 0.0) frexp(mx, &e);
    bad |= e > 400 || e < -400;
    const double nrm = gamma * (s + c);
    if (lane == 0) {
        if (ex) ex[r] = e;
        h[r] = nrm;
        if (bad) atomicOr(stat, F64S_BAD);
        else {
            const double cut = dst && mx > 0.0 ? ldexp(0.5 * gamma * sqrt((double)n), 2 * e) : 0.0;
            atomicMax(stat + 1, (unsigned long long)__double_as_longlong(fmax(fabs(nrm), cut)));
        }
    }
    if (bad || !dst) return;
    const double sc = __hiloint2double((1023 + 55 - e) << 20, 0);  // 2^(55 - e)
    __nv_bfloat162 *d = dst + r * (NSL / 2) * n_pad;
    long long mid = 0;
    bool lng = false;
    for (int64_t k = 2 * lane; k < n_pad; k += 64) {
        const double v0 = k < n ? ar[k] : 0.0, v1 = k + 1 < n ? ar[k + 1] : 0.0;
        long long x0 = __double2ll_rn(v0 * sc), x1 = __double2ll_rn(v1 * sc);
        f64s_row_flags(v0, x0, e, mid, lng);
        f64s_row_flags(v1, x1, e, mid, lng);
#pragma unroll
        for (int p = NSL - 1; p >= 1; --p) {
            const int d0 = (int)((x0 + 64) & 127) - 64, d1 = (int)((x1 + 64) & 127) - 64;
            x0 = (x0 - d0) >> 7;
            x1 = (x1 - d1) >> 7;
            d[(p * n_pad + k) >> 1] = __floats2bfloat162_rn((float)d0, (float)d1);
        }
        d[k >> 1] = __floats2bfloat162_rn((float)(int)x0, (float)(int)x1);
    }
    for (int o = 16; o > 0; o >>= 1) mid += __shfl_xor_sync(0xffffffffu, mid, o);
    lng = __any_sync(0xffffffffu, lng);
    if (lane == 0 && mx > 0.0) {
        const unsigned long long f = (mid < n * (9LL << 17) ? F64S_UNEVEN : 0) | (lng ? F64S_LONG : 0);
        if ((*(volatile unsigned long long *)stat & f) != f) atomicOr(stat, f);  // the first few rows only
    }
}

template <int KIND>
cudaError_t launch_kind(int grid, const CUtensorMap &mA, const CUtensorMap &mB, const F64Args &a, cudaStream_t st)
{
    // set on every launch: cheap beside the launch, and safe with several devices and threads
    cudaError_t e = cudaFuncSetAttribute(block_f64s_kernel<KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         F64S_SMEM);
    if (e != cudaSuccess) return e;
    block_f64s_kernel<KIND><<<grid, F64S_THREADS, F64S_SMEM, st>>>(mA, mB, a);
    return cudaGetLastError();
}

}  // namespace

int64_t f64s_row_bytes(int64_t n) { return 2 * NSL * ((n + 63) / 64 * 64); }

size_t f64s_part_bytes(int64_t m, int64_t ncols)
{
    const int64_t nc = (ncols < F64S_COLS ? ncols : F64S_COLS);
    return sizeof(double) * (size_t)((nc + FN - 1) / FN) * 2 * (size_t)((m + FM - 1) / FM * FM);
}

int64_t f64s_tiles(int64_t m) { return (m + FM - 1) / FM; }

cudaError_t launch_pack_f64s(const double *A, int64_t lda, int64_t m, int64_t n, const KernelParams &kp, void *packed,
                             int32_t *ex, double *h, unsigned long long *stat, cudaStream_t st)
{
    if (m <= 0 || n <= 0 || (packed && n > F64S_N_MAX)) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemsetAsync(stat, 0, 2 * sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
    pack_f64s_kernel<<<(unsigned)((m * 32 + 255) / 256), 256, 0, st>>>(
        A, lda, m, n, kp.kind == DCD_RBF ? kp.gamma : 0.0, (__nv_bfloat162 *)packed, (n + 63) / 64 * 64, ex, h, stat);
    return cudaGetLastError();
}

cudaError_t launch_block_f64s(const F64Sliced &f, const void *rows, int64_t nrows, const int32_t *row_id,
                              const void *cols, int64_t ncols, const int32_t *col_id, const KernelParams &kp,
                              const double *w, const double *rs, double *g, double *out, int64_t ldo, int *err,
                              cudaStream_t st)
{
    if (nrows <= 0 || ncols <= 0) return cudaSuccess;
    const int64_t n_pad = (f.n + 63) / 64 * 64;
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    }
    CUtensorMap mA, mB;
    if (!make_map_bf16_2d(&mA, rows, NSL * n_pad, nrows, FM)) return cudaErrorInvalidValue;
    for (int64_t c0 = 0; c0 < ncols; c0 += F64S_COLS) {
        const int64_t nc = ncols - c0 < F64S_COLS ? ncols - c0 : F64S_COLS;
        if (!make_map_bf16_2d(&mB, (const char *)cols + c0 * f64s_row_bytes(f.n), NSL * n_pad, nc, FN))
            return cudaErrorInvalidValue;
        F64Args a;
        a.row_id = row_id;
        a.col_id = col_id ? col_id + c0 : nullptr;
        a.ex = f.ex;
        a.h = f.h;
        a.w = w ? w + c0 : nullptr;
        a.rs = rs;
        a.g = g;
        a.out = out ? out + c0 : nullptr;
        a.ldo = ldo;
        a.nrows = nrows;
        a.m = f.m;
        a.ncols = (int)nc;
        a.ntiles = (int)((nrows + FM - 1) / FM);
        a.nchunks = (int)((nc + FN - 1) / FN);
        a.kblocks = (int)(n_pad / 64);
        a.n_pad = n_pad;
        a.two_gamma = 2.0 * kp.gamma;
        a.coef0 = kp.coef0;
        a.degree = kp.degree;
        a.part = f.part;
        a.cnt = f.cnt;
        a.err = err;
        const int64_t units = (int64_t)a.ntiles * a.nchunks;
        const int grid = (int)(units < sms ? units : sms);
        cudaError_t e = kp.kind == DCD_RBF    ? launch_kind<DCD_RBF>(grid, mA, mB, a, st)
                        : kp.kind == DCD_POLY ? launch_kind<DCD_POLY>(grid, mA, mB, a, st)
                                              : launch_kind<DCD_LINEAR>(grid, mA, mB, a, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace dcd
