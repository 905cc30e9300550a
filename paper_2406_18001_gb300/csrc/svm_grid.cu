// svm_grid.cu -- resident K-SVM steps: the outer s-steps of Algorithm 2 on a small dense FP64 problem,
// many per launch, on one co-resident grid.
//
// A step of a small problem is a chain of latencies (sample, Gram, recurrence, block, update), and as
// kernels each link adds its launch: 18 us a step at m = 2000, n = 64, s = 8 as replayed graphs, 27 us
// at m = 300, n = 16, s = 1 as direct launches, for a few microseconds of FP64 work.  Here CTA c owns
// rows c R .. c R + R - 1 with their values, labels, alpha and g in shared memory, and a step needs one
// exchange: the owners of the next step's coordinates publish alpha and g at them (2 s doubles), every
// CTA runs the recurrence on them for itself and updates its own rows.  Two groups of warps run beside
// each other in a CTA:
//   main (4 warps)     step k: read the exchange and the couplings, the chain (dcd_chain.cuh), g_i +=
//                      y_i sum_j K(a_i, a_Sj) w_j and alpha on the own rows, publish, grid barrier;
//   block (12 warps)   ahead of it, as it needs the index stream only: the rows of step q, this CTA's
//                      share of its Gram (to memory, read by all a step later) and the own rows' kernel
//                      values against them, KS lanes an entry, into one of two buffers.
// So the FP64 pipe's work (m s (n + 14) operations a step) runs beside the latencies (barrier, L2
// read, chain).  Kernel values: dot products, the RBF from the expansion with compensated norms where
// gamma |a|^2 <= F64S_HMAX for every row, else from coordinate differences; K = 1 on a row's own
// sample.
//
// Measured (FP64, hinge): m = 2000, n = 64, s = 8: 15.3 us a step as long graphs -> 5.6; m = 300,
// n = 16, s = 1 on the default stream: 27 -> 4.1.
#include "dcd_chain.cuh"
#include "dcd_internal.cuh"
#include "f64_math.cuh"
#include "ptx.cuh"

#include <algorithm>

namespace dcd {

namespace {

constexpr int GM_WARPS = 4, GB_WARPS = 12;  // main and block warps
constexpr int GM = 32 * GM_WARPS, GB = 32 * GB_WARPS;
constexpr int GRID_THREADS = GM + GB;
constexpr size_t GRID_SMEM_MAX = 200 * 1024;
constexpr long long GRID_WAIT_CYCLES = 4200000000LL;  // about 2 s: bound on a wait at the grid barrier
// kernel-value forms
constexpr int GK_LINEAR = 0, GK_POLY = 1, GK_RBF = 2, GK_RBF_DIRECT = 3;
// named barriers (0 is __syncthreads)
constexpr int NB_MAIN = 1, NB_BLOCK = 2, NB_FULL = 3, NB_FREE = 5, NB_GRAM = 7;  // the last three + parity

struct GridArgs {
    const double *A;
    int64_t lda;
    int m, n;
    KernelParams kp;
    const double *h;  // gamma |a|^2 (RBF, expansion)
    const double *y;
    double *alpha, *g;
    uint64_t seed;
    uint64_t *ctr;
    int steps, s, R, ks, nls;  // rows per CTA, lanes per entry, row stride in shared memory
    double omega, nu;
    double *xbuf;   // [2][s][2]: g and alpha at the step's coordinates
    double *kss;    // [4][s * s + 2 s] by step (a CTA may be two steps ahead of another's reads): K(S_t, S_j) for j < t at [j * s + t], then 1 / eta_t, eta_t
    unsigned *bar;  // arrivals, zero at the start
    int *err;
};

struct GridLayout {
    size_t own, as, kb, gs, al, hr, hs, C, slot, th, w, tab, ints, total;
};

__host__ __device__ inline GridLayout grid_layout(int n, int s, int R, int nls)
{
    GridLayout L;
    size_t c = 0;
    auto take = [&](size_t doubles) {
        const size_t o = c;
        c += doubles;
        return o;
    };
    L.own = take((size_t)R * nls);
    L.as = take(2 * (size_t)s * n);
    L.kb = take(2 * (size_t)s * R);
    L.gs = take(R);
    L.al = take(R);
    L.hr = take(R);
    L.hs = take(2 * (size_t)s);
    L.C = take((size_t)s * (s | 1));
    L.slot = take(s);
    L.th = take(s);
    L.w = take(s);
    L.tab = take(64);
    L.ints = c;  // S 2 s; sign of y: at S 2 s, own rows R; rep 4 s
    L.total = 8 * c + 4 * ((size_t)(2 + 2 + DCD_FAST_K) * s + R);
    return L;
}

template <int N> __device__ __forceinline__ void nb_sync(int id)
{
    asm volatile("barrier.cta.sync %0, %1;" ::"r"(id), "n"(N) : "memory");
}
template <int N> __device__ __forceinline__ void nb_arrive(int id)
{
    asm volatile("barrier.cta.arrive %0, %1;" ::"r"(id), "n"(N) : "memory");
}

// sum over k = l0, l0 + stride, ... of a product or a squared difference of two rows
template <int FORM>
__device__ __forceinline__ double dot_part(const double *a, const double *b, int n, int l0, int stride)
{
    double s0 = 0.0, s1 = 0.0;
    int k = l0;
    for (; k + stride < n; k += 2 * stride) {
        if (FORM == GK_RBF_DIRECT) {
            const double d0 = a[k] - b[k], d1 = a[k + stride] - b[k + stride];
            s0 = fma(d0, d0, s0);
            s1 = fma(d1, d1, s1);
        } else {
            s0 = fma(a[k], b[k], s0);
            s1 = fma(a[k + stride], b[k + stride], s1);
        }
    }
    if (k < n) {
        if (FORM == GK_RBF_DIRECT) {
            const double d = a[k] - b[k];
            s0 = fma(d, d, s0);
        } else {
            s0 = fma(a[k], b[k], s0);
        }
    }
    return s0 + s1;
}

template <int FORM>
__device__ __forceinline__ double k_value(double v, double hi, double hj, bool own, const GridArgs &a, const double *tab)
{
    if (FORM == GK_LINEAR) return v;
    if (FORM == GK_POLY) {
        const double t = a.kp.coef0 + v;
        double r = t;
        for (int e = 1; e < a.kp.degree; ++e) r *= t;
        return r;
    }
    if (FORM == GK_RBF_DIRECT) return exp(-a.kp.gamma * v);
    double x = fma(2.0 * a.kp.gamma, v, -(hi + hj));
    x = own || __double2hiint(x) >= 0 ? 0.0 : x;
    return exp_tab(x, tab);
}

template <int FORM>
__global__ void __launch_bounds__(GRID_THREADS, 1) svm_grid_kernel(GridArgs a)
{
    extern __shared__ __align__(16) double gsm[];
    const int s = a.s, R = a.R, n = a.n, nls = a.nls, ldc = s | 1;
    const GridLayout L = grid_layout(n, s, R, nls);
    double *own = gsm + L.own, *As = gsm + L.as, *kb = gsm + L.kb, *gs = gsm + L.gs, *al = gsm + L.al,
           *hr = gsm + L.hr, *hS = gsm + L.hs, *C = gsm + L.C, *slot = gsm + L.slot, *th_s = gsm + L.th, *w_s = gsm + L.w,
           *tab = gsm + L.tab;
    int32_t *SS = (int32_t *)(gsm + L.ints);             // S of a step, by its parity
    uint32_t *sy = (uint32_t *)(SS + 2 * s);             // sign bits of y at S, by parity
    uint32_t *yr = sy + 2 * s;                           // sign bits of the own rows' y
    uint32_t *rep = yr + R;
    __shared__ int stop_s;                               // the grid barrier's wait ran out
    const int cta = blockIdx.x, G = gridDim.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int r0 = cta * R, rows = max(min(R, a.m - r0), 0);
    const uint64_t t0 = *a.ctr;

    for (int e = tid; e < rows * n; e += GRID_THREADS) own[e / n * nls + e % n] = a.A[(int64_t)(r0 + e / n) * a.lda + e % n];
    for (int r = tid; r < rows; r += GRID_THREADS) {
        gs[r] = a.g[r0 + r];
        al[r] = a.alpha[r0 + r];
        yr[r] = (uint32_t)__double2hiint(a.y[r0 + r]) & 0x80000000u;
        hr[r] = FORM == GK_RBF ? a.h[r0 + r] : 0.0;
    }
    if (FORM == GK_RBF && tid < 64) tab[tid] = exp_tab_entry(tid);
    if (tid == 0) stop_s = 0;
    auto index_of = [&](int k, int j) {  // coordinate j of step k
        return (int32_t)below(sm64_draw(a.seed, 0, t0 + (uint64_t)k * s + (uint64_t)j), (uint64_t)a.m);
    };
    __syncthreads();

    if (warp >= GM_WARPS) {
        // ----------------------------------------------------------- block --
        const int bt = tid - GM, bw = warp - GM_WARPS, ks = a.ks;
        for (int q = 0; q < a.steps; ++q) {
            const int p = q & 1;
            double *Aq = As + (size_t)p * s * n, *kq = kb + (size_t)p * s * R;
            int32_t *Sq = SS + p * s;
            double *hq = hS + p * s;
            if (q >= 2) nb_sync<GRID_THREADS>(NB_FREE + p);  // main is done with step q - 2's buffer
            if (*(volatile int *)&stop_s) break;
            for (int j = bt; j < s; j += GB) {
                const int32_t i = index_of(q, j);
                Sq[j] = i;
                sy[p * s + j] = (uint32_t)__double2hiint(a.y[i]) & 0x80000000u;
                hq[j] = FORM == GK_RBF ? a.h[i] : 0.0;
            }
            nb_sync<GB>(NB_BLOCK);
            for (int e = bt; e < s * n; e += GB) Aq[e] = a.A[(int64_t)Sq[e / n] * a.lda + e % n];
            nb_sync<GB>(NB_BLOCK);
            // this CTA's entries of the step's Gram: pairs j <= t, a warp each
            double *kss = a.kss + (size_t)(q & 3) * (s * s + 2 * s);
            for (int e = cta + G * bw; e < s * (s + 1) / 2; e += G * GB_WARPS) {
                int t = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
                while (t * (t + 1) / 2 > e) --t;
                while ((t + 1) * (t + 2) / 2 <= e) ++t;
                const int j = e - t * (t + 1) / 2;
                double v = dot_part<FORM>(Aq + (size_t)t * n, Aq + (size_t)j * n, n, lane, 32);
                for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                const int st = Sq[t], sj = Sq[j];
                const double kv = k_value<FORM>(v, hq[t], hq[j], st == sj, a, tab);
                if (lane == 0) {
                    if (j < t) {
                        kss[j * s + t] = kv;
                    } else {
                        const double eta = kv + a.omega;  // G_k = V^T U_k + omega I, y_t^2 = 1
                        kss[s * s + t] = eta > 0.0 ? 1.0 / eta : 0.0;
                        kss[s * s + s + t] = eta;
                    }
                }
            }
            __threadfence();
            nb_arrive<GRID_THREADS>(NB_GRAM + p);
            // the own rows' kernel values against the step's: entry (j, r), ks lanes each
            const int items = s * R * ks;
            for (int e0 = 0; e0 < items; e0 += GB) {
                const int e = e0 + bt, l = e & (ks - 1), en = e / ks, j = en / R, r = en - j * R;
                const bool in = e < items && r < rows;
                double v = in ? dot_part<FORM>(own + (size_t)r * nls, Aq + (size_t)j * n, n, l, ks) : 0.0;
                for (int o = ks >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (in) {
                    const double kv = k_value<FORM>(v, hr[r], hq[j], Sq[j] == r0 + r, a, tab);
                    if (l == 0) kq[j * R + r] = kv;
                }
            }
            nb_arrive<GRID_THREADS>(NB_FULL + p);
        }
        return;
    }

    // ---------------------------------------------------------------- main --
    const int ng = (s + 31) / 32;
    auto publish = [&](int k) {  // the own rows' alpha and g at step k's coordinates
        const int p = k & 1;
        for (int j = tid; j < s; j += GM) {
            const int32_t i = SS[p * s + j];
            if (i >= r0 && i < r0 + rows) {
                double *x = a.xbuf + ((size_t)p * s + j) * 2;
                x[0] = gs[i - r0];
                x[1] = al[i - r0];
            }
        }
    };
    auto grid_barrier = [&](int k) -> bool {  // every CTA is past its publish(k)
        nb_sync<GM>(NB_MAIN);
        if (tid == 0) {
            __threadfence();
            const unsigned want = (unsigned)G * (unsigned)(k + 1);
            atomicAdd(a.bar, 1u);
            const long long c0 = clock64();
            unsigned v;
            for (;;) {
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a.bar) : "memory");
                if ((int)(v - want) >= 0) break;
                if (clock64() - c0 > GRID_WAIT_CYCLES) {
                    set_error(a.err, DEV_TIMEOUT);
                    stop_s = 1;
                    break;
                }
            }
            __threadfence();
        }
        nb_sync<GM>(NB_MAIN);
        return !*(volatile int *)&stop_s;
    };
    nb_sync<GRID_THREADS>(NB_GRAM);
    publish(0);
    bool ok = grid_barrier(0);
    int k = 0;
    for (; ok && k < a.steps; ++k) {
        const int p = k & 1;
        const int32_t *S = SS + p * s;
        const uint32_t *yk = sy + p * s;
        const double *kss = a.kss + (size_t)(k & 3) * (s * s + 2 * s);
        double rho = 0.0, gj = 0.0, ie = 0.0, eta = 0.0;
        if (tid < s) {
            const double *x = a.xbuf + ((size_t)p * s + tid) * 2;
            gj = __ldcg(x);
            rho = __ldcg(x + 1);
            ie = __ldcg(kss + s * s + tid);
            eta = __ldcg(kss + s * s + s + tid);
            slot[tid] = __longlong_as_double(CHAIN_OPEN);
        }
        for (int j = warp; j < s; j += GM_WARPS)
            for (int q = 0; q < ng; ++q) {
                const int t = 32 * q + lane;
                const bool later = t < s && t > j;
                const bool same = later && S[later ? t : 0] == S[j];
                double v = later ? __ldcg(kss + j * s + t) : 0.0;
                v = __hiloint2double((int)((uint32_t)__double2hiint(v) ^ (later ? yk[t] ^ yk[j] : 0u)), __double2loint(v));
                if (same) v += a.omega;
                if (t < s) C[j * ldc + t] = v;
                const uint32_t mask = __ballot_sync(0xffffffffu, same);
                if (lane == 0) rep[j * DCD_FAST_K + q] = mask;
            }
        nb_sync<GM>(NB_MAIN);
        if (warp < ng) {
            const double th = dcd_chain_group(C, ldc, rep, slot, s, warp, lane, rho, gj, eta, ie, a.nu, a.err);
            if (tid < s) {
                th_s[tid] = th;
                w_s[tid] = __hiloint2double((int)((uint32_t)__double2hiint(th) ^ yk[tid]), __double2loint(th));
            }
        }
        nb_sync<GM>(NB_MAIN);
        nb_sync<GRID_THREADS>(NB_FULL + p);  // the own rows' kernel values are there
        const double *kq = kb + (size_t)p * s * R;
        for (int r = tid; r < rows; r += GM) {
            double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0, sum = 0.0;
            bool mine = false;
            int j = 0;
            for (; j + 3 < s; j += 4) {
                s0 = fma(kq[j * R + r], w_s[j], s0);
                s1 = fma(kq[(j + 1) * R + r], w_s[j + 1], s1);
                s2 = fma(kq[(j + 2) * R + r], w_s[j + 2], s2);
                s3 = fma(kq[(j + 3) * R + r], w_s[j + 3], s3);
                mine |= S[j] == r0 + r || S[j + 1] == r0 + r || S[j + 2] == r0 + r || S[j + 3] == r0 + r;
            }
            for (; j < s; ++j) {
                s0 = fma(kq[j * R + r], w_s[j], s0);
                mine |= S[j] == r0 + r;
            }
            double v = (s0 + s1) + (s2 + s3);
            v = __hiloint2double((int)((uint32_t)__double2hiint(v) ^ yr[r]), __double2loint(v));  // y_r
            double gn = gs[r] + v;
            if (mine) {  // this row's own steps, in position order
                for (j = 0; j < s; ++j)
                    if (S[j] == r0 + r) sum += th_s[j];
                al[r] += sum;
                gn += a.omega * sum;
            }
            gs[r] = gn;
        }
        if (k + 2 < a.steps) nb_arrive<GRID_THREADS>(NB_FREE + p);
        if (k + 1 < a.steps) {
            nb_sync<GM>(NB_MAIN);
            nb_sync<GRID_THREADS>(NB_GRAM + (p ^ 1));
            publish(k + 1);
            ok = grid_barrier(k + 1);
        }
    }
    nb_sync<GM>(NB_MAIN);
    for (int r = tid; r < rows; r += GM) {
        a.g[r0 + r] = gs[r];
        a.alpha[r0 + r] = al[r];
    }
    if (cta == 0 && tid == 0) *a.ctr = t0 + (uint64_t)k * (uint64_t)s;
    // a wait that ran out: the block warps may be at their next buffer; let them see the stop
    if (!ok && k + 2 < a.steps) nb_arrive<GRID_THREADS>(NB_FREE + (k & 1));
}

template <int FORM>
cudaError_t launch_form(const GridArgs &a, int G, size_t smem, cudaStream_t st)
{
    auto kfn = svm_grid_kernel<FORM>;
    cudaError_t e = cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GRID_SMEM_MAX);
    if (e != cudaSuccess) return e;
    GridArgs args = a;
    void *p[] = {&args};
    return cudaLaunchCooperativeKernel((const void *)kfn, dim3((unsigned)G), dim3(GRID_THREADS), p, smem, st);
}

}  // namespace

SvmGrid svm_grid_plan(int64_t m, int64_t n, int s)
{
    SvmGrid g;
    if (s < 1 || s > DCD_FAST_MAX || n < 1 || n > 4096 || m < 1 || m > (1 << 24)) return g;
    int dev = 0, sms = 0, coop = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return g;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (!coop || sms < 1) return g;
    // as many CTAs as leave each at least 32 entries a step: fewer meet at a barrier sooner
    const int R = (int)std::max<int64_t>((m + sms - 1) / sms, (32 + s - 1) / s);
    const int nls = (int)n | 1;
    const size_t smem = grid_layout((int)n, s, R, nls).total;
    if (smem > GRID_SMEM_MAX) return g;
    int ks = 1;
    while (ks < 8 && 2 * ks * R * s <= GB && 8 * ks <= n) ks *= 2;
    g.R = R;
    g.ks = ks;
    g.ctas = (int)((m + R - 1) / R);
    g.smem = smem;
    return g;
}

size_t svm_grid_scratch_bytes(int s) { return sizeof(double) * (4 * (size_t)s + 4 * ((size_t)s * s + 2 * s)) + 256; }

cudaError_t launch_svm_grid(const SvmGrid &gp, const double *A, int64_t lda, int64_t m, int64_t n,
                            const KernelParams &kp, const double *h, const double *y, double *alpha, double *g,
                            uint64_t seed, uint64_t *ctr, int steps, int s, double omega, double nu, void *scratch,
                            int *err, cudaStream_t st)
{
    if (steps <= 0) return cudaSuccess;
    GridArgs a;
    a.A = A;
    a.lda = lda;
    a.m = (int)m;
    a.n = (int)n;
    a.kp = kp;
    a.h = h;
    a.y = y;
    a.alpha = alpha;
    a.g = g;
    a.seed = seed;
    a.ctr = ctr;
    a.steps = steps;
    a.s = s;
    a.R = gp.R;
    a.ks = gp.ks;
    a.nls = (int)n | 1;
    a.omega = omega;
    a.nu = nu;
    a.bar = (unsigned *)scratch;
    a.xbuf = (double *)((char *)scratch + 256);
    a.kss = a.xbuf + 4 * (size_t)s;
    a.err = err;
    cudaError_t e = cudaMemsetAsync(a.bar, 0, sizeof(unsigned), st);
    if (e != cudaSuccess) return e;
    if (kp.kind == DCD_LINEAR) return launch_form<GK_LINEAR>(a, gp.ctas, gp.smem, st);
    if (kp.kind == DCD_POLY) return launch_form<GK_POLY>(a, gp.ctas, gp.smem, st);
    return h ? launch_form<GK_RBF>(a, gp.ctas, gp.smem, st) : launch_form<GK_RBF_DIRECT>(a, gp.ctas, gp.smem, st);
}

}  // namespace dcd
