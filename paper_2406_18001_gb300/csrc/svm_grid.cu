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
//                      y_i sum_j K(a_i, a_Sj) w_j and alpha on the own rows, publish;
//   block (12 warps)   ahead of it, as it needs the index stream only: four warps fetch the rows of step
//                      q + 1 by asynchronous copies and form this CTA's share of step q's Gram (to
//                      memory, read by all a step later); beside them eight form the own rows' kernel
//                      values against step q's rows, KS lanes an entry, into one of two buffers.
// So the FP64 pipe's work (m s (n + 14) operations a step) runs beside the latencies (L2 round trips,
// chain).  Kernel values: dot products, the RBF from the expansion with compensated norms where
// gamma |a|^2 <= F64S_HMAX for every row, else from coordinate differences; K = 1 on a row's own
// sample.
//
// The exchange is no grid barrier.  A published value is its own signal: the four slots x(k) of xbuf
// take turns, X_OPEN stands in an entry that is not there yet, and the readers poll the entries.  The
// rest is ordered by one counter: a CTA arrives in step k, between its chain and its update, when it has
// read x(k), emptied its share of x(k + 2)'s slot and finished its share of step k + 1's Gram, and
// it begins step k + 1 when all have arrived -- by then mostly long past.  So the couplings may be
// read in step k + 1 (all shares are there), x(k + 2) may be written at its end (all entries are open)
// and the slot of x(k - 2) may be emptied in step k (all have read it).  Barriers with a fence on
// both sides took 4.4 k of a step's 11 k cycles at m = 2000, s = 8.
//
// Measured (FP64, hinge): m = 2000, n = 64, s = 8: 15.3 us a step as long graphs, 5.8 with a grid
// barrier a step, 4.7 now (the FP64 pipe of the own rows' values 3.4 of it); m = 300, n = 16, s = 1 on
// the default stream: 27, 4.5, 3.6 (1 of it host work).
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
constexpr int GX_WARPS = 4, GX = 32 * GX_WARPS, GY = GB - GX;  // block warps of samples and Gram; threads of the own rows' values
constexpr int GRAM_THREADS = GB + 32;  // at NB_GRAM: the block and the main warp that counts arrivals
constexpr size_t GRID_SMEM_MAX = 200 * 1024;
constexpr int GU = GM - 32;  // threads that update; the last main warp counts arrivals meanwhile
constexpr long long GRID_WAIT_CYCLES = 4200000000LL;  // about 2 s: bound on a wait for other CTAs
constexpr long long X_OPEN = -1;  // the bits of an entry that is not published
// kernel-value forms
constexpr int GK_LINEAR = 0, GK_POLY = 1, GK_RBF = 2, GK_RBF_DIRECT = 3;
// named barriers (0 is __syncthreads)
constexpr int NB_MAIN = 1, NB_BLOCK = 2, NB_FULL = 3, NB_FREE = 5, NB_GRAM = 7, NB_UPD = 9, NB_X = 10;  // FULL, FREE, GRAM: + parity

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
    double *xbuf;   // [4][s][2]: g and alpha at the step's coordinates
    double *kss;    // [4][s * s + 2 s] by step (a CTA may be two steps ahead of another's reads): K(S_t, S_j) for j < t at [j * s + t], then 1 / eta_t, eta_t
    unsigned *bar;  // arrivals, zero at the start
    int *err;
};

struct GridLayout {
    size_t own, as, kb, gs, al, hr, hs, yv, C, slot, th, w, tab, ints, total;
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
    L.yv = take(4 * (size_t)s);
    L.C = take((size_t)s * (s | 1));
    L.slot = take(s);
    L.th = take(s);
    L.w = take(s);
    L.tab = take(64);
    L.ints = c;  // S 4 s; sign bits of the own rows' y R; rep 4 s
    L.total = 8 * c + 4 * ((size_t)(4 + DCD_FAST_K) * s + R);
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

__device__ __forceinline__ double x_ld(const double *p)
{
    double v;
    asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void x_st(double *p, double v)
{
    asm volatile("st.relaxed.gpu.global.f64 [%0], %1;" ::"l"(p), "d"(v) : "memory");
}

template <int FORM>
__global__ void __launch_bounds__(GRID_THREADS, 1) svm_grid_kernel(GridArgs a)
{
    extern __shared__ __align__(16) double gsm[];
    const int s = a.s, R = a.R, n = a.n, nls = a.nls, ldc = s | 1;
    const GridLayout L = grid_layout(n, s, R, nls);
    double *own = gsm + L.own, *As = gsm + L.as, *kb = gsm + L.kb, *gs = gsm + L.gs, *al = gsm + L.al,
           *hr = gsm + L.hr, *hS = gsm + L.hs, *yv = gsm + L.yv, *C = gsm + L.C, *slot = gsm + L.slot, *th_s = gsm + L.th, *w_s = gsm + L.w,
           *tab = gsm + L.tab;
    int32_t *SS = (int32_t *)(gsm + L.ints);             // S of a step, by step mod 4
    uint32_t *yr = (uint32_t *)(SS + 4 * s);             // sign bits of the own rows' y
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
        // the sample of step q with its labels and RBF terms; its rows (asynchronous; S is there)
        auto sample = [&](int q) {
            for (int j = bt; j < s; j += GX) {
                const int32_t i = index_of(q, j);
                SS[(q & 3) * s + j] = i;
                ptx::cp_async8(yv + (q & 3) * s + j, a.y + i);
                if (FORM == GK_RBF) ptx::cp_async8(hS + (q & 1) * s + j, a.h + i);
            }
        };
        auto gather = [&](int q) {
            double *Aq = As + (size_t)(q & 1) * s * n;
            const int32_t *Sq = SS + (q & 3) * s;
            for (int j = bw; j < s; j += GX_WARPS) {
                const double *row = a.A + (int64_t)Sq[j] * a.lda;
                for (int c = lane; c < n; c += 32) ptx::cp_async8(Aq + (size_t)j * n + c, row + c);
            }
        };
        const bool is_x = bw < GX_WARPS;
        if (is_x) {
            sample(0);
            nb_sync<GX>(NB_X);
            gather(0);
            ptx::cp_async_wait_all();
        }
        nb_sync<GB>(NB_BLOCK);
        for (int q = 0; q < a.steps; ++q) {
            const int p = q & 1;
            double *Aq = As + (size_t)p * s * n, *kq = kb + (size_t)p * s * R;
            const int32_t *Sq = SS + (q & 3) * s;
            double *hq = hS + p * s;
            if (q >= 2) nb_sync<GRID_THREADS>(NB_FREE + p);  // main is done with step q - 2's buffer
            if (*(volatile int *)&stop_s) break;
            // this CTA's entries of the step's Gram: pairs j <= t, a warp each
            double *kss = a.kss + (size_t)(q & 3) * (s * s + 2 * s);
            if (!is_x) nb_arrive<GRAM_THREADS>(NB_GRAM + p);
            for (int e = cta + G * bw; is_x && e < s * (s + 1) / 2; e += G * GX_WARPS) {
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
            if (is_x) {
                __threadfence();
                nb_arrive<GRAM_THREADS>(NB_GRAM + p);
                if (q + 1 < a.steps) {  // after the Gram, which the other CTAs wait for
                    sample(q + 1);
                    nb_sync<GX>(NB_X);
                    gather(q + 1);
                }
            }
            // the own rows' kernel values against the step's: entry (j, r), ks lanes each
            const int items = s * R * ks;
            for (int e0 = 0; !is_x && e0 < items; e0 += GY) {
                const int e = e0 + bt - GX, l = e & (ks - 1), en = e / ks, j = en / R, r = en - j * R;
                const bool in = e < items && r < rows;
                double v = in ? dot_part<FORM>(own + (size_t)r * nls, Aq + (size_t)j * n, n, l, ks) : 0.0;
                for (int o = ks >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (in) {
                    const double kv = k_value<FORM>(v, hr[r], hq[j], Sq[j] == r0 + r, a, tab);
                    if (l == 0) kq[j * R + r] = kv;
                }
            }
            nb_arrive<GRID_THREADS>(NB_FULL + p);
            if (is_x) ptx::cp_async_wait_all();  // step q + 1's rows
            nb_sync<GB>(NB_BLOCK);
        }
        return;
    }

    // ---------------------------------------------------------------- main --
    const int ng = (s + 31) / 32;
    auto give_up = [&] {
        set_error(a.err, DEV_TIMEOUT);
        stop_s = 1;
    };
    auto publish = [&](int k) {  // the own rows' alpha and g at step k's coordinates
        for (int j = tid; j < s; j += GU) {
            const int32_t i = SS[(k & 3) * s + j];
            if (i >= r0 && i < r0 + rows) {
                double *x = a.xbuf + ((size_t)(k & 3) * s + j) * 2;
                const double v[2] = {gs[i - r0], al[i - r0]};
                for (int u = 0; u < 2; ++u)  // a NaN that looks like an open entry: another one
                    x_st(x + u, __double_as_longlong(v[u]) == X_OPEN ? __longlong_as_double(X_OPEN - 1) : v[u]);
            }
        }
    };
    // one thread: this CTA's arrival number k (from 0), and the wait until every CTA has made it
    auto arrive = [&](int k) {
        asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(a.bar), "r"(1u) : "memory");
        const unsigned want = (unsigned)G * (unsigned)(k + 1);
        const long long c0 = clock64();
        for (;;) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a.bar) : "memory");
            if ((int)(v - want) >= 0) break;
            if (clock64() - c0 > GRID_WAIT_CYCLES) {
                give_up();
                break;
            }
        }
    };
    // lanes per row of the update
    int nls2 = 0;  // their log2
    while (nls2 < 5 && (2 << nls2) <= s && (2 << nls2) * R <= GU) ++nls2;
    const int nl = 1 << nls2;
    if (warp == GM_WARPS - 1) nb_sync<GRAM_THREADS>(NB_GRAM);
    nb_sync<GM>(NB_MAIN);
    if (warp == GM_WARPS - 1) {
        if (lane == 0) arrive(0);
        __syncwarp();
    } else {
        publish(0);
    }
    bool ok = true;
    int k = 0;
    for (; k < a.steps; ++k) {
        const int p = k & 1;
        const int32_t *S = SS + (k & 3) * s;
        const double *yk = yv + (k & 3) * s;
        auto ysign = [&](int t) { return (uint32_t)__double2hiint(yk[t]) & 0x80000000u; };
        const double *kss = a.kss + (size_t)(k & 3) * (s * s + 2 * s);
        double rho = 0.0, gj = 0.0, ie = 0.0, eta = 0.0;
        if (tid < s) {
            const double *x = a.xbuf + ((size_t)(k & 3) * s + tid) * 2;
            const long long c0 = clock64();
            for (;;) {
                gj = x_ld(x);
                rho = x_ld(x + 1);
                if (__double_as_longlong(gj) != X_OPEN && __double_as_longlong(rho) != X_OPEN) break;
                if (clock64() - c0 > GRID_WAIT_CYCLES) {
                    give_up();
                    break;
                }
            }
        }
        nb_sync<GM>(NB_MAIN);
        if (*(volatile int *)&stop_s) {  // the same in every main thread: it changes between barriers only
            ok = false;
            break;
        }
        if (k + 2 < a.steps)
            for (int j = cta + G * tid; j < s; j += G * GM) {
                double *x = a.xbuf + ((size_t)((k + 2) & 3) * s + j) * 2;
                x_st(x, __longlong_as_double(X_OPEN));
                x_st(x + 1, __longlong_as_double(X_OPEN));
            }
        if (tid < s) {
            ie = __ldcg(kss + s * s + tid);
            eta = __ldcg(kss + s * s + s + tid);
            slot[tid] = __longlong_as_double(CHAIN_OPEN);
        }
        constexpr int U = 4;  // rows' couplings in flight
        for (int q = 0; q < ng; ++q) {
            const int t = 32 * q + lane;
            const uint32_t yt = t < s ? ysign(t) : 0u;
            const int32_t St = t < s ? S[t] : -1;
            for (int j0 = warp; j0 < s; j0 += GM_WARPS * U) {
                double v[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int j = j0 + GM_WARPS * u;
                    v[u] = j < s && t < s && t > j ? __ldcg(kss + j * s + t) : 0.0;
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int j = j0 + GM_WARPS * u;
                    if (j >= s) break;  // warp-uniform
                    const bool later = t < s && t > j, same = later && St == S[j];
                    double c = __hiloint2double((int)((uint32_t)__double2hiint(v[u]) ^ (later ? yt ^ ysign(j) : 0u)),
                                                __double2loint(v[u]));
                    if (same) c += a.omega;
                    if (t < s) C[j * ldc + t] = c;
                    const uint32_t mask = __ballot_sync(0xffffffffu, same);
                    if (lane == 0) rep[j * DCD_FAST_K + q] = mask;
                }
            }
        }
        nb_sync<GM>(NB_MAIN);
        if (warp < ng) {
            const double th = dcd_chain_group(C, ldc, rep, slot, s, warp, lane, rho, gj, eta, ie, a.nu, a.err);
            if (tid < s) {
                th_s[tid] = th;
                w_s[tid] = __hiloint2double((int)((uint32_t)__double2hiint(th) ^ ysign(tid)), __double2loint(th));
            }
        }
        nb_sync<GM>(NB_MAIN);
        nb_sync<GRID_THREADS>(NB_FULL + p);  // the own rows' kernel values are there
        if (warp == GM_WARPS - 1) {
            if (k + 1 < a.steps) {
                nb_sync<GRAM_THREADS>(NB_GRAM + (p ^ 1));
                if (lane == 0) arrive(k + 1);
            }
            __syncwarp();
        } else {
            const double *kq = kb + (size_t)p * s * R;
            for (int e0 = 32 * warp; e0 < R * nl; e0 += GU) {  // nl lanes per own row
                const int r = (e0 + lane) >> nls2, l = (e0 + lane) & (nl - 1);
                const bool in = r < rows;
                double v = 0.0, own = 0.0;
                bool hit = false;
                for (int j = l; j < s; j += nl) {
                    if (in) v = fma(kq[j * R + r], w_s[j], v);
                    if (in && S[j] == r0 + r) {
                        own += th_s[j];
                        hit = true;
                    }
                }
                for (int o = nl >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (__any_sync(0xffffffffu, hit))
                    for (int o = nl >> 1; o > 0; o >>= 1) {
                        own += __shfl_xor_sync(0xffffffffu, own, o);
                        hit |= __shfl_xor_sync(0xffffffffu, (int)hit, o) != 0;
                    }
                if (in && l == 0) {
                    v = __hiloint2double((int)((uint32_t)__double2hiint(v) ^ yr[r]), __double2loint(v));  // y_r
                    double gn = gs[r] + v;
                    if (hit) {  // this row's own steps
                        al[r] += own;
                        gn += a.omega * own;
                    }
                    gs[r] = gn;
                }
            }
            nb_sync<GU>(NB_UPD);
            if (k + 1 < a.steps) publish(k + 1);
        }
        if (k + 2 < a.steps) nb_arrive<GRID_THREADS>(NB_FREE + p);
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
    while (ks < 8 && 2 * ks * R * s <= GY && 8 * ks <= n) ks *= 2;
    g.R = R;
    g.ks = ks;
    g.ctas = (int)((m + R - 1) / R);
    g.smem = smem;
    // A launch of some 60 ms at most, so that what is queued behind it gets its turn: a step takes less than
    // 4 us, 0.4 us a coordinate of the chain, and m s (2 n + 40) FP64 operations (distances from
    // differences) at the pipe's 0.46 M a us.  m = 3500, n = 600, s = 8: 725 steps a launch, 22 ms, 46 with
    // distances from differences (4096 took 126 and 262); m = 2000, n = 64, s = 8: 4096 steps, 18 and 26 ms.
    const double us = 4.0 + 0.4 * s + (double)m * s * (2.0 * (double)n + 40.0) / 0.46e6;
    g.steps = std::min<int64_t>(std::max<int64_t>((int64_t)(60000.0 / us), 1), 4096);
    return g;
}

size_t svm_grid_scratch_bytes(int s) { return sizeof(double) * (8 * (size_t)s + 4 * ((size_t)s * s + 2 * s)) + 256; }

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
    a.kss = a.xbuf + 8 * (size_t)s;
    a.err = err;
    cudaError_t e = cudaMemsetAsync(a.bar, 0, sizeof(unsigned), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(a.xbuf, 0xff, sizeof(double) * 8 * (size_t)s, st);  // X_OPEN
    if (e != cudaSuccess) return e;
    if (kp.kind == DCD_LINEAR) return launch_form<GK_LINEAR>(a, gp.ctas, gp.smem, st);
    if (kp.kind == DCD_POLY) return launch_form<GK_POLY>(a, gp.ctas, gp.smem, st);
    return h ? launch_form<GK_RBF>(a, gp.ctas, gp.smem, st) : launch_form<GK_RBF_DIRECT>(a, gp.ctas, gp.smem, st);
}

}  // namespace dcd
