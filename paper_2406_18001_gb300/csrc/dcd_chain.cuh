// dcd_chain.cuh -- the sequential chain of the s-step DCD recurrence (Algorithm 2), shared by the
// recurrence kernel (recur.cu, which says how it is built) and the resident K-SVM kernel (svm_grid.cu).
#pragma once

#include "dcd_internal.cuh"
#include "ptx.cuh"

namespace dcd {

constexpr int DCD_FAST_MAX = 128;
constexpr int DCD_FAST_K = DCD_FAST_MAX / 32;

__device__ __forceinline__ int ld_acquire_shared(const int *p)
{
    int v;
    asm volatile("ld.acquire.cta.shared::cta.b32 %0, [%1];" : "=r"(v) : "r"(ptx::su32(p)) : "memory");
    return v;
}

__device__ __forceinline__ void st_release_shared(int *p, int v)
{
    asm volatile("st.release.cta.shared::cta.b32 [%0], %1;" ::"r"(ptx::su32(p)), "r"(v) : "memory");
}

// clip(x, 0, nu) by the bit patterns (nub: those of nu, +infinity for no upper bound); a NaN gives 0,
// as fmin(fmax(x, 0), nu) does
__device__ __forceinline__ double clip_bits(double x, long long nub)
{
    const long long b = __double_as_longlong(x);
    if (b <= 0 || b > 0x7ff0000000000000LL) return 0.0;
    return __longlong_as_double(b > nub ? nub : b);
}

// Warp `warp`'s 32 coordinates t = 32 warp + lane of a chain of cnt <= DCD_FAST_MAX: returns the lane's
// step.  C[j ldc + t]: the coupling of t to the step of j < t (zero for t <= j); rep[j DCD_FAST_K +
// q]: bit l set where coordinate 32 q + l > j holds j's row; list_t, list_j (cnt entries) and pub (two
// words, zero at the start): the published steps; rho, gj, ie: alpha_t, g_t, 1 / eta_t (0: no step).
__device__ __forceinline__ double dcd_chain_group(const double *C, int ldc, const uint32_t *rep, double *list_t,
                                                  int *list_j, int *pub, int cnt, int warp, int lane, double rho,
                                                  double gj, double ie, double nu, int *err)
{
    const int t = 32 * warp + lane;
    const bool mine = t < cnt;
    const int tc = mine ? t : cnt - 1;  // a valid column for lanes past the end
    auto apply = [&](int j, double tj) {
        gj = fma(C[j * ldc + tc], tj, gj);
        const uint32_t m = rep[j * DCD_FAST_K + warp];
        if (m) rho += (m >> lane) & 1u ? tj : 0.0;  // repeats are rare (warp-uniform)
    };
    int n = 0;  // published steps applied (or, in the chain below, published)
    if (warp > 0) {
        const long long t0 = clock64();
        for (;;) {
            const int dn = ld_acquire_shared(pub + 1);
            const int np = ld_acquire_shared(pub);
            for (; n < np; ++n) apply(list_j[n], list_t[n]);
            if (dn >= warp) break;
            if (clock64() - t0 > 4200000000LL) {  // about 2 s
                set_error(err, DEV_TIMEOUT);
                break;
            }
        }
        __syncwarp();
    }
    const bool more = 32 * (warp + 1) < cnt;
    const long long nub = __double_as_longlong(nu);
    double th = 0.0;
    uint32_t left = __ballot_sync(0xffffffffu, mine);  // coordinates not yet decided
    const bool solvable = (__double_as_longlong(ie) << 1) != 0;
    for (;;) {
        const double c1 = clip_bits(rho - gj, nub), c2 = clip_bits(fma(-gj, ie, rho), nub);
        // the projected gradient clip(rho - g) - rho is nonzero iff the clip moved rho
        const long long b1 = __double_as_longlong(c1), b0 = __double_as_longlong(rho);
        const bool moved = b1 != b0 && ((b1 | b0) << 1) != 0;  // +0 and -0 are the same value
        const double st = moved && solvable ? c2 - rho : 0.0;
        const uint32_t nz = __ballot_sync(0xffffffffu, (__double_as_longlong(st) << 1) != 0) & left;
        if (!nz) break;
        const int l = __ffs(nz) - 1, j = 32 * warp + l;
        const double tj = __shfl_sync(0xffffffffu, st, l);
        if (lane == l) {
            th = tj;
            if (more) {
                list_j[n] = j;
                list_t[n] = tj;
                st_release_shared(pub, n + 1);
            }
        }
        ++n;
        left &= ~((2u << l) - 1u);
        apply(j, tj);
    }
    __syncwarp();
    if (more && lane == 0) st_release_shared(pub + 1, warp + 1);
    return th;
}

}  // namespace dcd
