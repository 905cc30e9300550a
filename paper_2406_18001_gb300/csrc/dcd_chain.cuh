// dcd_chain.cuh -- the sequential chain of the s-step DCD recurrence (Algorithm 2), shared by the
// recurrence kernel (recur.cu, which says how it is built) and the resident K-SVM kernel (svm_grid.cu).
#pragma once

#include "dcd_internal.cuh"
#include "ptx.cuh"

namespace dcd {

constexpr int DCD_FAST_MAX = 128;
constexpr int DCD_FAST_K = DCD_FAST_MAX / 32;

// a step that is not decided yet: a signalling NaN, which no FP64 operation returns
constexpr long long CHAIN_OPEN = 0x7ff4000000000000LL;

__device__ __forceinline__ double chain_ld(const double *p)
{
    double v;
    asm volatile("ld.volatile.shared.f64 %0, [%1];" : "=d"(v) : "r"(ptx::su32(p)) : "memory");
    return v;
}

__device__ __forceinline__ void chain_st(double *p, double v)
{
    asm volatile("st.volatile.shared.f64 [%0], %1;" ::"r"(ptx::su32(p)), "d"(v) : "memory");
}

// clip(x, 0, nu) by the bit patterns (nub: those of nu, +infinity for no upper bound); a NaN gives 0,
// as fmin(fmax(x, 0), nu) does
__device__ __forceinline__ double clip_bits(double x, long long nub)
{
    const long long b = __double_as_longlong(x);
    if (b <= 0 || b > 0x7ff0000000000000LL) return 0.0;
    return __longlong_as_double(b > nub ? nub : b);
}

// The chain of one group.  SCALED (each eta in [2^-20, 2^300], a usual nu): the lane keeps u = eta_t
// alpha_t - g_t, so a round on the critical path is one FMA into u, the clip of u to [0, eta nu] by
// integer compares, a ballot (the step is nonzero iff the clip differs from eta alpha_t) and, beside
// the ballot, one FMA to the step clip(u) / eta - alpha: 0.15 us a round.
// Otherwise the candidate steps are formed as Algorithm 2 writes them, with three more FP64
// instructions a round: rho - g, rho - g / eta, and the difference to rho (0.38 us).
template <bool SCALED>
__device__ __forceinline__ double dcd_chain_run(const double *C, int ldc, const uint32_t *rep, double *slot, int cnt,
                                                int warp, int lane, double rho, double gj, double eta, double ie,
                                                double nu, int *err)
{
    const int t = 32 * warp + lane;
    const bool mine = t < cnt;
    const int tc = mine ? t : cnt - 1;  // a valid column for lanes past the end
    double re = rho * eta, x = SCALED ? fma(rho, eta, -gj) : gj;
    auto repeat = [&](double tj) {  // an earlier coordinate with this one's index moved
        rho += tj;
        if (SCALED) {
            re = rho * eta;
            x = fma(eta, tj, x);
        }
    };
    if (warp > 0) {  // the earlier groups' steps, as they are published, in order
        const long long t0 = clock64();
        int spins = 0;
        for (int g = 0; g < warp; ++g) {
            const uint32_t row = rep[(32 * g + lane) * DCD_FAST_K + warp];
            const bool any = __any_sync(0xffffffffu, row != 0);
            for (uint32_t seen = 0; seen != 0xffffffffu;) {
                const double v = chain_ld(slot + 32 * g + lane);
                const uint32_t open = __ballot_sync(0xffffffffu, __double_as_longlong(v) == CHAIN_OPEN);
                const uint32_t ready = (open & (0u - open)) - 1u;  // those below the first open one
                if (ready == seen) {
                    if ((++spins & 255) == 0 && __any_sync(0xffffffffu, clock64() - t0 > 4200000000LL)) {  // about 2 s
                        if (lane == 0) set_error(err, DEV_TIMEOUT);
                        return 0.0;
                    }
                    continue;
                }
                uint32_t nz = __ballot_sync(0xffffffffu, (__double_as_longlong(v) << 1) != 0) & ready & ~seen;
                seen = ready;
                while (nz) {
                    const int l = __ffs(nz) - 1;
                    nz &= nz - 1;
                    const double tj = __shfl_sync(0xffffffffu, v, l), c = C[(32 * g + l) * ldc + tc];
                    x = fma(SCALED ? -c : c, tj, x);
                    if (any && (__shfl_sync(0xffffffffu, row, l) >> lane) & 1u) repeat(tj);
                }
            }
        }
    }
    const bool more = 32 * (warp + 1) < cnt;
    const uint32_t own = mine ? rep[t * DCD_FAST_K + warp] : 0u;  // row t's repeats within the group
    const bool any = __any_sync(0xffffffffu, own != 0);
    const long long nub = __double_as_longlong(SCALED ? nu * eta : nu);
    double th = 0.0;
    uint32_t left = __ballot_sync(0xffffffffu, mine && ie > 0.0);  // coordinates not yet decided
    int told = 0;                                                  // coordinates published
    for (;;) {
        double st;
        bool moved;
        if (SCALED) {
            const long long b = __double_as_longlong(x);
            const bool lo = (uint32_t)__double2hiint(x) > 0x7ff00000u;  // negative, or a NaN
            const bool hi = b >= nub;
            moved = (lo ? 0LL : hi ? nub : b) != __double_as_longlong(re);
            st = fma(lo ? 0.0 : hi ? nu : x, hi ? 1.0 : ie, -rho);
        } else {
            const double c1 = clip_bits(rho - x, nub), c2 = clip_bits(fma(-x, ie, rho), nub);
            // the projected gradient clip(rho - g) - rho is nonzero iff the clip moved rho
            st = __double_as_longlong(c1) != __double_as_longlong(rho) ? c2 - rho : 0.0;
            moved = (__double_as_longlong(st) << 1) != 0;
        }
        const uint32_t nz = __ballot_sync(0xffffffffu, moved) & left;
        if (!nz) break;
        const int l = __ffs(nz) - 1, j = 32 * warp + l;
        const double tj = __shfl_sync(0xffffffffu, st, l), c = C[j * ldc + tc];
        x = fma(SCALED ? -c : c, tj, x);
        left &= ~((2u << l) - 1u);
        th = lane == l ? tj : th;
        if (more && lane >= told && lane <= l) chain_st(slot + t, lane == l ? tj : 0.0);
        told = l + 1;
        if (any && (__shfl_sync(0xffffffffu, own, l) >> lane) & 1u) repeat(tj);  // repeats are rare
    }
    if (more && lane >= told) chain_st(slot + t, 0.0);
    return th;
}

// Warp `warp`'s 32 coordinates t = 32 warp + lane of a chain of cnt <= DCD_FAST_MAX: returns the lane's
// step.  C[j ldc + t]: the coupling of t to the step of j < t (any number for t <= j in the same 32);
// rep[j DCD_FAST_K + q]: bit l set where coordinate 32 q + l > j holds j's row; slot (cnt entries,
// CHAIN_OPEN at the start): the steps published to the later groups; rho, gj, eta, ie: alpha_t, g_t,
// eta_t, 1 / eta_t (0: no step).
__device__ __forceinline__ double dcd_chain_group(const double *C, int ldc, const uint32_t *rep, double *slot, int cnt,
                                                  int warp, int lane, double rho, double gj, double eta, double ie,
                                                  double nu, int *err)
{
    const int e = __double2hiint(eta) >> 20, en = __double2hiint(nu) >> 20;  // biased exponents
    const bool scaled = (ie == 0.0 || (e >= 1023 - 20 && e <= 1023 + 300)) &&
                        (nu == __longlong_as_double(0x7ff0000000000000LL) || (en >= 1023 - 300 && en <= 1023 + 300));
    rho += 0.0;  // -0 to +0: the comparisons are of bits
    if (__all_sync(0xffffffffu, scaled))
        return dcd_chain_run<true>(C, ldc, rep, slot, cnt, warp, lane, rho, gj, eta, ie, nu, err);
    return dcd_chain_run<false>(C, ldc, rep, slot, cnt, warp, lane, rho, gj, eta, ie, nu, err);
}

}  // namespace dcd
