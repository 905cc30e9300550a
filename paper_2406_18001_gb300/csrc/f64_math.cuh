// f64_math.cuh -- FP64 device functions shared by the FP64 kernels (block_f64.cu, svm_grid.cu), sized by
// GB300's FP64 pipe: a warp instruction takes some 80 cycles of a scheduler's.
#pragma once

#include <cuda_runtime.h>

namespace dcd {

// 2^(j / 64), j < 64: the table of exp_tab
__device__ __forceinline__ double exp_tab_entry(int j) { return exp2((double)j * (1.0 / 64.0)); }

// e^x for -700 < x <= 0 by table and polynomial (Tang, ACM TOMS 15, 1989): x = k ln2 / 64 + r,
// |r| <= ln2 / 128, e^x = 2^(k / 64) e^r with 2^(j / 64) from the table tab[j] and e^r - 1 by its
// Taylor polynomial of degree 5 (truncation below 4e-17).  Ten FP64 operations; within about one ulp.
__device__ __forceinline__ double exp_tab(double x, const double *tab)
{
    const double t = fma(x, 92.332482616893656877, 6755399441055744.0);  // 64 / ln 2
    const int k = __double2loint(t);
    const double kd = t - 6755399441055744.0;
    double r = fma(kd, -0x1.62e42fee00000p-7, x);  // ln 2 / 64: 33 leading bits, exact with |k| < 2^17
    r = fma(kd, -0x1.a39ef35793c76p-39, r);
    double p = fma(r, 1.0 / 120.0, 1.0 / 24.0);
    p = fma(p, r, 1.0 / 6.0);
    p = fma(p, r, 0.5);
    p = fma(p, r * r, r);
    const double c = tab[k & 63];
    const double v = fma(c, p, c);
    return __hiloint2double(__double2hiint(v) + ((k >> 6) << 20), __double2loint(v));
}

}  // namespace dcd
