// fp64.cuh -- arithmetic of the FP64 deposit and gather.
//
// The FP64 pipe does two multiply-adds a clock and SM on this part, so the FP64 kernels are
// bound by the number of FP64 operations a (particle, node) pair takes.
#pragma once

#include "common.cuh"

// 2^(-(s^2)) as T (1 + q): T = 2^(j / 2048) from a table (built once per context, copied to
// shared memory) and the binary exponent, q = 2^r - 1 by its Taylor series to third order
// (|r| <= 2^-12, remainder 4e-17).  Six FP64 operations from s against about twenty of exp2.
// |s| above 31 counts as 31 (2^-961).
#define F64_TAB 2048
__device__ __forceinline__ void f64_tab_load(double *dst, const double *__restrict__ src, int tid, int nthreads)
{
    for (int i = tid; i < F64_TAB / 2; i += nthreads) ((double2 *)dst)[i] = ((const double2 *)src)[i];
}
__device__ __forceinline__ void f64_exp2neg(const double *tab, double s, double &T, double &q)
{
    if ((__double2hiint(s) & 0x7fffffff) >= 0x403F0000) s = 31.0;
    const double C = 6755399441055744.0 / F64_TAB;  // 1.5 2^52 / 2048: rounds to multiples of 1 / 2048
    const double t = fma(-s, s, C);
    const int j = __double2loint(t);  // round(-2048 s^2), two's complement
    const double r = fma(-s, s, C - t);
    q = r * fma(r, fma(r, 0.0555041086648215760, 0.240226506959100700), KDE_LN2);
    const double e = tab[j & (F64_TAB - 1)];
    T = __hiloint2double(__double2hiint(e) + ((j >> 11) << 20), __double2loint(e));
}

// 1 / k^2 and (2k - 1)^2 / (8k), k = 0 .. 63 (k = 0 unused)
struct F64Series {
    double inv_sq[64], hankel[64];
    constexpr F64Series() : inv_sq(), hankel()
    {
        for (int k = 1; k < 64; ++k) {
            inv_sq[k] = 1.0 / ((double)k * k);
            hankel[k] = (2.0 * k - 1.0) * (2.0 * k - 1.0) / (8.0 * k);
        }
    }
};
static __constant__ F64Series f64_series{};

// 1 / (2 pi I0e(kappa)) in FP64: the series of kde_i0e with their coefficients tabulated, so
// that a term takes two operations and no division.
//  kappa < 30: I0 = sum q^k / k!^2, q = kappa^2 / 4; 1 / k^2
//  else:       I0e sqrt(2 pi kappa) = sum of terms t_k = t_{k-1} (2k - 1)^2 / (8 kappa k)
__device__ __forceinline__ double f64_norm(double x)
{
    if (x < 30.0) {
        const double q = 0.25 * x * x;
        double term = 1.0, sum = 1.0;
        for (int k = 1; k < 64; ++k) {  // 50 terms at kappa = 30
            term *= q * f64_series.inv_sq[k];
            sum += term;
            if (term < 1e-17 * sum) break;
        }
        return exp(x) / (KDE_TWO_PI * sum);
    }
    const double ix = 1.0 / x;
    double term = 1.0, sum = 1.0;
    for (int k = 1; k < 60; ++k) {
        const double nx = term * (ix * f64_series.hankel[k]);
        if (nx >= term) break;
        term = nx;
        sum += term;
        if (term < 1e-17 * sum) break;
    }
    return sqrt(KDE_TWO_PI * x) / (KDE_TWO_PI * sum);
}
