// corr.cuh -- the correlation families of gp_correlation on the device.
//
// Power-exponential (eq. 2):  rho = exp(-S),  S = sum_k theta_k |dx_k|^p.
// Matern, nu = 1/2, 3/2, 5/2, in the same product form over dimensions: with
// h_k = c theta_k |dx_k| (c = 1, sqrt 3, sqrt 5),
//   rho = exp(-sum_k h_k) prod_k q(h_k),  q(h) = 1, 1 + h, 1 + h + h^2 / 3,
// so one exponential per entry remains and the theta-independent part of each
// term (|dx_k|^p, or |dx_k|) is shared by every candidate, as the assembly
// kernels arrange.  The kernels therefore take theta pre-multiplied by c and
// the powers with p = 1 for the Matern families.
#pragma once

#include <cmath>

#include "df.cuh"
#include "gp_internal.cuh"

namespace gp {

// c of h = c theta |dx| (1 for the power-exponential family)
__host__ __device__ __forceinline__ double corr_theta_scale(int corr) {
    return corr == GP_CORR_MATERN32 ? 1.7320508075688772935 : (corr == GP_CORR_MATERN52 ? 2.2360679774997896964 : 1.0);
}

__host__ __device__ __forceinline__ bool corr_is_matern(int corr) { return corr != GP_CORR_POWEXP; }

// q(h) in double
__device__ __forceinline__ double matern_q(double h, int corr) {
    if (corr == GP_CORR_MATERN32) return 1.0 + h;
    if (corr == GP_CORR_MATERN52) return 1.0 + h + h * h / 3.0;
    return 1.0;
}

// q(h) in double-float (h >= 0); third = 1/3 as double-float
__device__ __forceinline__ dfl matern_q_df(dfl h, int corr, dfl third) {
    if (corr == GP_CORR_MATERN32) return df_add_float(1.f, h);
    if (corr == GP_CORR_MATERN52) return df_add_float(1.f, df_fma(df_mul(h, h), third, h));
    return dfl{1.f, 0.f};
}

// the same for two values at once, bit for bit (nthird: the negated high word)
__device__ __forceinline__ df2 matern_q_df2(df2 h, int corr, df2 third, f32x2 nthird) {
    const f32x2 one = f2_pack(1.f, 1.f), zero = f2_pack(0.f, 0.f);
    if (corr != GP_CORR_MATERN32 && corr != GP_CORR_MATERN52) return {one, zero};
    df2 w = h;
    if (corr == GP_CORR_MATERN52) {
        const df2 m = df2_mul(f2_neg(h.hi), h, h);
        const f32x2 pn = f2_mul(m.hi, nthird);
        f32x2 e = f2_fma(m.hi, third.hi, pn);
        e = f2_fma(m.hi, third.lo, e);
        e = f2_fma(m.lo, third.hi, e);
        f32x2 s, t;
        f2_two_diff(h.hi, pn, s, t);
        f2_fast_two_sum(s, f2_add(t, f2_add(h.lo, e)), w.hi, w.lo);
    }
    const f32x2 s = f2_add(one, w.hi), bb = f2_sub(s, one);
    const f32x2 e = f2_add(f2_sub(one, f2_sub(s, bb)), f2_sub(w.hi, bb));
    df2 r;
    f2_fast_two_sum(s, f2_add(e, w.lo), r.hi, r.lo);
    return r;
}

// exp(-S) in double without CUDA's exp (the reduction of P. T. P. Tang, ACM TOMS
// 15 (1989)): an FP64 instruction is worth 64 FP32 ones here, so what counts is
// their number, 11 against about 20.
// exp(-S) = 2^(k/128) exp(r), k = round(-128 S / ln 2), r = -S - k ln2/128
// (two fmas against ln2/128 as 33 + 53 bits), exp(r) - 1 = r + r^2 (1/2 + r/6 +
// r^2/24 + r^3/120) (the next term is below 2^-60), times the table's 2^(j/128)
// as a double-double, scaled by its exponent bits: 11 double operations.  S
// above 700 takes exp.
constexpr int kE64NBits = 7;
constexpr int kE64N = 1 << kE64NBits;
struct ExpTab64 {
    double2 e2[kE64N];            // 2^(j/128) as (hi, lo)
};

__device__ __forceinline__ double exp_neg_tab64(double s, const ExpTab64& t) {
    if (!(s < 700.0)) return exp(-s);
    constexpr double kInv = 128.0 / 0.693147180559945309417232121458176568;
    constexpr double kHi = 0x1.62e42fefp-8;                                // ln2 / 128, 33 bits
    constexpr double kLo = 0x1.473de6af278edp-41;                          // and the rest
    constexpr double kRound = 6755399441055744.0;                          // 1.5 2^52
    const double kr = fma(-s, kInv, kRound);
    const int k = __double2loint(kr);
    const double kd = kr - kRound;
    const double r = fma(-kd, kLo, fma(-kd, kHi, -s));
    double q = fma(r, 1.0 / 120.0, 1.0 / 24.0);
    q = fma(r, q, 1.0 / 6.0);
    q = fma(r, q, 0.5);
    const double w = fma(r * r, q, r);
    const double2 T = t.e2[k & (kE64N - 1)];
    const double v = T.x + fma(T.x, w, T.y);
    return __hiloint2double(__double2hiint(v) + ((k >> kE64NBits) << 20), __double2loint(v));
}

// The table, in long double (64 significant bits or more).
inline void exp_tab64_fill(ExpTab64& t) {
    for (int j = 0; j < kE64N; ++j) {
        const long double v = exp2l((long double)j / (long double)kE64N);
        t.e2[j].x = (double)v;
        t.e2[j].y = (double)(v - (long double)t.e2[j].x);
    }
}

}  // namespace gp
