// df.cuh -- double-float ("float-float") arithmetic on the FP32 pipes.
//
// A value is the unevaluated sum hi + lo of two floats with |lo| <= ulp(hi)/2,
// about 48 significant bits.  On this GPU an FP64 instruction costs about 64
// FP32 instructions, so the split-precision path keeps its working matrix,
// its combination of tensor-core partial sums and its solves in this form.
//
// The error-free transformations are the published ones: TwoSum (D. Knuth,
// TAOCP vol. 2), FastTwoSum (T. J. Dekker, "A floating-point technique for
// extending the available precision", Numer. Math. 18, 1971) and the exact
// product through a fused multiply-add.  The _rn intrinsics keep the compiler
// from contracting or reordering them.
#pragma once

#include <cuda_runtime.h>

namespace gp {

struct dfl {
    float hi, lo;
};

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// requires |a| >= |b| (or a == 0)
__device__ __forceinline__ void fast_two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    e = __fsub_rn(b, __fsub_rn(s, a));
}

__device__ __forceinline__ dfl df_make(float hi, float lo) {
    dfl r;
    fast_two_sum(hi, lo, r.hi, r.lo);
    return r;
}

__device__ __forceinline__ dfl df_add(dfl a, dfl b) {
    float s, e, t, f;
    two_sum(a.hi, b.hi, s, e);
    two_sum(a.lo, b.lo, t, f);
    e = __fadd_rn(e, t);
    fast_two_sum(s, e, s, e);
    e = __fadd_rn(e, f);
    fast_two_sum(s, e, s, e);
    return {s, e};
}

// a + b for a float a: the bits of df_add({a, 0}, b), whose second TwoSum and
// last FastTwoSum change nothing then
__device__ __forceinline__ dfl df_add_float(float a, dfl b) {
    float s, e;
    two_sum(a, b.hi, s, e);
    e = __fadd_rn(e, b.lo);
    fast_two_sum(s, e, s, e);
    return {s, e};
}

__device__ __forceinline__ dfl df_neg(dfl a) { return {-a.hi, -a.lo}; }

__device__ __forceinline__ dfl df_sub(dfl a, dfl b) { return df_add(a, df_neg(b)); }

// c + a * b
__device__ __forceinline__ dfl df_fma(dfl a, dfl b, dfl c) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, e);
    e = __fmaf_rn(a.lo, b.hi, e);
    float s, t;
    two_sum(c.hi, p, s, t);
    t = __fadd_rn(t, __fadd_rn(c.lo, e));
    fast_two_sum(s, t, s, t);
    return {s, t};
}

// c - a * b
__device__ __forceinline__ dfl df_fms(dfl a, dfl b, dfl c) { return df_fma(df_neg(a), b, c); }

// a * b: the exact product of the high words, its error and the cross terms
// (what df_fma gives with c = 0, without the additions of zero)
__device__ __forceinline__ dfl df_mul(dfl a, dfl b) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, e);
    e = __fmaf_rn(a.lo, b.hi, e);
    float s, t;
    fast_two_sum(p, e, s, t);
    return {s, t};
}

// Two double-float values side by side in 64-bit register pairs, for the
// paired FP32 instructions of sm_100 and later: each half rounds as the
// scalar instruction does, and one issue does the work of two.
typedef unsigned long long f32x2;

struct df2 {
    f32x2 hi, lo;
};

__device__ __forceinline__ f32x2 f2_pack(float a, float b) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float f2_first(f32x2 v) {
    float a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
    return a;
}
__device__ __forceinline__ float f2_second(f32x2 v) {
    float a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
    return b;
}
__device__ __forceinline__ f32x2 f2_add(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 f2_sub(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 f2_mul(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 f2_fma(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 f2_neg(f32x2 a) { return a ^ 0x8000000080000000ull; }
// a b where its only use is an addition, rounded by itself: a pair's mul.rn and
// add.rn were seen contracted into one fma there, the scalar ones are not
__device__ __forceinline__ f32x2 f2_mul_alone(f32x2 a, f32x2 b) {
    return f2_pack(__fmul_rn(f2_first(a), f2_first(b)), __fmul_rn(f2_second(a), f2_second(b)));
}

// c - a b, half by half the bits of df_fma(df_neg(a), b, c) and of
// df_fma(a, df_neg(b), c): p = -(a.hi b.hi), which the caller forms with
// whichever negated factor it shares between calls, and the product's error
// and cross terms with the opposite sign (every step rounds symmetrically).
__device__ __forceinline__ df2 df2_fnma(f32x2 p, df2 a, df2 b, df2 c) {
    f32x2 en = f2_fma(a.hi, b.hi, p);
    en = f2_fma(a.hi, b.lo, en);
    en = f2_fma(a.lo, b.hi, en);
    const f32x2 s = f2_add(c.hi, p);
    const f32x2 bb = f2_sub(s, c.hi);
    f32x2 t = f2_add(f2_sub(c.hi, f2_sub(s, bb)), f2_sub(p, bb));
    t = f2_add(t, f2_sub(c.lo, en));
    df2 r;
    r.hi = f2_add(s, t);
    r.lo = f2_sub(t, f2_sub(r.hi, s));
    return r;
}

// Sum of a and -bn, half by half the bits of two_sum(a, -bn)
__device__ __forceinline__ void f2_two_diff(f32x2 a, f32x2 bn, f32x2& s, f32x2& e) {
    const f32x2 s0 = f2_sub(a, bn), bb = f2_sub(s0, a);
    e = f2_sub(f2_sub(a, f2_sub(s0, bb)), f2_add(bn, bb));
    s = s0;
}
// fast_two_sum(a, b), half by half
__device__ __forceinline__ void f2_fast_two_sum(f32x2 a, f32x2 b, f32x2& s, f32x2& e) {
    const f32x2 s0 = f2_add(a, b);
    e = f2_sub(b, f2_sub(s0, a));
    s = s0;
}
// a b from an = -a.hi: the bits of df_mul
__device__ __forceinline__ df2 df2_mul(f32x2 an, df2 a, df2 b) {
    const f32x2 pn = f2_mul(an, b.hi);
    f32x2 e = f2_fma(a.hi, b.hi, pn);
    e = f2_fma(a.hi, b.lo, e);
    e = f2_fma(a.lo, b.hi, e);
    df2 r;
    r.hi = f2_sub(e, pn);
    r.lo = f2_sub(e, f2_add(r.hi, pn));
    return r;
}

// c + l x for one l and two x: bit for bit df_fma(l, x, c) of each half
// (xn = -x.hi)
__device__ __forceinline__ df2 df2_fma_shared(dfl l, df2 x, f32x2 xn, df2 c) {
    const f32x2 lh = f2_pack(l.hi, l.hi), ll = f2_pack(l.lo, l.lo);
    const f32x2 pn = f2_mul(lh, xn);
    f32x2 e = f2_fma(lh, x.hi, pn);
    e = f2_fma(lh, x.lo, e);
    e = f2_fma(ll, x.hi, e);
    f32x2 s, t;
    f2_two_diff(c.hi, pn, s, t);
    df2 r;
    f2_fast_two_sum(s, f2_add(t, f2_add(c.lo, e)), r.hi, r.lo);
    return r;
}

__device__ __forceinline__ dfl df2_first(df2 v) { return {f2_first(v.hi), f2_first(v.lo)}; }
__device__ __forceinline__ dfl df2_second(df2 v) { return {f2_second(v.hi), f2_second(v.lo)}; }
__device__ __forceinline__ df2 df2_pack(dfl a, dfl b) { return {f2_pack(a.hi, b.hi), f2_pack(a.lo, b.lo)}; }
__device__ __forceinline__ df2 df2_dup(dfl a) { return {f2_pack(a.hi, a.hi), f2_pack(a.lo, a.lo)}; }

// a / b to about 46 bits: one Newton correction of the float quotient
__device__ __forceinline__ dfl df_div(dfl a, dfl b) {
    const float q1 = __fdiv_rn(a.hi, b.hi);
    const dfl r = df_fms(dfl{q1, 0.f}, b, a);      // a - q1 b
    const float q2 = __fdiv_rn(r.hi, b.hi);
    return df_make(q1, q2);
}

__device__ __forceinline__ dfl df_from_double(double v) {
    const float h = __double2float_rn(v);
    const float l = __double2float_rn(v - (double)h);
    return {h, l};
}

__device__ __forceinline__ double df_to_double(dfl a) { return (double)a.hi + (double)a.lo; }

// The same for values with a positive high word in the middle of the float
// range (others take the general form), whose conversions to and from double
// are integer shifts: two double instructions instead of four and three.
__device__ __forceinline__ dfl df_from_positive(double v) {
    const long long b = __double_as_longlong(v);
    if ((unsigned long long)(b - (923LL << 52)) >= (200ULL << 52)) return df_from_double(v);   // 2^-100 .. 2^100
    const long long u = b + (1LL << 28);
    const float h = __uint_as_float((unsigned)(u >> 29) - (896u << 23));
    return {h, __double2float_rn(v - __longlong_as_double(u & ~((1LL << 29) - 1)))};
}

__device__ __forceinline__ double df_to_double_positive(dfl a) {
    if (!(a.hi >= 0x1p-100f && a.hi <= 0x1p100f)) return df_to_double(a);
    const long long b = ((long long)__float_as_uint(a.hi) << 29) + (896LL << 52);
    return __longlong_as_double(b) + (double)a.lo;
}

__device__ __forceinline__ dfl df_load(const float2* p) {
    const float2 v = *p;
    return {v.x, v.y};
}

__device__ __forceinline__ void df_store(float2* p, dfl a) { *p = make_float2(a.hi, a.lo); }

// Entries of the table of 2^(-j/N) that df_exp_neg reads (N = 1024: 8 KB
// of double-float values in shared memory).
constexpr int kExpTabBits = 10;
constexpr int kExpTab = 1 << kExpTabBits;

// exp(-S) to about 46 bits, after P. T. P. Tang, "Table-driven
// implementation of the exponential function in IEEE floating-point
// arithmetic", ACM TOMS 15 (1989), with a table of N = 1024 entries:
//   k = round(S N / ln 2),  r = S - k ln2/N  (|r| <= ln2/(2N) = 3.4e-4, a
//   Cody-Waite reduction with ln2/N held as two floats),
//   exp(-S) = 2^(-k/N) exp(-r),  2^(-k/N) = 2^(-m) tab[j] for k = N m + j,
//   exp(-r) = 1 - r + q,  q = r^2/2 - r^3/6 (the r^4 term is below 2^-50).
// q < 6e-8 is needed to float precision only, so past the reduction the
// only double-float steps are 1 - r and the product with the table.  S may
// be negative down to -83 (the logarithms of df_log's Newton step).
// tab[j] = 2^(-j/N) as double-float (load_exp2_table).  Results
// below 2^-125 (S > 86.6) are returned as zero.
__device__ __forceinline__ dfl df_exp_neg(dfl S, const dfl* tab) {
    constexpr double kLn2OverN = 0.693147180559945309417232121458176568 / kExpTab;
    constexpr float kCHi = (float)kLn2OverN;
    constexpr float kCLo = (float)(kLn2OverN - (double)kCHi);
    constexpr float kNOverLn2 = (float)(kExpTab / 0.693147180559945309417232121458176568);
    if (!(S.hi < 86.6f)) return {0.f, 0.f};
    const float kf = rintf(__fmul_rn(S.hi, kNOverLn2));
    const int k = (int)kf;
    // r = S - k (C_hi + C_lo); k C_hi as p1 + e1 exactly
    const float p1 = __fmul_rn(kf, kCHi);
    const float e1 = __fmaf_rn(kf, kCHi, -p1);
    const float p2 = __fmul_rn(kf, kCLo);
    float rh = __fsub_rn(S.hi, p1);   // exact: p1 is within a factor 2 of S.hi, or 0
    float rl = __fsub_rn(__fsub_rn(S.lo, e1), p2);
    two_sum(rh, rl, rh, rl);
    // q = rh^2/2 - rh^3/6 + rh rl  (r^2/2 to first order in rl)
    float q = __fmaf_rn(rh, -1.f / 6.f, 0.5f);
    q = __fmaf_rn(rh, q, rl);
    q = __fmul_rn(rh, q);
    float s, t;
    fast_two_sum(1.f, -rh, s, t);     // |rh| < 1
    t = __fadd_rn(__fsub_rn(t, rl), q);
    fast_two_sum(s, t, s, t);
    dfl e = df_mul(dfl{s, t}, tab[k & (kExpTab - 1)]);
    const float sc = __int_as_float((127 - (k >> kExpTabBits)) << 23);   // 2^-m, -120 <= m <= 125
    e.hi = __fmul_rn(e.hi, sc);
    e.lo = __fmul_rn(e.lo, sc);
    return e;
}

// The same for two values at once, their operations in pairs where both halves
// take them: bit for bit df_exp_neg of each half (S >= 0 here).  The rounding to
// an integer goes through an added 1.5 2^23, which also leaves k in the
// low bits of the sum.
__device__ __forceinline__ df2 df2_exp_neg(df2 S, const dfl* tab) {
    constexpr double kLn2OverN = 0.693147180559945309417232121458176568 / kExpTab;
    constexpr float kCHi = (float)kLn2OverN;
    constexpr float kCLo = (float)(kLn2OverN - (double)kCHi);
    constexpr float kNOverLn2 = (float)(kExpTab / 0.693147180559945309417232121458176568);
    const f32x2 round = f2_pack(12582912.f, 12582912.f);
    const f32x2 kr = f2_add(f2_mul_alone(S.hi, f2_pack(kNOverLn2, kNOverLn2)), round);
    const f32x2 kf = f2_sub(kr, round);
    const int k0 = __float_as_int(f2_first(kr)) - 0x4b400000, k1 = __float_as_int(f2_second(kr)) - 0x4b400000;
    const f32x2 p1n = f2_mul(kf, f2_pack(-kCHi, -kCHi));
    const f32x2 e1 = f2_fma(kf, f2_pack(kCHi, kCHi), p1n);
    const f32x2 p2 = f2_mul_alone(kf, f2_pack(kCLo, kCLo));
    const f32x2 r0 = f2_add(S.hi, p1n);
    const f32x2 l0 = f2_sub(f2_sub(S.lo, e1), p2);
    const f32x2 rh = f2_add(r0, l0), bb = f2_sub(rh, r0);
    const f32x2 rl = f2_add(f2_sub(r0, f2_sub(rh, bb)), f2_sub(l0, bb));
    f32x2 q = f2_fma(rh, f2_pack(-1.f / 6.f, -1.f / 6.f), f2_pack(0.5f, 0.5f));
    q = f2_fma(rh, q, rl);
    q = f2_mul_alone(rh, q);
    const f32x2 one = f2_pack(1.f, 1.f);
    const f32x2 s0 = f2_sub(one, rh);
    const f32x2 t0 = f2_sub(q, f2_add(f2_add(rh, f2_sub(s0, one)), rl));
    df2 w;
    f2_fast_two_sum(s0, t0, w.hi, w.lo);
    const df2 T = df2_pack(tab[k0 & (kExpTab - 1)], tab[k1 & (kExpTab - 1)]);
    df2 e = df2_mul(f2_neg(w.hi), w, T);
    // 2^-m by the exponent bits
    const f32x2 sc = f2_pack(__int_as_float((127 - (k0 >> kExpTabBits)) << 23),
                             __int_as_float((127 - (k1 >> kExpTabBits)) << 23));
    e.hi = f2_mul(e.hi, sc);
    e.lo = f2_mul(e.lo, sc);
    const bool in0 = f2_first(S.hi) < 86.6f, in1 = f2_second(S.hi) < 86.6f;
    e.hi = f2_pack(in0 ? f2_first(e.hi) : 0.f, in1 ? f2_second(e.hi) : 0.f);
    e.lo = f2_pack(in0 ? f2_first(e.lo) : 0.f, in1 ? f2_second(e.lo) : 0.f);
    return e;
}

// ln x for x > 0 (x in [2^-60, 2^60]): a float seed y0 = logf(x) and one
// Newton step y = y0 + x exp(-y0) - 1 in double-float, which doubles the
// seed's ~22 correct bits.
__device__ __forceinline__ dfl df_log(dfl x, const dfl* tab) {
    const float y0 = logf(x.hi);
    const dfl e = df_exp_neg(dfl{y0, 0.f}, tab);          // exp(-y0)
    const dfl t = df_fma(x, e, dfl{-1.f, 0.f});            // x exp(-y0) - 1
    return df_add(dfl{y0, 0.f}, t);
}

// Exponent modes of |d|^p: the two exact cases and the general one.
enum : int { kPowGeneral = 0, kPowOne = 1, kPowTwo = 2 };

__host__ __device__ __forceinline__ int pow_mode(double p) {
    return p == 2.0 ? kPowTwo : (p == 1.0 ? kPowOne : kPowGeneral);
}

// |d|^p for p in (0, 2] as exp(p ln |d|) in double-float (pd = p as
// double-float).  |d| outside [2^-60, 2^60] (far from any realistic
// coordinate difference) takes the double pow instead, with the result
// clamped to [0, 2^120] so that a zero theta still gives a zero term.
__device__ __forceinline__ dfl df_powabs(dfl d, int mode, double p, dfl pd, const dfl* tab) {
    if (d.hi < 0.f) d = df_neg(d);
    if (d.hi == 0.f) return {0.f, 0.f};
    if (!(d.hi >= 0x1p-60f && d.hi <= 0x1p60f)) {
        const double a = df_to_double(d);
        const double v = (mode == kPowTwo) ? a * a : (mode == kPowOne ? a : pow(a, p));
        return df_from_double(fmin(v, 0x1p120));
    }
    if (mode == kPowTwo) return df_mul(d, d);
    if (mode == kPowOne) return d;
    return df_exp_neg(df_neg(df_mul(pd, df_log(d, tab))), tab);
}

// tab[j] = 2^(-j/N), j = 0 .. N - 1, as double-float (the block's threads in
// turn; the caller synchronises before the table is read).  `src` is the
// device's copy (exp2_table): a CTA of its own 1024 exp2 is 7 us of an SM's FP64
// pipe, which small problems spent half of their assembly on (n = 64, T = 100:
// 41 -> 24 us).
__device__ __forceinline__ void load_exp2_table(dfl* tab, const float2* src) {
    for (int j = threadIdx.x; j < kExpTab; j += blockDim.x) tab[j] = df_load(src + j);
}
__device__ __forceinline__ dfl exp2_entry(int j) { return df_from_double(exp2(-(double)j / (double)kExpTab)); }

}  // namespace gp
