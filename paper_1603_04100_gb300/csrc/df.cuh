// Double-float arithmetic on the FP32 pipe.
//
// A value is the unevaluated sum hi + lo of two FP32 numbers, normalised so
// that hi = fl32(hi + lo); it carries about 48 significant bits.  On this part
// an FP32 instruction issues at 64 times the FP64 rate, so a double-float
// operation of 3-12 FP32 instructions is still several times cheaper than one
// FP64 instruction.
//
// The building blocks are the classical error-free transformations: Knuth's
// TwoSum (a + b = s + e exactly), Dekker's Fast2Sum (the same when |a| >= |b|)
// and the FMA-based TwoProduct (a * b = p + e exactly).  The compound
// operations are the plain double-word algorithms ("sloppy" addition,
// double-word times double-word) as analysed by Joldes, Muller and Popescu
// (ACM TOMS 2017): each result is within a small multiple of 2^-48 of the
// operands' magnitudes, which is what residuals of least-squares systems need.
// Every step uses an explicit round-to-nearest intrinsic so that neither FMA
// contraction nor reassociation can alter the error-free transformations.
#pragma once

#include <cuda_runtime.h>

namespace mvgd {

struct df {
    float hi, lo;
};

__device__ __forceinline__ df df_make(float a) { return {a, 0.0f}; }

__device__ __forceinline__ df two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return {s, e};
}

// Requires |a| >= |b| (or a == 0).
__device__ __forceinline__ df fast_two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}

__device__ __forceinline__ df two_prod(float a, float b) {
    const float p = __fmul_rn(a, b);
    return {p, __fmaf_rn(a, b, -p)};
}

__device__ __forceinline__ df df_neg(df a) { return {-a.hi, -a.lo}; }

__device__ __forceinline__ df df_add(df a, df b) {
    const df s = two_sum(a.hi, b.hi);
    return fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}

__device__ __forceinline__ df df_sub(df a, df b) { return df_add(a, df_neg(b)); }

__device__ __forceinline__ df df_mul(df a, df b) {
    const df p = two_prod(a.hi, b.hi);
    const float t = __fmaf_rn(a.hi, b.lo, __fmul_rn(a.lo, b.hi));
    return fast_two_sum(p.hi, __fadd_rn(p.lo, t));
}

__device__ __forceinline__ df df_mul_f(df a, float b) {
    const df p = two_prod(a.hi, b);
    return fast_two_sum(p.hi, __fmaf_rn(a.lo, b, p.lo));
}

// acc + a * b
__device__ __forceinline__ df df_fma(df acc, df a, df b) { return df_add(acc, df_mul(a, b)); }

// a / b: one FP32 quotient, its remainder in double-float, one correction.
__device__ __forceinline__ df df_div(df a, df b) {
    const float q1 = __fdiv_rn(a.hi, b.hi);
    const df r = df_sub(a, df_mul_f(b, q1));
    const float q2 = __fdiv_rn(r.hi, b.hi);
    return fast_two_sum(q1, q2);
}

// sqrt(a) for a >= 0: the FP32 root corrected by one Newton step on the
// double-float remainder a - s^2.
__device__ __forceinline__ df df_sqrt(df a) {
    if (!(a.hi > 0.0f)) return {__fsqrt_rn(fmaxf(a.hi, 0.0f)), 0.0f};
    const float s = __fsqrt_rn(a.hi);
    const df e = df_sub(a, two_prod(s, s));
    return fast_two_sum(s, __fdiv_rn(e.hi, __fmul_rn(2.0f, s)));
}

__device__ __forceinline__ bool df_less(df a, df b) { return a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo); }

__device__ __forceinline__ double df_to_double(df a) { return (double)a.hi + (double)a.lo; }

__device__ __forceinline__ df df_from_double(double x) {
    const float hi = __double2float_rn(x);
    return {hi, __double2float_rn(x - (double)hi)};
}

// Sums of a few terms: hi collects by TwoSum, lo what it loses, normalised once at
// the end (8 instructions a term instead of df_add's 11, 12 a product instead of
// df_fma's 18).  lo grows with the terms and rounds with it, so the sums that decide
// a row's accuracy (the moments, the residuals of the 6x6 solves) keep df_add: with
// these in their place rows came out 20 to 30 % further from 64 bits.
struct df_acc {
    float hi, lo;
};

__device__ __forceinline__ df_acc acc_zero() { return {0.0f, 0.0f}; }
__device__ __forceinline__ df_acc acc_from(df a) { return {a.hi, a.lo}; }

__device__ __forceinline__ void acc_add(df_acc& t, df a) {
    const df s = two_sum(t.hi, a.hi);
    t.hi = s.hi;
    t.lo = __fadd_rn(t.lo, __fadd_rn(s.lo, a.lo));
}

// t += a * b
__device__ __forceinline__ void acc_fma(df_acc& t, df a, df b) {
    const float p = __fmul_rn(a.hi, b.hi);
    const float e = __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, __fmaf_rn(a.hi, b.hi, -p)));
    const df s = two_sum(t.hi, p);
    t.hi = s.hi;
    t.lo = __fadd_rn(t.lo, __fadd_rn(s.lo, e));
}

__device__ __forceinline__ df acc_value(df_acc t) { return fast_two_sum(t.hi, t.lo); }

// a0 b0 + a1 b1 + a2 b2
__device__ __forceinline__ df df_dot3(df a0, df b0, df a1, df b1, df a2, df b2) {
    const float p = __fmul_rn(a0.hi, b0.hi);
    df_acc t = {p, __fmaf_rn(a0.hi, b0.lo, __fmaf_rn(a0.lo, b0.hi, __fmaf_rn(a0.hi, b0.hi, -p)))};
    acc_fma(t, a1, b1);
    acc_fma(t, a2, b2);
    return acc_value(t);
}

// x as a pair by integer instructions: the conversions of df_from_double run on the FP64
// pipe, four instructions of 16 clocks a warp each.  hi is x truncated to 24 bits, lo the
// 29 bits below, and a Fast2Sum normalises them; lo's rounding is up to 2^-48 of x, twice
// that of df_from_double, which sums do not show (rows of the mean-distance rule, 30,000
// points, K = 20: 4.9e-15 off in the median with this, 4.8e-15 with df_split_rn).  Zero,
// tiny, huge and non-finite x go the other way.
__device__ __forceinline__ df df_split(double x) {
    const unsigned hx = (unsigned)__double2hiint(x), lx = (unsigned)__double2loint(x);
    const unsigned e = (hx >> 20) & 0x7ffu;
    if (e < 1023u - 60u || e > 1023u + 120u) return df_from_double(x);
    const unsigned sign = hx & 0x80000000u;
    const float hi = __uint_as_float(sign | ((e - 896u) << 23) | ((hx & 0xfffffu) << 3) | (lx >> 29));
    const float lo = __fmul_rn(__uint2float_rn(lx & 0x1fffffffu), __uint_as_float(sign | ((e - 948u) << 23)));
    return fast_two_sum(hi, lo);
}

// The same with the 29 bits read as a signed number: hi is x rounded to nearest, lo at
// most half its last place, and its rounding 2^-49 of x, as in df_from_double.
__device__ __forceinline__ df df_split_rn(double x) {
    const unsigned hx = (unsigned)__double2hiint(x), lx = (unsigned)__double2loint(x);
    const unsigned e = (hx >> 20) & 0x7ffu;
    if (e < 1023u - 60u || e > 1023u + 120u) return df_from_double(x);
    const unsigned sign = hx & 0x80000000u;
    const int low = (int)(lx << 3) >> 3;  // 29 bits, signed: from -half to half a place of hi
    const unsigned hi = (((e - 896u) << 23) | ((hx & 0xfffffu) << 3) | (lx >> 29)) + (low < 0 ? 1u : 0u);
    return {__uint_as_float(sign | hi), __fmul_rn(__int2float_rn(low), __uint_as_float(sign | ((e - 948u) << 23)))};
}

__device__ __forceinline__ bool df_isfinite(df a) { return isfinite(a.hi) && isfinite(a.lo); }

}  // namespace mvgd
