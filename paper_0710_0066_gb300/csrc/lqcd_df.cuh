// lqcd_df.cuh -- double-float ("df") arithmetic for the double-precision
// hopping sweeps of the mixed-precision path.
//
// GB300 runs FP64 at a small fraction of its FP32 rate, so a double hopping
// sweep is bound by the FP64 pipe, not by memory.  A df number is the
// unevaluated sum hi + lo of two floats (about 47 significant bits here);
// its sums and products use only FP32 adds and FMAs:
//   - Knuth's TwoSum: s + e = a + b exactly (six adds);
//   - the FMA product: p = a b, e = fma(a, b, -p), p + e = a b exactly.
// (T. J. Dekker, Numer. Math. 18 (1971) 224; D. E. Knuth, TAOCP vol. 2,
// Sec. 4.2.2; Y. Hida, X. S. Li, D. H. Bailey, ARITH-15 (2001) 155.)
//
// Doubles are split into df with integer operations only (no conversion
// through the FP64 pipe): hi takes the sign, the exponent and the leading
// 23 fraction bits; lo the next 23 of the remaining 29 fraction bits, so
// the split is exact to a relative 2^-46.  Values below 2^-80 in magnitude
// (and zeros) split to hi only.
// Results go back to double as (double) hi + (double) lo.
//
// Every function is host- and device-callable so that the host compiler
// can test them against long-double arithmetic.
#pragma once
#include <math.h>
#include <stdint.h>
#include <string.h>

#ifndef LQ_HD
#define LQ_HD __host__ __device__ __forceinline__
#endif

LQ_HD uint64_t df_bits64(double x)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t b;
    memcpy(&b, &x, 8);
    return b;
#endif
}

LQ_HD float df_f32(uint32_t b)
{
#ifdef __CUDA_ARCH__
    return __uint_as_float(b);
#else
    float x;
    memcpy(&x, &b, 4);
    return x;
#endif
}

// a * b and fma(a, b, c), each rounded once and never merged by the compiler
LQ_HD float df_mul_rn(float a, float b)
{
#ifdef __CUDA_ARCH__
    return __fmul_rn(a, b);
#else
    volatile float p = a * b;
    return p;
#endif
}

LQ_HD float df_fma_rn(float a, float b, float c)
{
#ifdef __CUDA_ARCH__
    return __fmaf_rn(a, b, c);
#else
    return fmaf(a, b, c);
#endif
}

struct df;
LQ_HD df df_split(double x);

struct df {
    float hi, lo;
    df() = default;
    LQ_HD constexpr df(float h, float l) : hi(h), lo(l) {}
    LQ_HD explicit df(int z) : hi((float)z), lo(0.f) {}
    LQ_HD explicit df(double x) { *this = df_split(x); }
};

// s + e = a + b exactly
LQ_HD void df_two_sum(float a, float b, float& s, float& e)
{
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// Sums and products leave the pair unnormalised (|lo| may exceed half an
// ulp of hi): no FastTwoSum after every operation, which cuts the sweep's
// instruction count by a third.  The value hi + lo keeps its ~2^-46
// accuracy relative to the operands' magnitudes (after a cancellation the
// small result sits partly in lo and carries float precision of itself,
// which is the same absolute accuracy).
LQ_HD df operator+(df a, df b)
{
    float s, e;
    df_two_sum(a.hi, b.hi, s, e);
    return df(s, e + (a.lo + b.lo));
}

LQ_HD df operator-(df a) { return df(-a.hi, -a.lo); }

LQ_HD df operator-(df a, df b) { return a + (-b); }

LQ_HD df operator*(df a, df b)
{
    const float p = df_mul_rn(a.hi, b.hi);
    float e = df_fma_rn(a.hi, b.hi, -p);
    e = df_fma_rn(a.hi, b.lo, e);
    e = df_fma_rn(a.lo, b.hi, e);
    return df(p, e);
}

// hi + lo as a normalised pair (|lo| <= half an ulp of hi)
LQ_HD df df_norm(df a)
{
    df r;
    df_two_sum(a.hi, a.lo, r.hi, r.lo);
    return r;
}

// Nine instructions for the pair and four for the range: a df sweep splits
// 336 doubles a site.
LQ_HD df df_split(double x)
{
    const uint64_t b = df_bits64(x);
    const uint32_t top = (uint32_t)(b >> 32), low = (uint32_t)b;
    // the leading 32 bits below sign and two exponent bits, the exponent e
    // taken from the double's bias to the float's: for 897 <= e <= 1150
    const uint32_t hb = (((uint32_t)(b >> 29) + 0x40000000u) & 0x7fffffffu) | (top & 0x80000000u);
    // remainder: the low 29 fraction bits m, worth m 2^(e - 1075); keep the
    // top 23 (m23 = m >> 6, worth m23 2^(e - 1069)).  float(m23) is exact:
    // 2^23 + m23 has the float bit pattern 0x4B000000 | m23.  The factor
    // 2^(e - 1069), with the sign, is hi's exponent less 46.
    float h = df_f32(hb);
    float l = (df_f32(((low >> 6) & 0x7fffffu) | 0x4B000000u) - 8388608.0f) *
              df_f32((hb & 0xff800000u) - (46u << 23));
    // outside 2^-80 <= |x| < 2^128 (zero, tiny, inf, nan): the nearest float
    const uint32_t range = (top & 0x7fffffffu) - (943u << 20);
#ifdef __CUDA_ARCH__
    // (predicated: a branch per number would break the loads and the
    // arithmetic around it into pieces)
    asm("{\n\t.reg .pred p;\n\tsetp.ge.u32 p, %2, %3;\n\t@p cvt.rn.f32.f64 %0, %4;\n\t@p mov.f32 %1, 0f00000000;\n\t}"
        : "+f"(h), "+f"(l)
        : "r"(range), "r"(208u << 20), "d"(x));
#else
    if (range >= (208u << 20)) {
        h = (float)x;
        l = 0.f;
    }
#endif
    return df(h, l);
}

LQ_HD double df_to_double(df a) { return (double)a.hi + (double)a.lo; }
