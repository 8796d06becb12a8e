// Double-float arithmetic and FP64 <-> double-float conversion for the
// mixed-precision path.
//
// On GB300 every FP64 instruction, and every f32 <-> f64 conversion, issues
// at about 1/65 of the FP32 rate.  The mixed path therefore keeps the FP64
// storage of momenta, positions and optical depths, but converts them to
// floats or double-float pairs (hi + lo, two FP32 numbers, ~47 significant
// bits) with integer and FP32 instructions only, carries the
// precision-critical quantities (chi_e's cancellation, optical depths) in
// double-float, and spends the FP64 pipe on one addition a component: the
// new state's (add_fd).  Everything here also compiles for the host, where it
// is tested against exact arithmetic.
//
// The error-free transformations are the classical ones: TwoSum (Knuth),
// FastTwoSum (Dekker) and TwoProd with a fused multiply-add.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define QP_HD __host__ __device__ __forceinline__
// repeated many times per particle: one called copy keeps the step kernel's
// instruction footprint small
#define QP_HD_SHARED __host__ __device__ inline __noinline__
#else
#define QP_HD inline
#define QP_HD_SHARED inline
#include <math.h>
#include <string.h>
#endif

namespace qp {

// ------------------------------------------------------------------ bit casts

QP_HD uint32_t f2u(float f)
{
#ifdef __CUDA_ARCH__
    return __float_as_uint(f);
#else
    uint32_t u;
    memcpy(&u, &f, 4);
    return u;
#endif
}

QP_HD float u2f(uint32_t u)
{
#ifdef __CUDA_ARCH__
    return __uint_as_float(u);
#else
    float f;
    memcpy(&f, &u, 4);
    return f;
#endif
}

QP_HD uint64_t d2u(double d)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(d);
#else
    uint64_t u;
    memcpy(&u, &d, 8);
    return u;
#endif
}

QP_HD double u2d(uint64_t u)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    double d;
    memcpy(&d, &u, 8);
    return d;
#endif
}

QP_HD float fma32(float a, float b, float c)
{
#ifdef __CUDA_ARCH__
    return __fmaf_rn(a, b, c);
#else
    return fmaf(a, b, c);
#endif
}

// Plain FP32 operations that the compiler must neither fuse nor reorder
// (the error-free transformations depend on each rounding).
QP_HD float add_rn(float a, float b)
{
#ifdef __CUDA_ARCH__
    return __fadd_rn(a, b);
#else
    volatile float r = a + b;
    return r;
#endif
}

QP_HD float sub_rn(float a, float b)
{
#ifdef __CUDA_ARCH__
    return __fsub_rn(a, b);
#else
    volatile float r = a - b;
    return r;
#endif
}

QP_HD float mul_rn(float a, float b)
{
#ifdef __CUDA_ARCH__
    return __fmul_rn(a, b);
#else
    volatile float r = a * b;
    return r;
#endif
}

// ------------------------------------------------------------------ double-float

struct df2 {
    float hi, lo;
};

QP_HD df2 two_sum(float a, float b)
{
    const float s = add_rn(a, b);
    const float bb = sub_rn(s, a);
    const float e = add_rn(sub_rn(a, sub_rn(s, bb)), sub_rn(b, bb));
    return {s, e};
}

// requires |a| >= |b| (or a == 0)
QP_HD df2 fast_two_sum(float a, float b)
{
    const float s = add_rn(a, b);
    return {s, sub_rn(b, sub_rn(s, a))};
}

QP_HD df2 two_prod(float a, float b)
{
    const float p = mul_rn(a, b);
    return {p, fma32(a, b, -p)};
}

QP_HD df2 df_add(df2 a, df2 b)
{
    const df2 s = two_sum(a.hi, b.hi);
    const df2 t = two_sum(a.lo, b.lo);
    df2 r = fast_two_sum(s.hi, add_rn(s.lo, t.hi));
    return fast_two_sum(r.hi, add_rn(r.lo, t.lo));
}

QP_HD df2 df_add_f(df2 a, float b)
{
    const df2 s = two_sum(a.hi, b);
    return fast_two_sum(s.hi, add_rn(s.lo, a.lo));
}

QP_HD df2 df_neg(df2 a) { return {-a.hi, -a.lo}; }

QP_HD df2 df_sub(df2 a, df2 b) { return df_add(a, df_neg(b)); }

QP_HD df2 df_mul_f(df2 a, float b)
{
    const df2 p = two_prod(a.hi, b);
    return fast_two_sum(p.hi, fma32(a.lo, b, p.lo));
}

QP_HD df2 df_mul(df2 a, df2 b)
{
    const df2 p = two_prod(a.hi, b.hi);
    return fast_two_sum(p.hi, fma32(a.hi, b.lo, fma32(a.lo, b.hi, p.lo)));
}

QP_HD df2 df_sqr(df2 a)
{
    const df2 p = two_prod(a.hi, a.hi);
    return fast_two_sum(p.hi, fma32(a.hi + a.hi, a.lo, p.lo));
}

// sqrt of a >= 0: one Newton correction of the FP32 root
QP_HD df2 df_sqrt(df2 a)
{
    if (!(a.hi > 0.0f)) return {0.0f, 0.0f};
#ifdef __CUDA_ARCH__
    const float s = __fsqrt_rn(a.hi);
#else
    const float s = sqrtf(a.hi);
#endif
    const df2 s2 = two_prod(s, s);
    const float r = (((a.hi - s2.hi) - s2.lo) + a.lo) / (2.0f * s);
    return fast_two_sum(s, r);
}

QP_HD float df_to_f(df2 a) { return a.hi + a.lo; }

// ------------------------------------------------------------------ FP64 <-> double-float

// Split a double into hi (its first 24 significand bits, truncated) and lo
// (the remainder rounded to FP32), using integer and FP32 instructions only.
// |d| below 2^-126 gives (0, 0); |d| at or above 2^128 is not supported
// (the caller's values are far inside this range).  hi + lo == d to within
// 2^-47 |d|.
QP_HD df2 split_d(double d)
{
    const uint64_t b = d2u(d);
    const uint32_t dh = (uint32_t)(b >> 32), dl = (uint32_t)b;
    const uint32_t e = (dh >> 20) & 0x7FFu, sign = dh & 0x80000000u;
    // sign | (e - 896) << 23 | top 23 mantissa bits
    const uint32_t top = (dh << 3) | (dl >> 29);
    const uint32_t hb = ((top - (384u << 23)) & 0x7FFFFFFFu) | sign;
    // remainder: the low 29 mantissa bits, worth 2^(e - 1075) each, rounded
    // to 24 by the conversion
    const float lo = (float)(dl & 0x1FFFFFFFu) * u2f(((e - 948u) << 23) | sign);
    return {e < 897u ? 0.0f : u2f(hb), e < 949u ? 0.0f : lo};
}

// d rounded to the nearest float (ties away from zero) by integer
// instructions; |d| below 2^-126 gives 0.  Rounding to nearest matters where
// an FP32 update acts on this value in place of d: a truncated (always
// smaller) value would let, e.g., a rotation shrink |u| by a biased amount
// every step.  A carry out of the mantissa rounds up into the exponent.
QP_HD float hi_d(double d)
{
    const uint64_t b = d2u(d);
    const uint32_t dh = (uint32_t)(b >> 32), dl = (uint32_t)b;
    const uint32_t e = (dh >> 20) & 0x7FFu;
    if (e < 897u) return 0.0f;
    const uint32_t top = ((dh << 3) | (dl >> 29)) + ((dl >> 28) & 1u);
    return u2f(((top - (384u << 23)) & 0x7FFFFFFFu) | (dh & 0x80000000u));
}

// Exact conversion of a finite float to double by integer instructions (normal
// floats; zero and denormals give 0).
QP_HD double finite_to_d(float f)
{
    const uint32_t b = f2u(f);
    const uint32_t e = (b >> 23) & 0xFFu;
    if (e == 0u) return 0.0;
    return u2d(((uint64_t)(b & 0x80000000u) << 32) | ((uint64_t)(e + 896u) << 52) |
               ((uint64_t)(b & 0x7FFFFFu) << 29));
}

// The same with infinities and NaN.  (Two instructions more, and add_fd and the
// FP64 path's seeds, which convert most, tell such values by other means: with
// this conversion there the 4.2e6-lepton collision took 4 % longer.)
QP_HD double f_to_d(float f)
{
    const uint32_t b = f2u(f);
    const uint32_t e = (b >> 23) & 0xFFu;
    if (e == 0u) return 0.0;
    const uint32_t bias = e == 0xFFu ? 2u * 896u : 896u;
    return u2d(((uint64_t)(b & 0x80000000u) << 32) | ((uint64_t)(e + bias) << 52) |
               ((uint64_t)(b & 0x7FFFFFu) << 29));
}

// hi + lo rounded to double.
QP_HD double merge_df(df2 a) { return f_to_d(a.hi) + f_to_d(a.lo); }

// d + f rounded to double: the FP64 accumulation of an FP32 increment.  The
// stored double keeps all its bits; only the increment carries FP32 error.
//   f below 2^29 units of d's last place: one FP64 addition of the exactly
//     converted f.  The FP64 pipe is nearly idle on this path, and seven
//     additions a lepton keep it 30 % busy; the same sum by some 25 integer
//     instructions and a call each took more issue slots than the rest of the
//     write-back;
//   larger f, or a sum below a quarter of d: a double-float sum (split_d,
//     two_sum, one rounded low part), exact to 2^-47 relative.  A momentum
//     turning through zero, an optical depth near its end and every recoil
//     are here, so nearly every warp of a step has such lanes: one short
//     function, called.
// (Three integer functions calling one another, decoding the operands again
// each, were 30 % of the 4.2e6-lepton collision step.)
QP_HD_SHARED double add_fd_wide(double d, float f)
{
    const uint32_t ed = (uint32_t)(d2u(d) >> 52) & 0x7FFu, ef = (f2u(f) >> 23) & 0xFFu;
    if (ed == 0x7FFu || ef == 0xFFu || ed < 897u || ed > 1150u) return d + (double)f;
    const df2 a = split_d(d);
    const df2 s = two_sum(a.hi, f);
    return finite_to_d(s.hi) + finite_to_d(add_rn(s.lo, a.lo));
}

QP_HD double add_fd(double d, float f)
{
    const uint32_t ed = (uint32_t)(d2u(d) >> 52) & 0x7FFu, ef = (f2u(f) >> 23) & 0xFFu;
    // f in units of d's last place: (its 24-bit significand) * 2^k; more for the
    // largest d, so that an infinity or NaN goes to add_fd_wide beside any d
    const int k = (int)ef - (int)(ed < 1150u ? ed : 1150u) + 925;
    const double r = d + finite_to_d(f);
    if (k < 28 || (k == 28 && ((uint32_t)(d2u(r) >> 52) & 0x7FFu) + 1u >= ed)) return r;
    return add_fd_wide(d, f);
}

// ------------------------------------------------------------------ equal steps

// The increments that repeat_step takes: sum(x) is x and the exact increment
// rounded once, one(x) the step as it is defined, equal to sum(x) where
// exact(e) holds for x's biased exponent e and sum(x) has that exponent too;
// rest(D) is the increment less D, rounded.
struct StepFloat {  // add_fd(x, f)
    double d;
    float f;
    QP_HD explicit StepFloat(float f_) : d(f_to_d(f_)), f(f_) {}
    QP_HD double one(double x) const { return add_fd(x, f); }
    QP_HD double sum(double x) const { return x + d; }
    QP_HD double rest(double D) const { return d - D; }
    QP_HD bool exact(int e) const { return (int)((f2u(f) >> 23) & 0xFFu) - e + 925 <= 28; }
};
struct StepProduct {  // fma(a, b, x)
    double a, b;
    QP_HD double one(double x) const { return fma(a, b, x); }
    QP_HD double sum(double x) const { return fma(a, b, x); }
    QP_HD double rest(double D) const { return fma(a, b, -D); }
    QP_HD bool exact(int) const { return true; }
};

// x after n equal steps: the bits of taking them one by one.  While x keeps its
// exponent its values lie on one grid, so every step that is no tie rounds to
// the same difference D (exact), and k of them are x + k D, exact as well: one
// addition a binade crossed, not one a step.  k keeps clear of the binade's end
// by an FP32 estimate; the sum is taken only if it stays inside, and a step
// otherwise.  (A fused window's photons move up to its length, each step an
// instruction of the FP64 pipe and coordinate: 250 steps of 4096 electrons
// 1570 -> 1469 us.)
template <class Step>
QP_HD double repeat_step(double x, int n, const Step &s)
{
    while (n > 0) {
        const uint64_t bx = d2u(x);
        const int e = (int)(bx >> 52) & 0x7FF;
        const double y = s.sum(x);
        const uint64_t by = d2u(y);
        bool stepped = false;
        if (n > 3 && e >= 960 && e < 1150 && s.exact(e) && (by >> 52) == (bx >> 52)) {
            if (by == bx) return x;
            const double D = y - x;
            if ((d2u(s.rest(D)) << 1 >> 1) == (uint64_t)(e - 53) << 52) {  // ties: parity decides
                for (; n > 0; --n) x = s.one(x);
                return x;
            }
            const uint64_t mant = bx & 0xFFFFFFFFFFFFFull;
            const bool inward = ((d2u(D) ^ bx) >> 63) != 0u;
            const uint32_t room = (uint32_t)((inward ? mant : 0xFFFFFFFFFFFFFull - mant) >> 20);
            // room 2^20 units of the last place, 2^(e - 1055), over |D|
            const float q = (float)room * u2f((uint32_t)(e - 928) << 23) /
                            u2f(f2u(hi_d(D)) & 0x7FFFFFFFu);
            const float c = q * 0.99999f - 1.0f;
            if (c >= 2.0f) {
                const int k = c < (float)n ? (int)c : n;
                const double t = fma(k < (1 << 24) ? finite_to_d((float)k) : (double)k, D, x);
                const uint64_t bt = d2u(t);
                if ((bt >> 52) == (bx >> 52) && (bt << 12) != 0u) {
                    x = t;
                    n -= k;
                    stepped = true;
                }
            }
        }
        if (!stepped) {
            const double z = s.one(x);
            if (d2u(z) == bx) return x;
            x = z;
            --n;
        }
    }
    return x;
}

}  // namespace qp
