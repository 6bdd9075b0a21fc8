// Double-float arithmetic on the FP32 pipes for sm_103a.
//
// A value is the unevaluated sum hi + lo of two FP32 numbers (about 48 significant bits),
// built from the error-free transformations TwoSum (Knuth) and TwoProduct by FMA (Dekker's
// double-length arithmetic).  On this part FP32 issues about 60 times faster than FP64, so the
// few places that need more than FP32 in O(N^2) loops use these instead of FP64.  Products
// that feed an error-free step are rounded on their own (__fmul_rn) and sums use __fadd_rn /
// __fsub_rn, so that FMA contraction cannot break the transformations.
#pragma once

#include <cuda_runtime.h>

namespace frost {
namespace df {

struct dfloat {
    float h, l;
};

// Conversions between FP32 and FP64 in integer arithmetic, the bits of (double)f and (float)d.
// On this part a conversion is an instruction of the FP64 unit, which takes a warp
// instruction in about 64 cycles; these take about 8 and 14 instructions of the integer pipe
// (16 lanes a cycle).  Values outside the common range (denormals, infinities, NaN, FP32
// overflow) go to the instruction.
__device__ __forceinline__ double f2d(float f)
{
    const unsigned u = __float_as_uint(f), t = u & 0x7fffffffu;
    if (t != 0u && t - 0x00800000u >= 0x7f000000u) return (double)f;
    const unsigned hi = (t == 0u) ? 0u : (t >> 3) + 0x38000000u;
    return __hiloint2double((int)(hi | (u & 0x80000000u)), (int)(u << 29));
}

__device__ __forceinline__ float d2f(double d)
{
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    const unsigned t = hi & 0x7fffffffu;
    // FP64 exponents 897 .. 1150 are the normal FP32 range
    if (t - 0x38100000u >= 0x0fe00000u) return ((t | lo) == 0u) ? __uint_as_float(hi) : (float)d;
    // exponent and 23 bits of the fraction, then round to nearest even on the 29 bits below
    const unsigned m = ((t - 0x38000000u) << 3) | (lo >> 29);
    const unsigned low = lo & 0x1fffffffu;
    const unsigned up = (low + (m & 1u) > 0x10000000u) ? 1u : 0u;
    return __uint_as_float((hi & 0x80000000u) | (m + up));
}

// s + e = a + b exactly
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// s + e = a + b exactly, for |a| >= |b| (or a = 0)
__device__ __forceinline__ void fast_two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    e = __fsub_rn(b, __fsub_rn(s, a));
}

__device__ __forceinline__ dfloat make(float h, float l)
{
    dfloat r;
    fast_two_sum(h, l, r.h, r.l);
    return r;
}

// the nearest double-float of an FP64 value (48 of its 53 bits)
__device__ __forceinline__ dfloat from_double(double v)
{
    dfloat r;
    r.h = d2f(v);
    r.l = d2f(v - f2d(r.h));
    return r;
}

__device__ __forceinline__ double to_double(dfloat a) { return f2d(a.h) + f2d(a.l); }

__device__ __forceinline__ dfloat add(dfloat a, dfloat b)
{
    float s, e;
    two_sum(a.h, b.h, s, e);
    e = __fadd_rn(e, __fadd_rn(a.l, b.l));
    return make(s, e);
}

__device__ __forceinline__ dfloat neg(dfloat a)
{
    a.h = -a.h;
    a.l = -a.l;
    return a;
}

__device__ __forceinline__ dfloat sub(dfloat a, dfloat b) { return add(a, neg(b)); }

__device__ __forceinline__ dfloat mul(dfloat a, dfloat b)
{
    const float p = __fmul_rn(a.h, b.h);
    float e = fmaf(a.h, b.h, -p);
    e = fmaf(a.h, b.l, fmaf(a.l, b.h, e));
    return make(p, e);
}

__device__ __forceinline__ dfloat mul_f(dfloat a, float b)
{
    const float p = __fmul_rn(a.h, b);
    const float e = fmaf(a.l, b, fmaf(a.h, b, -p));
    return make(p, e);
}

// 1 / sqrt(a) for a > 0: the MUFU estimate y0 and the residual res = 1 - a y0^2 in
// double-float, then y0 (1 - res)^(-1/2) = y0 (1 + res/2 + 3 res^2/8 + ...), |res| < 2^-21
__device__ __forceinline__ dfloat rsqrt(dfloat a)
{
    const float y0 = rsqrtf(a.h);
    const float q = __fmul_rn(y0, y0), qe = fmaf(y0, y0, -q);
    const float pp = __fmul_rn(a.h, q), pe = fmaf(a.h, q, -pp);
    const float res = __fsub_rn(__fsub_rn(__fsub_rn(1.f, pp), pe), fmaf(a.h, qe, __fmul_rn(a.l, q)));
    const float c = __fmul_rn(__fmul_rn(y0, res), fmaf(0.375f, res, 0.5f));
    return make(y0, c);
}

// x = h + l + ll exactly (three FP32 parts hold the 53 bits of an FP64 value)
__device__ __forceinline__ void split3(double v, float &h, float &l, float &ll)
{
    h = d2f(v);
    const double r = v - f2d(h);
    l = d2f(r);
    ll = d2f(r - f2d(l));
}

// x_j - x_i from three-part splits: the two larger differences are exact (TwoSum), the
// smallest parts' difference is rounded once.  The result is renormalised (TwoSum of the
// high word and the collected tail): with splits of 12 + 12 + 24 bits (the gradient records)
// a pair closer than ~2^-24 |x| has equal or one-unit-apart high and middle parts, so the
// tail can be as large as the high word, and the products of df::mul, which drop lo x lo,
// need |lo| <= ulp(hi) / 2.
__device__ __forceinline__ dfloat sep(float jh, float jl, float jll, float ih, float il, float ill)
{
    float a, e1, b, e2, h, e4;
    two_sum(jh, -ih, a, e1);
    two_sum(jl, -il, b, e2);
    two_sum(a, b, h, e4);
    const float tail = __fadd_rn(e4, __fadd_rn(e1, __fadd_rn(e2, __fsub_rn(jll, ill))));
    dfloat r;
    two_sum(h, tail, r.h, r.l);
    return r;
}

// m / sqrt(x^2 + y^2 + z^2 + e2) = w + we from the separation's high and low parts (|low| up to a
// few units of the high part: without their squares, always positive, U would be 2e-15 too large)
__device__ __forceinline__ void mass_over_r(float xh, float xl, float yh, float yl, float zh, float zl, float e2h,
                                            float e2l, float mh, float ml, float &w, float &we)
{
    // r^2 + eps^2: exact squares of the high parts, (2 high + low) low for the rest
    // (products feeding an error-free transformation are rounded on their own, __fmul_rn,
    // so that the compiler cannot contract them into the following add)
    const float px = __fmul_rn(xh, xh), py = __fmul_rn(yh, yh), pz = __fmul_rn(zh, zh);
    const float qx = fmaf(fmaf(2.f, xh, xl), xl, fmaf(xh, xh, -px));
    const float qy = fmaf(fmaf(2.f, yh, yl), yl, fmaf(yh, yh, -py));
    const float qz = fmaf(fmaf(2.f, zh, zl), zl, fmaf(zh, zh, -pz));
    float s, t, S, u, S2, u2;
    two_sum(px, py, s, t);
    two_sum(s, pz, S, u);
    two_sum(S, e2h, S2, u2);
    const float lo = ((t + u) + (u2 + e2l)) + ((qx + qy) + qz);
    // 1 / r: MUFU estimate y0 and the residual res = 1 - r^2 y0^2 in double-float; then
    // 1/r = y0 (1 - res)^(-1/2) = y0 (1 + res/2 + 3 res^2/8 + ...), |res| < 2^-21
    const float y0 = rsqrtf(S2);
    const float q = __fmul_rn(y0, y0), qe = fmaf(y0, y0, -q);
    const float pp = __fmul_rn(S2, q), pe = fmaf(S2, q, -pp);
    const float res = ((1.f - pp) - pe) - fmaf(S2, qe, lo * q);
    const float c = y0 * res * fmaf(0.375f, res, 0.5f);
    // m / r = (m_h + m_l)(y0 + c)
    w = __fmul_rn(mh, y0);
    we = fmaf(mh, y0, -w) + fmaf(mh, c, ml * y0);
}

}  // namespace df
}  // namespace frost
