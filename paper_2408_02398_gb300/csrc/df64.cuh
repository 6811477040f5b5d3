// df64.cuh -- double-float arithmetic: a value is the unevaluated sum
// hi + lo of two FP32 numbers (|lo| <= ulp(hi)/2), giving a ~48-bit
// significand with FP32 range, computed on the FP32 pipes.
//
// Building blocks are the classical error-free transformations:
//   TwoSum (Knuth): s = a + b exactly as s + e;
//   FastTwoSum (Dekker), valid for |a| >= |b|;
//   TwoProd via FMA: p = a * b exactly as p + fma(a, b, -p).
// Addition is the "sloppy" variant (error bounded relative to |a| + |b|),
// which suits FFTs whose error is measured against the signal norm.
// None of these may be reassociated; the library is built without
// fast-math, and products are written with explicit fmaf.
#pragma once

#include <cuda_runtime.h>

#include "ttm_common.cuh"

namespace ttm {

struct df64 {
    float hi, lo;
    df64() = default;
    __host__ __device__ constexpr df64(float h, float l) : hi(h), lo(l) {}
    // split a double into hi + lo (exact to ~48 bits)
    __host__ __device__ constexpr df64(double d) : hi((float)d), lo((float)(d - (double)(float)d)) {}
    __host__ __device__ constexpr df64(int i) : hi((float)i), lo(0.f) {}
};

__device__ __forceinline__ df64 two_sum(float a, float b)
{
    const float s = a + b;
    const float v = s - a;
    const float e = (a - (s - v)) + (b - v);
    return df64(s, e);
}

__device__ __forceinline__ df64 fast_two_sum(float a, float b)
{
    const float s = a + b;
    const float e = b - (s - a);
    return df64(s, e);
}

__device__ __forceinline__ df64 two_prod(float a, float b)
{
    const float p = a * b;
    return df64(p, fmaf(a, b, -p));
}

__device__ __forceinline__ df64 operator+(df64 a, df64 b)
{
    const df64 s = two_sum(a.hi, b.hi);
    return fast_two_sum(s.hi, s.lo + (a.lo + b.lo));
}
__device__ __forceinline__ df64 operator-(df64 a) { return df64(-a.hi, -a.lo); }
__device__ __forceinline__ df64 operator-(df64 a, df64 b) { return a + (-b); }
__device__ __forceinline__ df64 operator*(df64 a, df64 b)
{
    const float p = a.hi * b.hi;
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    return fast_two_sum(p, e);
}
__device__ __forceinline__ df64& operator+=(df64& a, df64 b) { a = a + b; return a; }
__device__ __forceinline__ df64& operator-=(df64& a, df64 b) { a = a - b; return a; }
__device__ __forceinline__ df64& operator*=(df64& a, df64 b) { a = a * b; return a; }

// a / b by one Newton correction of the FP32 quotient
__device__ __forceinline__ df64 ddiv(df64 a, df64 b)
{
    const float q1 = a.hi / b.hi;
    const df64 r = a - b * df64(q1, 0.f);
    const float q2 = r.hi / b.hi;
    return fast_two_sum(q1, q2);
}

// A complex value as (heads of x and y, tails of x and y), 16 bytes that move
// with one vector access. Both parts go through the same operations, so the
// arithmetic below is written on the pairs with Blackwell's packed FP32
// instructions (two IEEE operations per issue slot, the same results as the
// scalar ones). The FMA pipe does not get wider by them (127 against 124
// lane operations per clock and SM), but the passes were short of issue
// slots: 80 % of them taken, 73 % of the FMA pipe's cycles.
struct __align__(16) dcx {
    float2 h, l;
    __device__ __forceinline__ df64 x() const { return df64(h.x, l.x); }
    __device__ __forceinline__ df64 y() const { return df64(h.y, l.y); }
};
__device__ __forceinline__ dcx make_dcx(df64 x, df64 y)
{
    dcx r;
    r.h = make_float2(x.hi, y.hi);
    r.l = make_float2(x.lo, y.lo);
    return r;
}

template <> struct cx_of<df64> { using type = dcx; };

template <> __host__ __device__ __forceinline__ dcx mk<df64>(df64 a, df64 b)
{
    dcx r;
    r.h.x = a.hi; r.h.y = b.hi;
    r.l.x = a.lo; r.l.y = b.lo;
    return r;
}

__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, neg2(b)); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }

// s + e = a + b exactly, in both parts (TwoSum)
__device__ __forceinline__ void two_sum2(float2 a, float2 b, float2& s, float2& e)
{
    s = add2(a, b);
    const float2 v = sub2(s, a);
    e = add2(sub2(a, sub2(s, v)), sub2(b, v));
}
__device__ __forceinline__ dcx fast_two_sum2(float2 a, float2 b)
{
    dcx r;
    r.h = add2(a, b);
    r.l = sub2(b, sub2(r.h, a));
    return r;
}
__device__ __forceinline__ dcx renormalise(dcx a) { return fast_two_sum2(a.h, a.l); }
__device__ __forceinline__ dcx operator-(dcx a)
{
    a.h = neg2(a.h);
    a.l = neg2(a.l);
    return a;
}

// Addition without the final renormalisation: the head sum is exact
// (TwoSum) and the tails are summed in FP32, so |lo| may exceed half an ulp
// of hi by a few ulps. The butterflies of one DFT add with it and
// renormalise their outputs once (dft in fft.cuh): 8 operations per
// addition instead of 11. Emulated on 3 000 random radix-8 DFTs the largest
// error grew from 1.29e-14 to 1.51e-14 of the input norm.
__device__ __forceinline__ dcx cadd(dcx a, dcx b)
{
    dcx r;
    float2 e;
    two_sum2(a.h, b.h, r.h, e);
    r.l = add2(e, add2(a.l, b.l));
    return r;
}
__device__ __forceinline__ dcx csub(dcx a, dcx b) { return cadd(a, -b); }
__device__ __forceinline__ dcx cconj(dcx a)
{
    a.h.y = -a.h.y;
    a.l.y = -a.l.y;
    return a;
}
// multiply by DIR * i
template <int DIR> __device__ __forceinline__ dcx cmul_diri(dcx a)
{
    dcx r;
    r.h = DIR > 0 ? make_float2(-a.h.y, a.h.x) : make_float2(a.h.y, -a.h.x);
    r.l = DIR > 0 ? make_float2(-a.l.y, a.l.x) : make_float2(a.l.y, -a.l.x);
    return r;
}
// by a real value
__device__ __forceinline__ dcx cscale(dcx a, df64 s)
{
    const float2 sh = dup2(s.hi);
    const float2 p = mul2(a.h, sh);
    float2 e = fma2(a.h, sh, neg2(p));
    e = fma2(a.h, dup2(s.lo), e);
    e = fma2(a.l, sh, e);
    return fast_two_sum2(p, e);
}

// The complex product, each part a b + c d in one pass: TwoProd of the two
// head products (their errors by FMA), TwoSum of the heads, every low-order
// term gathered into one FP32 sum, and a single FastTwoSum renormalisation.
// 19 operations per part where two products and an addition take 25, with
// one rounding of the low part fewer; the error bound is that of the sloppy
// addition of the two exact products.
__device__ __forceinline__ dcx cmul(dcx a, dcx b)
{
    const float2 axh = dup2(a.h.x), ayh = dup2(a.h.y), axl = dup2(a.l.x), ayl = dup2(a.l.y);
    const float2 rh = make_float2(-b.h.y, b.h.x), rl = make_float2(-b.l.y, b.l.x);  // i b
    const float2 p = mul2(axh, b.h);
    const float2 q = mul2(ayh, rh);
    float2 e = fma2(axh, b.h, neg2(p));
    e = add2(e, fma2(ayh, rh, neg2(q)));
    float2 s, se;
    two_sum2(p, q, s, se);
    e = fma2(axh, b.l, e);
    e = fma2(axl, b.h, e);
    e = fma2(ayh, rl, e);
    e = fma2(ayl, rh, e);
    return fast_two_sum2(s, add2(se, e));
}

// x h (1 + DIR i) and x h (-1 + DIR i): the sum and difference with DIR i x,
// renormalised, times h
template <int DIR> __device__ __forceinline__ dcx mul_w8_df(dcx x, df64 h, bool minus)
{
    const dcx r = cmul_diri<DIR>(x);
    return cscale(renormalise(minus ? csub(r, x) : cadd(x, r)), h);
}

}  // namespace ttm
