// Float-float arithmetic: a number as the unevaluated sum h + l of two FP32
// numbers (48 significand bits when |l| <= ulp(h) / 2).
//
// GB300 issues 128 FP32 operations per clock and SM but only 2 FP64 ones, so
// a multiply-add of float-floats (12 FP32 operations, no branch) costs a fifth
// of an FP64 one in issue slots. The error-free transformations are the
// published ones: the sum with its rounding error of Knuth (TAOCP vol. 2,
// 4.2.2; 6 operations, any order of the operands), the fast one of Dekker
// (Numer. Math. 18, 224 (1971); 3 operations, |a| >= |b|), and the product
// with its error from one fused multiply-add.
//
// Results are not renormalised: l keeps the sum of the rounding errors, which
// stays a few 2^-24 of the largest term of the sum that made it, and every
// operation takes both parts in. What is dropped is of the order of l l', so
// the error of an operation is a few 2^-48 of its largest term, as if the
// significand had 46 to 47 bits. The intrinsics keep the compiler from
// contracting a product and a sum, which would break the transformations.
#pragma once
#include <cuda_runtime.h>

namespace pimd {

using ::fma;   // beside the overload below

struct dfloat {
    float h, l;
    __host__ __device__ dfloat() {}
    __host__ __device__ constexpr dfloat(float a, float b) : h(a), l(b) {}
    // a double to 48 bits (exact for small integers)
    __host__ __device__ constexpr explicit dfloat(double a) : h((float)a), l((float)(a - (double)(float)a)) {}
    __host__ __device__ constexpr explicit dfloat(int a) : h((float)a), l((float)(a - (double)(float)a)) {}
    __device__ explicit operator double() const { return (double)h + (double)l; }
};

__device__ __forceinline__ dfloat two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
    return dfloat(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t)));
}
// |a| >= |b| or a == 0
__device__ __forceinline__ dfloat fast_two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    return dfloat(s, __fsub_rn(b, __fsub_rn(s, a)));
}
__device__ __forceinline__ dfloat operator-(dfloat a) { return dfloat(-a.h, -a.l); }
__device__ __forceinline__ dfloat operator+(dfloat a, dfloat b)
{
    const dfloat s = two_sum(a.h, b.h);
    return dfloat(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ dfloat operator-(dfloat a, dfloat b) { return a + (-b); }
__device__ __forceinline__ dfloat operator*(dfloat a, dfloat b)
{
    const float p = __fmul_rn(a.h, b.h);
    return dfloat(p, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p))));
}
__device__ __forceinline__ dfloat& operator+=(dfloat& a, dfloat b) { return a = a + b; }
__device__ __forceinline__ dfloat& operator-=(dfloat& a, dfloat b) { return a = a - b; }
// a b + c
__device__ __forceinline__ dfloat fma(dfloat a, dfloat b, dfloat c)
{
    const dfloat p = a * b, s = two_sum(c.h, p.h);
    return dfloat(s.h, __fadd_rn(__fadd_rn(s.l, c.l), p.l));
}
// a 2^k exactly (c a power of two)
__device__ __forceinline__ dfloat scale2(dfloat a, float c) { return dfloat(__fmul_rn(a.h, c), __fmul_rn(a.l, c)); }
// |l| <= ulp(h) / 2 again
__device__ __forceinline__ dfloat renorm(dfloat a) { return fast_two_sum(a.h, a.l); }

__device__ __forceinline__ dfloat ldg(const dfloat* p)
{
    const float2 v = __ldg((const float2*)p);
    return dfloat(v.x, v.y);
}
__device__ __forceinline__ double ldg(const double* p) { return __ldg(p); }
__device__ __forceinline__ float ldg(const float* p) { return __ldg(p); }

// 1/sqrt(x) for normal positive x: the hardware's single-precision estimate
// y0, then one step of Newton's iteration for y^-2 - x carried to second order,
// y = y0 (1 + e/2 + 3 e^2/8) with e = 1 - x y0^2 formed exactly enough by fused
// multiply-adds (|e| < 2^-21)
__device__ __forceinline__ dfloat rsqrt_r(dfloat x)
{
    const float y = rsqrtf(x.h);
    const float q = __fmul_rn(y, y), ql = __fmaf_rn(y, y, -q);
    float e = __fmaf_rn(-x.h, q, 1.0f);
    e = __fmaf_rn(-x.h, ql, e);
    e = __fmaf_rn(-x.l, q, e);
    return dfloat(y, __fmul_rn(y, __fmaf_rn(__fmul_rn(0.375f, e), e, __fmul_rn(0.5f, e))));
}

// Two float-floats side by side: every operation is the packed (f32x2) form of
// the scalar one, which issues one instruction for both lanes.
struct dfloat2 {
    float2 h, l;
    __device__ dfloat2() {}
    __device__ dfloat2(float2 a, float2 b) : h(a), l(b) {}
    __device__ dfloat2(dfloat a, dfloat b) : h(make_float2(a.h, b.h)), l(make_float2(a.l, b.l)) {}
    __device__ dfloat lane0() const { return dfloat(h.x, l.x); }
    __device__ dfloat lane1() const { return dfloat(h.y, l.y); }
};
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ dfloat2 exchange(dfloat2 a)
{
    return dfloat2(make_float2(a.h.y, a.h.x), make_float2(a.l.y, a.l.x));
}
__device__ __forceinline__ dfloat2 two_sum(float2 a, float2 b)
{
    const float2 s = __fadd2_rn(a, b), t = __fadd2_rn(s, neg2(a));
    return dfloat2(s, __fadd2_rn(__fadd2_rn(a, neg2(__fadd2_rn(s, neg2(t)))), __fadd2_rn(b, neg2(t))));
}
__device__ __forceinline__ dfloat2 operator*(dfloat2 a, dfloat2 b)
{
    const float2 p = __fmul2_rn(a.h, b.h);
    return dfloat2(p, __ffma2_rn(a.l, b.h, __ffma2_rn(a.h, b.l, __ffma2_rn(a.h, b.h, neg2(p)))));
}
__device__ __forceinline__ dfloat2 operator+(dfloat2 a, dfloat2 b)
{
    const dfloat2 s = two_sum(a.h, b.h);
    return dfloat2(s.h, __fadd2_rn(s.l, __fadd2_rn(a.l, b.l)));
}
__device__ __forceinline__ dfloat2 fma(dfloat2 a, dfloat2 b, dfloat2 c)
{
    const dfloat2 p = a * b, s = two_sum(c.h, p.h);
    return dfloat2(s.h, __fadd2_rn(__fadd2_rn(s.l, c.l), p.l));
}

}  // namespace pimd
