// iod_ff_ops.cuh -- FP32 words and their error-free transformations, single and in pairs
// (FADD2/FMUL2/FFMA2 take one issue slot for two operations).  Every operation is rounded
// to nearest by itself: the _rn intrinsics keep the compiler from fusing a product into a
// sum, which would change the rounding that the transformations account for.
#pragma once

#ifdef __CUDACC__
#include <cuda_runtime.h>
#define IOD_HD __device__ __forceinline__
#define IOD_CALL static __device__ __noinline__
#else
#include <math.h>
#include <string.h>
#define IOD_HD static inline
#define IOD_CALL static
struct float2 {
    float x, y;
};
#endif

namespace iod {
namespace ff {

#ifdef __CUDACC__
IOD_HD float add(float a, float b) { return __fadd_rn(a, b); }
IOD_HD float sub(float a, float b) { return __fsub_rn(a, b); }
IOD_HD float mul(float a, float b) { return __fmul_rn(a, b); }
IOD_HD float ffma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
IOD_HD float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
IOD_HD float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
IOD_HD float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// the hardware's estimate of x^(-1/2) (relative error below 2^-22)
IOD_HD float rsqrt_est(float x)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// the hardware's x^(2/3) for x >= 0 (limits only)
IOD_HD float pow23_est(float x)
{
    float r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    r = __fmul_rn(r, 0.6666667f);
    asm("ex2.approx.ftz.f32 %0, %0;" : "+f"(r));
    return r;
}
// bits of a value
IOD_HD unsigned int bits_of(float a) { return __float_as_uint(a); }
IOD_HD float float_of(unsigned int b) { return __uint_as_float(b); }
IOD_HD unsigned int high_word(double d) { return (unsigned int)__double2hiint(d); }
IOD_HD unsigned int low_word(double d) { return (unsigned int)__double2loint(d); }
IOD_HD double from_halves(unsigned int hi, unsigned int lo) { return __hiloint2double((int)hi, (int)lo); }
#else
IOD_HD float add(float a, float b) { return a + b; }
IOD_HD float sub(float a, float b) { return a - b; }
IOD_HD float mul(float a, float b) { return a * b; }
IOD_HD float ffma(float a, float b, float c) { return fmaf(a, b, c); }
IOD_HD float2 add2(float2 a, float2 b) { return float2{a.x + b.x, a.y + b.y}; }
IOD_HD float2 mul2(float2 a, float2 b) { return float2{a.x * b.x, a.y * b.y}; }
IOD_HD float2 fma2(float2 a, float2 b, float2 c) { return float2{fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y)}; }
IOD_HD float rsqrt_est(float x) { return IOD_RSQRT_EST(x); }
IOD_HD float pow23_est(float x) { return powf(x, 0.6666667f); }
IOD_HD unsigned int bits_of(float a)
{
    unsigned int b;
    memcpy(&b, &a, sizeof b);
    return b;
}
IOD_HD float float_of(unsigned int b)
{
    float a;
    memcpy(&a, &b, sizeof a);
    return a;
}
IOD_HD unsigned long long word_of(double d)
{
    unsigned long long b;
    memcpy(&b, &d, sizeof b);
    return b;
}
IOD_HD unsigned int high_word(double d) { return (unsigned int)(word_of(d) >> 32); }
IOD_HD unsigned int low_word(double d) { return (unsigned int)word_of(d); }
IOD_HD double from_halves(unsigned int hi, unsigned int lo)
{
    const unsigned long long b = ((unsigned long long)hi << 32) | lo;
    double d;
    memcpy(&d, &b, sizeof d);
    return d;
}
#endif

IOD_HD float2 mk2(float a, float b)
{
    float2 r;
    r.x = a;
    r.y = b;
    return r;
}
IOD_HD float2 bc2(float a) { return mk2(a, a); }
IOD_HD float2 neg2(float2 a) { return mk2(-a.x, -a.y); }
IOD_HD float2 sub2(float2 a, float2 b) { return add2(a, neg2(b)); }

// s + e = a + b exactly.  One value: the larger first, then Dekker's three operations (the
// comparison and the selections run on the otherwise idle ALU; 3% of a step against
// Knuth's six FP32 ones).  Pairs: Knuth's, six instructions for both, where sorting would
// take nine.
IOD_HD void two_sum(float a, float b, float &s, float &e)
{
    const bool g = fabsf(a) >= fabsf(b);
    const float x = g ? a : b, y = g ? b : a;
    s = add(x, y);
    e = sub(y, sub(s, x));
}
IOD_HD void two_sum2(float2 a, float2 b, float2 &s, float2 &e)
{
    s = add2(a, b);
    const float2 t = sub2(s, a);
    e = add2(sub2(a, sub2(s, t)), sub2(b, t));
}
// the same for |a| >= |b| (Dekker)
IOD_HD void fast_two_sum(float a, float b, float &s, float &e)
{
    s = add(a, b);
    e = sub(b, sub(s, a));
}
IOD_HD void fast_two_sum2(float2 a, float2 b, float2 &s, float2 &e)
{
    s = add2(a, b);
    e = sub2(b, sub2(s, a));
}

}  // namespace ff
}  // namespace iod
