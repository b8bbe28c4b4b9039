// Arithmetic on pairs of floats: a value is the unevaluated sum h + l of two binary32 numbers
// with |l| at most about one unit in the last place of h, good for about 46 significant bits.
//
// The mixed-precision Kalman update is built from it (kf_math.cuh).  This GPU issues a
// double-precision instruction at 1/64 of the single-precision rate, so a pair operation of 3 to
// 18 single-precision instructions is several times cheaper than the one double instruction it
// stands for.  The building blocks are the error-free transformations of Knuth (two_sum) and
// Dekker (fast_two_sum; the product's error comes from one fused multiply-add), as in T. J.
// Dekker, "A floating-point technique for extending the available precision", Numer. Math. 18
// (1971).  Every operation is written with the rounding intrinsics, which the compiler never
// contracts or reorders.  Host and device share the code (a test runs it on the host).
#pragma once

#include <cuda_runtime.h>
#include <math.h>

namespace tkf {

#define TKF_PAIR __host__ __device__ __forceinline__
#ifdef __CUDA_ARCH__
TKF_PAIR float add_rn(float a, float b) { return __fadd_rn(a, b); }
TKF_PAIR float sub_rn(float a, float b) { return __fsub_rn(a, b); }
TKF_PAIR float mul_rn(float a, float b) { return __fmul_rn(a, b); }
TKF_PAIR float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
TKF_PAIR float rcp_rn(float a) { return __frcp_rn(a); }
#else  // compiled with contraction off
TKF_PAIR float add_rn(float a, float b) { return a + b; }
TKF_PAIR float sub_rn(float a, float b) { return a - b; }
TKF_PAIR float mul_rn(float a, float b) { return a * b; }
TKF_PAIR float fma_rn(float a, float b, float c) { return fmaf(a, b, c); }
TKF_PAIR float rcp_rn(float a) { return 1.0f / a; }
#endif

struct pair32 {
    float h, l;
};

// a + b = s + e exactly
TKF_PAIR pair32 two_sum(float a, float b)
{
    const float s = add_rn(a, b), t = sub_rn(s, a);
    return {s, add_rn(sub_rn(a, sub_rn(s, t)), sub_rn(b, t))};
}
// the same for |a| >= |b|
TKF_PAIR pair32 fast_two_sum(float a, float b)
{
    const float s = add_rn(a, b);
    return {s, sub_rn(b, sub_rn(s, a))};
}
// a b = p + e exactly
TKF_PAIR pair32 two_prod(float a, float b)
{
    const float p = mul_rn(a, b);
    return {p, fma_rn(a, b, -p)};
}
TKF_PAIR pair32 add(pair32 a, pair32 b)
{
    const pair32 s = two_sum(a.h, b.h);
    return fast_two_sum(s.h, add_rn(s.l, add_rn(a.l, b.l)));
}
TKF_PAIR pair32 add(pair32 a, float b)
{
    const pair32 s = two_sum(a.h, b);
    return fast_two_sum(s.h, add_rn(s.l, a.l));
}
// Products keep the rounding error of h b.h in l and are not renormalised: l stays within about
// two units of h's last place, which every user above and below allows for.
TKF_PAIR pair32 mul(pair32 a, float b)
{
    const float p = mul_rn(a.h, b);
    return {p, fma_rn(a.l, b, fma_rn(a.h, b, -p))};
}
TKF_PAIR pair32 mul(float b, pair32 a) { return mul(a, b); }
TKF_PAIR pair32 mul(pair32 a, pair32 b)
{
    const float p = mul_rn(a.h, b.h);
    return {p, fma_rn(a.l, b.h, fma_rn(a.h, b.l, fma_rn(a.h, b.h, -p)))};
}
TKF_PAIR pair32 mul(float a, float b) { return two_prod(a, b); }
// 1 / a: one Newton step y + y (1 - a y) from the rounded reciprocal of a.h
TKF_PAIR pair32 recip(pair32 a)
{
    const float y = rcp_rn(a.h);
    return fast_two_sum(y, mul_rn(y, fma_rn(-a.l, y, fma_rn(-a.h, y, 1.0f))));
}
// p - a b - c d rounded once: the four parts that follow the leading sums are far smaller
template <class A, class B, class C, class D> TKF_PAIR float minus_products(float p, A a, B b, C c, D d)
{
    const pair32 ab = mul(a, b), cd = mul(c, d);
    const pair32 s = two_sum(p, -ab.h), t = two_sum(s.h, -cd.h);
    return add_rn(t.h, add_rn(sub_rn(s.l, ab.l), sub_rn(t.l, cd.l)));
}
#undef TKF_PAIR

}  // namespace tkf
