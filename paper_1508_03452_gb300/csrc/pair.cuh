// pair.cuh -- a number as the unevaluated sum of two float32 (high, low; about 48
// bits), for results that end as float32: GB300 has 128 float32 lanes and two float64
// lanes per SM, so the 7 to 11 float32 instructions of an operation here take a sixth
// of the time of the float64 one. Addition and multiplication are the error-free
// transformations of Knuth (two-sum) and of the fused multiply-add (Dekker's product),
// renormalised. Intrinsics keep the compiler from fusing across the steps.
#pragma once

#include "lattice.cuh"

namespace lb {

// (the overloads below would hide them here)
using ::fma;
using ::sqrt;

struct __align__(8) FloatPair {
    float h, l;
    FloatPair() = default;
    __host__ __device__ __forceinline__ constexpr FloatPair(float high, float low) : h(high), l(low) {}
    __host__ __device__ __forceinline__ constexpr explicit FloatPair(double v) : h((float)v), l((float)(v - (double)(float)v)) {}
    __host__ __device__ __forceinline__ constexpr explicit FloatPair(int v) : h((float)v), l(0.0f) {}
};

__device__ __forceinline__ FloatPair pair_norm(float s, float e)  // |s| >= |e|
{
    const float h = __fadd_rn(s, e);
    return {h, __fsub_rn(e, __fsub_rn(h, s))};
}
__device__ __forceinline__ FloatPair operator+(FloatPair a, FloatPair b)
{
    const float s = __fadd_rn(a.h, b.h), t = __fsub_rn(s, a.h);
    const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, t)), __fsub_rn(b.h, t));
    return pair_norm(s, __fadd_rn(e, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ FloatPair operator-(FloatPair a) { return {-a.h, -a.l}; }
__device__ __forceinline__ FloatPair operator-(FloatPair a, FloatPair b) { return a + (-b); }
__device__ __forceinline__ FloatPair operator*(FloatPair a, FloatPair b)
{
    const float p = __fmul_rn(a.h, b.h);
    return pair_norm(p, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p))));
}
// 1/x and 1/sqrt(x) by Newton's iteration from the float32 value
__device__ __forceinline__ FloatPair pair_rcp(FloatPair x)
{
    const float r = __frcp_rn(x.h);
    const FloatPair e = FloatPair(1.0f, 0.0f) - x * FloatPair(r, 0.0f);
    return pair_norm(r, __fmul_rn(r, __fmaf_rn(e.h, e.h, __fadd_rn(e.h, e.l))));
}
__device__ __forceinline__ FloatPair pair_rsqrt(FloatPair x)
{
    const float r = rsqrtf(x.h);
    const FloatPair e = FloatPair(1.0f, 0.0f) - x * (FloatPair(r, 0.0f) * FloatPair(r, 0.0f));
    return pair_norm(r, __fmul_rn(r, __fmaf_rn(0.375f * e.h, e.h, 0.5f * __fadd_rn(e.h, e.l))));
}
__device__ __forceinline__ FloatPair operator/(FloatPair a, FloatPair b) { return a * pair_rcp(b); }
__device__ __forceinline__ FloatPair sqrt(FloatPair a) { return a * pair_rsqrt(a); }
__device__ __forceinline__ FloatPair fma(FloatPair a, FloatPair b, FloatPair c) { return a * b + c; }
__device__ __forceinline__ FloatPair mul_rn(FloatPair a, FloatPair b) { return a * b; }
__device__ __forceinline__ FloatPair rsqrt_newton(FloatPair x) { return pair_rsqrt(x); }
__device__ __forceinline__ FloatPair rcp_approx(FloatPair x) { return pair_rcp(x); }

// the parameters of a run as pairs
inline Phys<FloatPair> pair_phys(const Phys<double>& k)
{
    Phys<FloatPair> o;
    static_assert(sizeof(FloatPair) == sizeof(double) && sizeof(Phys<FloatPair>) == sizeof(Phys<double>) &&
                      offsetof(Phys<FloatPair>, maxit) == offsetof(Phys<double>, maxit),
                  "every member before maxit is a number");
    for (size_t i = 0; i < offsetof(Phys<double>, maxit) / sizeof(double); ++i) {
        double v;
        memcpy(&v, reinterpret_cast<const char*>(&k) + i * sizeof(double), sizeof(v));
        const FloatPair p(v);
        memcpy(reinterpret_cast<char*>(&o) + i * sizeof(p), &p, sizeof(p));
    }
    o.maxit = k.maxit;
    return o;
}

}  // namespace lb
