// Double-word ("float-float") arithmetic for the FP32 units: a value is the unevaluated sum h + l
// of two floats with |l| <= ulp(h)/2 (Dekker 1971; error bounds of Joldes, Muller & Popescu 2017).
#pragma once

#include <cmath>

#include <cuda_runtime.h>

namespace fcas {

struct ffloat {
    float h, l;
    ffloat() = default;
    __host__ __device__ constexpr ffloat(float hi, float lo) : h(hi), l(lo) {}
    __host__ __device__ ffloat(double d) : h((float)d), l((float)(d - (double)(float)d)) {}
};

struct ff2 {
    ffloat x, y;
};

__host__ __device__ __forceinline__ double ff_to_double(ffloat a) { return (double)a.h + (double)a.l; }

#ifdef __CUDACC__
// single roundings that the compiler may not contract (host code: compiled with -ffp-contract=off)
#ifdef __CUDA_ARCH__
__device__ __forceinline__ float f_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float f_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float f_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float f_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
#else
inline float f_add(float a, float b) { return a + b; }
inline float f_sub(float a, float b) { return a - b; }
inline float f_mul(float a, float b) { return a * b; }
inline float f_fma(float a, float b, float c) { return fmaf(a, b, c); }
#endif
// s + e = a + b exactly (Knuth's two-sum)
__host__ __device__ __forceinline__ float ff_two_sum(float a, float b, float& e) {
    const float s = f_add(a, b);
    const float bb = f_sub(s, a);
    e = f_add(f_sub(a, f_sub(s, bb)), f_sub(b, bb));
    return s;
}
// s + e = a + b exactly when |a| >= |b| (or a = 0)
__host__ __device__ __forceinline__ float ff_fast_two_sum(float a, float b, float& e) {
    const float s = f_add(a, b);
    e = f_sub(b, f_sub(s, a));
    return s;
}
// a + b with an absolute error of a few units of 2^-48 (|a| + |b|): enough for normwise-accurate
// transforms (the sloppy double-word sum: one two-sum of the high parts)
__host__ __device__ __forceinline__ ffloat ff_add(ffloat a, ffloat b) {
    float e;
    const float s = ff_two_sum(a.h, b.h, e);
    e = f_add(e, f_add(a.l, b.l));
    float lo;
    const float hi = ff_fast_two_sum(s, e, lo);
    return ffloat(hi, lo);
}
// a + b for a float b (the same sum with a zero low part of b)
__device__ __forceinline__ ffloat ff_add_f(ffloat a, float b) {
    float e;
    const float s = ff_two_sum(a.h, b, e);
    e = __fadd_rn(e, a.l);
    float lo;
    const float hi = ff_fast_two_sum(s, e, lo);
    return ffloat(hi, lo);
}
__host__ __device__ __forceinline__ ffloat ff_neg(ffloat a) { return ffloat(-a.h, -a.l); }
__host__ __device__ __forceinline__ ffloat ff_sub(ffloat a, ffloat b) { return ff_add(a, ff_neg(b)); }
// a b: the exact leading product by a fused multiply-add plus the cross terms (double-word product)
__device__ __forceinline__ ffloat ff_mul(ffloat a, ffloat b) {
    const float p = __fmul_rn(a.h, b.h);
    float e = __fmaf_rn(a.h, b.h, -p);
    e = __fmaf_rn(a.h, b.l, e);
    e = __fmaf_rn(a.l, b.h, e);
    float lo;
    const float hi = ff_fast_two_sum(p, e, lo);
    return ffloat(hi, lo);
}

__host__ __device__ __forceinline__ ffloat operator+(ffloat a, ffloat b) { return ff_add(a, b); }
__host__ __device__ __forceinline__ ffloat operator-(ffloat a, ffloat b) { return ff_sub(a, b); }
__host__ __device__ __forceinline__ ffloat operator-(ffloat a) { return ff_neg(a); }
__device__ __forceinline__ ffloat operator*(ffloat a, ffloat b) { return ff_mul(a, b); }
__device__ __forceinline__ ffloat& operator+=(ffloat& a, ffloat b) { return a = ff_add(a, b); }
__device__ __forceinline__ bool operator>(ffloat a, ffloat b) { return a.h > b.h || (a.h == b.h && a.l > b.l); }
__device__ __forceinline__ bool operator==(ffloat a, ffloat b) { return a.h == b.h && a.l == b.l; }

// a b as an unnormalised pair (p, e), |e| within a few ulp(p): for a sum that normalises its result
__host__ __device__ __forceinline__ ffloat ff_mul_pair(ffloat a, ffloat b) {
    const float p = f_mul(a.h, b.h);
    float e = f_fma(a.h, b.h, -p);
    e = f_fma(a.h, b.l, e);
    return ffloat(p, f_fma(a.l, b.h, e));
}
// a + b as an unnormalised pair, |second word| within two ulps of the first
__device__ __forceinline__ ffloat ff_add_pair(ffloat a, ffloat b) {
    float e;
    const float s = ff_two_sum(a.h, b.h, e);
    return ffloat(s, __fadd_rn(e, __fadd_rn(a.l, b.l)));
}
// a b + c, normalised once (15 instructions where product and sum take 18)
__host__ __device__ __forceinline__ ffloat ff_fma(ffloat a, ffloat b, ffloat c) { return ff_add(ff_mul_pair(a, b), c); }

__device__ __forceinline__ ff2 operator+(ff2 a, ff2 b) { return ff2{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ ff2 operator-(ff2 a, ff2 b) { return ff2{a.x - b.x, a.y - b.y}; }
// complex product: the four products stay unnormalised pairs (38 instructions instead of 50)
__host__ __device__ __forceinline__ ff2 cmul(ff2 a, ff2 b) {
    return ff2{ff_sub(ff_mul_pair(a.x, b.x), ff_mul_pair(a.y, b.y)), ff_add(ff_mul_pair(a.x, b.y), ff_mul_pair(a.y, b.x))};
}
__host__ __device__ __forceinline__ ff2 cconj(ff2 a) { return ff2{a.x, -a.y}; }
__host__ __device__ __forceinline__ ff2 mkc(ffloat x, ffloat y) { return ff2{x, y}; }
template <int S> __device__ __forceinline__ ff2 mul_si(ff2 a) { return S > 0 ? ff2{-a.y, a.x} : ff2{a.y, -a.x}; }

__device__ __forceinline__ float shfl_down_r(float v, int off) { return __shfl_down_sync(0xffffffffu, v, off); }
__device__ __forceinline__ double shfl_down_r(double v, int off) { return __shfl_down_sync(0xffffffffu, v, off); }
__device__ __forceinline__ ffloat shfl_down_r(ffloat v, int off) {
    return ffloat(__shfl_down_sync(0xffffffffu, v.h, off), __shfl_down_sync(0xffffffffu, v.l, off));
}
__device__ __forceinline__ double to_double(float v) { return (double)v; }
__device__ __forceinline__ double to_double(double v) { return v; }
__device__ __forceinline__ double to_double(ffloat v) { return ff_to_double(v); }
#endif

}  // namespace fcas
