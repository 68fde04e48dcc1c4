// Running sums of the adjoint (fcas_grad.cu).
#pragma once

#include "fcas_ff.cuh"

namespace fcas {

// One running sum of the adjoint. The FP32 form's terms are FP32 values times float-float weights; their sum is
// kept as a pair of floats on the FP32 units (the compensated sum and dot product of Ogita, Rump & Oishi 2005: the
// rounding error of every product and every addition is formed exactly and added to the second word), ~11 FP32
// instructions per term where a binary64 one holds the SM's binary64 unit for as long as 64 FP32 instructions
// would take. The pair has some 48 bits, not binary64's 53: the second word is itself a plain FP32 sum, so with
// u = 2^-24 a thread's n terms are off by at most (n + 2)^2 u^2 of the sum of their sizes (n <= 128 for the
// longest segment: 2^-34), and every addition of two pairs adds a few 2^-48 of theirs. That is a thousandth of
// the terms' own rounding, which is what the FP32 form's gradients are off by: against 64 bits they are 1.2e-7
// (rms over 2^12 to 2^23 points, 31 cases), the same to four digits with binary64 sums in the pairs' place.
struct SumF {
    float h, l;
};
__host__ __device__ __forceinline__ void sum_zero(SumF& a) { a.h = a.l = 0.0f; }
__host__ __device__ __forceinline__ void sum_zero(double& a) { a = 0.0; }
__host__ __device__ __forceinline__ void sum_add(SumF& a, float q) {
    float e;
    a.h = ff_two_sum(a.h, q, e);
    a.l = f_add(a.l, e);
}
// a += w q for an exact float w
__host__ __device__ __forceinline__ void sum_add_w(SumF& a, float w, float q) {
    const float p = f_mul(w, q);
    float e;
    a.h = ff_two_sum(a.h, p, e);
    a.l = f_add(a.l, f_add(e, f_fma(w, q, -p)));
}
// a += (w.x + w.y) q
__host__ __device__ __forceinline__ void sum_add_w(SumF& a, float2 w, float q) {
    const float p = f_mul(w.x, q);
    float e;
    a.h = ff_two_sum(a.h, p, e);
    a.l = f_add(a.l, f_add(e, f_fma(w.y, q, f_fma(w.x, q, -p))));
}
__host__ __device__ __forceinline__ void sum_add(double& a, double q) { a += q; }
__host__ __device__ __forceinline__ void sum_add_w(double& a, double w, double q) { a += w * q; }
__host__ __device__ __forceinline__ SumF sum_of(SumF a, SumF b) {
    const ffloat r = ff_add(ffloat(a.h, a.l), ffloat(b.h, b.l));
    return SumF{r.h, r.l};
}
__host__ __device__ __forceinline__ double sum_of(double a, double b) { return a + b; }
// the pair as a float-float number (the second word may have outgrown half an ulp of the first)
__host__ __device__ __forceinline__ void sum_normalise(SumF& a) {
    float e;
    a.h = ff_two_sum(a.h, a.l, e);
    a.l = e;
}
__host__ __device__ __forceinline__ void sum_normalise(double&) {}
__device__ __forceinline__ SumF sum_xor(SumF a, int off) {
    return SumF{__shfl_xor_sync(0xffffffffu, a.h, off), __shfl_xor_sync(0xffffffffu, a.l, off)};
}
__device__ __forceinline__ double sum_xor(double a, int off) { return __shfl_xor_sync(0xffffffffu, a, off); }
__host__ __device__ __forceinline__ double sum_value(SumF a) { return (double)a.h + (double)a.l; }
__host__ __device__ __forceinline__ double sum_value(double a) { return a; }

}  // namespace fcas
