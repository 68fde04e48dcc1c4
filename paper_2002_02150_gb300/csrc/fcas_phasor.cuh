// Runs of phasors in equal steps, for the accurate forms' pass A (binary64 and float-float).
#pragma once

#include <type_traits>

#include "fcas_ff.cuh"
#include "fcas_internal.cuh"

namespace fcas {

// a x + y and the next value of a three-term recurrence, c2 b - a per component
__host__ __device__ __forceinline__ double axpy(double a, double x, double y) { return fma(a, x, y); }
__host__ __device__ __forceinline__ ffloat axpy(ffloat a, ffloat x, ffloat y) { return ff_fma(a, x, y); }
// The phasor after b in the run a, b: 2 cos(theta) b - a, half the arithmetic of the product b step in binary64 and
// 30 instructions instead of 38 in float-float.
__host__ __device__ __forceinline__ double2 three_term(double2 a, double2 b, double2 step) {
    const double c2 = 2.0 * step.x;
    return make_double2(fma(c2, b.x, -a.x), fma(c2, b.y, -a.y));
}
__host__ __device__ __forceinline__ ff2 three_term(ff2 a, ff2 b, ff2 step) {
    const ffloat c2(2.0f * step.x.h, 2.0f * step.x.l);
    return ff2{ff_fma(c2, b.x, -a.x), ff_fma(c2, b.y, -a.y)};
}

// The index whose phasor phasor_run is given.
__host__ __device__ constexpr int phasor_anchor(int n) { return n >= 16 ? 5 : n >= 4 ? 1 : 0; }

// N phasors e^{i (phi + q theta)}, q = 0..N-1, given to use(q, phasor) from the one at q = phasor_anchor(N), the
// step e^{i theta} and, for N >= 8, step4 = e^{4 i theta} (each accurate by itself). Blocks of four: the anchors
// of the other blocks are products by step4 (at most two in a row), in a block the phasor above its anchor is a
// product by the step, and the outer two follow by one three-term step each way (eight float-float phasors: by
// products). Longer recurrences lose accuracy: a rounding k steps back grows by sin((k + 1) theta) / sin(theta),
// about k + 1 for a small theta. Largest error with theta in 0..0.39, N = 8 / 16: binary64 in units of 2^-53
// products in a row 7.1 / 12.3, one recurrence outwards from the middle 13.5 / 44.0, these blocks 5.0 / 5.7;
// float-float in units of 2^-48 products 7.7 / 9.0, these blocks 4.9 / 7.3 (eight with three-term steps 7.7, and
// more than the products on average). N <= 4: products outwards from the anchor (2.9 against 4.0 for products in a
// row and 4.5 for the recurrence). Measured against one recurrence throughout: binary64 pass A 6.20 -> 6.30 ms per 4
// particles of the 60-min workload, 432 -> 447 us per 40 of 64 s; float-float 3.64 -> 3.59 ms per 8 of 60 min, 1.89 ->
// 2.04 ms per 16 of 15 min.
template <typename Real, int N, typename F>
__host__ __device__ __forceinline__ void phasor_run(cplx<Real> at_anchor, cplx<Real> step, cplx<Real> step4, F&& use) {
    using C = cplx<Real>;
    constexpr int A = phasor_anchor(N);
    constexpr bool kThreeTerm = std::is_same<Real, double>::value || N >= 16;
    const C back = cconj(step);
    if constexpr (N >= 8) {
        C a = A > 1 ? cmul(at_anchor, cconj(step4)) : at_anchor;
#pragma unroll
        for (int q = 0; q < N; q += 4) {
            if (q + 1 == A) a = at_anchor;
            else if (q > 0) a = cmul(a, step4);
            const C up = cmul(a, step);
            use(q, kThreeTerm ? three_term(up, a, back) : cmul(a, back));
            use(q + 1, a);
            use(q + 2, up);
            use(q + 3, kThreeTerm ? three_term(a, up, step) : cmul(up, step));
        }
    } else {
        if constexpr (A > 0) use(0, cmul(at_anchor, back));
        C a = at_anchor;
#pragma unroll
        for (int q = A; q < N; ++q) {
            use(q, a);
            if (q + 1 < N) a = cmul(a, step);
        }
    }
}

}  // namespace fcas
