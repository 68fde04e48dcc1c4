// Internal declarations shared by the CUDA translation units of libfcas.
#pragma once

#include <cmath>

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/fcas.h"

namespace fcas {

constexpr double kTwoPi = 6.283185307179586476925286766559;
constexpr double kCLight = 299792458.0;
constexpr double kRank1Rtol = 1e-12;   // det G < kRank1Rtol (tr G / 2)^2 -> rank-1 projection
constexpr int kTwLoBits = 12;          // two-level table for e^{2 pi i m / N}: m = hi * 4096 + lo

// ------------------------------------------------------------------------------------------
// Overlapped launches. The kernels of one evaluation follow each other directly on the stream; each is
// launched so that its CTAs may be scheduled (and read what the call does not write) while the last CTAs of
// its predecessor drain, and waits for the predecessor's completion before anything else (chain_wait).
//  - A wait covers the predecessor alone. chain_go therefore stands after chain_wait: it lets the successor be
//    scheduled once every CTA of this grid has started and waited, so that a grid starts with all grids but its
//    predecessor complete. Letting it go before the wait gave wrong results (a group of mixed forms); which read
//    was too early was not established, and nothing here relies on it.
//  - What a kernel of the call writes is read through plain pointers: a const __restrict__ pointer or a read-only
//    load would let the compiler move the read ahead of the wait. The adjoint's kernels read theta and tc through
//    such pointers: these are complete before the call's first kernel, which is launched the ordinary way.
//  - Both do nothing in a kernel launched without the attribute or without a successor that has it.
// Used where a chunk covers at most 2^23 points of transform (chain_pays). us per call without / with, FP32:
// 512 particles of 2^12 points 43.1 / 39.1; 2^14: 128 42.6 / 34.9, 512 92.4 / 87.4; 2^16: 32 42.1 / 33.1, 128 90.6 /
// 84.0; 2^21: 1 47.3 / 39.2, 4 115 / 109; one of 2^23 141.7 / 135.2. The gaps between kernels count for less the
// more points there are; beyond the line they still do (512 particles of 2^16 331 / 304, 16 of 2^21 346 / 339, four
// of 2^23 410 / 403), so a line further up would gain there too.
// ------------------------------------------------------------------------------------------
#ifdef __CUDACC__
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_go() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

inline bool chain_pays(int64_t particles, int log_n) { return particles <= ((int64_t)1 << 23 >> log_n); }

template <typename... P, typename... A>
inline cudaError_t launch_chained(bool chained, void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                  A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = chained ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}
#endif

// ------------------------------------------------------------------------------------------
// complex helpers on float2 / double2
// ------------------------------------------------------------------------------------------
template <typename R> struct cplx_of;
template <> struct cplx_of<float> { using type = float2; };
template <> struct cplx_of<double> { using type = double2; };
template <typename R> using cplx = typename cplx_of<R>::type;

__host__ __device__ __forceinline__ float2 mkc(float x, float y) { return make_float2(x, y); }
__host__ __device__ __forceinline__ double2 mkc(double x, double y) { return make_double2(x, y); }
__device__ __forceinline__ float2 operator+(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 operator-(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 operator+(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 operator-(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__host__ __device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__host__ __device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
__host__ __device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }
__host__ __device__ __forceinline__ double2 cconj(double2 a) { return make_double2(a.x, -a.y); }
__device__ __forceinline__ float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
__device__ __forceinline__ double2 cscale(double2 a, double s) { return make_double2(a.x * s, a.y * s); }
// multiply by S*i (S = +1 or -1)
template <int S> __device__ __forceinline__ float2 mul_si(float2 a) {
    return S > 0 ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}
template <int S> __device__ __forceinline__ double2 mul_si(double2 a) {
    return S > 0 ? make_double2(-a.y, a.x) : make_double2(a.y, -a.x);
}

// ------------------------------------------------------------------------------------------
// Per-particle quantities computed once per evaluation in binary64 (geometry kernel).
// ------------------------------------------------------------------------------------------
struct ParticleParams {
    double c[4];                   // chirp phase coefficients [turns] of phi^-5/3, phi^-1, phi^-2/3, phi^-1/3
    double dturn[FCAS_MAX_DET];    // Delta^i * df: delay phase [turns] per frequency bin
    double u[FCAS_MAX_DET][2];     // U^i = (F+, Fx)(alpha, delta, psi = 0)
    double ginv[3];                // (G^-1)_{11}, (G^-1)_{12}, (G^-1)_{22} with the scaled template norms
    double chol[3];                // G^-1 = L L^T, L = [[l11, 0], [l21, l22]]: (l11, l21, l22)
    // Network weights: Gamma^2(t) = |sum_i w1_i Z_i(t)|^2 + |sum_i w2_i Z_i(t)|^2 with
    // w1_i = l11 U+^i + l21 Ux^i, w2_i = l22 Ux^i (L^T applied to U).
    double w1[FCAS_MAX_DET], w2[FCAS_MAX_DET];
    // float-float copies for the FP32 form (hi + lo)
    float ch[4], cl[4];
    float dh[FCAS_MAX_DET], dl[FCAS_MAX_DET];
    float w1f[FCAS_MAX_DET], w2f[FCAS_MAX_DET];
    float2 dstep[FCAS_MAX_DET];    // e^{2 pi i S Delta^i df}, S = N / V_A: the FP32 pass A's step of the
                                   // delay phasor between a thread's consecutive bins (binary64 phase)
    // binary64 and float-float pass A: delays relative to detector 0's (whose own phase joins the chirp
    // phase) and the phasors of the same step and of four, e^{2 pi i S rturn}; filled for those forms only
    double rturn[FCAS_MAX_DET];
    double2 rstep[FCAS_MAX_DET];
    double2 rstep4[FCAS_MAX_DET];  // e^{2 pi i 4 S rturn}
    int32_t valid;                 // 0: non-finite / non-positive input -> fitness NaN, tc -1
    int32_t taylor_ok;             // FP32 pass A may step the chirp phase from an anchor bin to the
                                   // next 3 (bit 0) or 7 (bit 1) bins: remainder below 1e-7 turns
};

// ------------------------------------------------------------------------------------------
// Launch shapes. Pass A transforms columns of length N2 (K1B columns per CTA), pass B rows of
// length N1 (TB rows per CTA); each transform is held by L / V threads with V = min(16, L)
// values per thread. Pass A also keeps K1B <= L so that K1B divides N1 (N1 >= N2 = L).
// ------------------------------------------------------------------------------------------
__host__ __device__ constexpr int imin_c(int a, int b) { return a < b ? a : b; }
__host__ __device__ constexpr int imax_c(int a, int b) { return a > b ? a : b; }
#ifndef FCAS_PASS_A_SUB
#define FCAS_PASS_A_SUB 16            // adjacent column blocks of one particle scheduled together
#endif
#ifndef FCAS_SPLIT_BIAS
#define FCAS_SPLIT_BIAS 0             // N2 = 2^(floor(log2 N / 2) - bias): a smaller pass-A transform
#endif
__host__ __device__ constexpr int shape_v(int log_l) { return log_l >= 4 ? 16 : (1 << log_l); }
// Columns per pass-A CTA of a form (FCAS_PREC_*). FP32: CTAs of 128 threads, but at least 4 columns (row pieces
// of 64 bytes; 2 columns write 32-byte pieces and lose 12 % at 2^11 points) while a CTA stays within 512
// threads. Several small CTAs per SM are in different phases (loads, arithmetic, exchanges) at any time, one
// large one is in the same phase throughout: us per 64 particles with 4 / 8 / 16 columns, 2^8 points 28.2 /
// 27.4 / 29.6, 2^9 points 101 / 110 / 121, 2^10 points 778 / 827 / -. Sixteen columns form every bin's chirp phase,
// two to eight step it from shared anchor bins where the particle's bound allows: the errors against 64 bits are the
// same to within their scatter (rms of Gamma^2 over 924 to 1232 particles against every bin's phase, 2^18 / 2^19 / 2^20 /
// 2^21 points: 4 columns 1.009 / 1.004 / 0.985 / 0.989, 8 columns 1.000 / 1.000 / 0.995 / 0.998, each +- 0.008). Binary64: 128 threads for the same reason
// (2^8 points, 40 particles: 8 / 16 columns 463 / 520 us; 2^11 points, 4 particles: 1 / 2 columns 6.78 / 6.92
// ms). Float-float: 256 threads, whose warps share the instruction fetches of its long unrolled code.
__host__ __device__ constexpr int pass_a_k1b(int log_l, int form) {
    const int g = (1 << log_l) / shape_v(log_l);   // threads per column
    const int k = form == FCAS_PREC_FP32 ? imax_c(128 / g, imin_c(4, 512 / g)) : (form == FCAS_PREC_FP64 ? 128 : 256) / g;
    return imin_c(imin_c(16, imax_c(1, k)), 1 << log_l);
}
// Threads a pass-B CTA holds where rows are shorter: FP32 64 (us per 64 particles with CTAs of 256 / 128 / 64
// threads: 2^8 points 19.9 / 17.3 / 16.8, 2^9 points 80 / 76 / 75, 2^11 points 469 / 411 / 411), binary64 128,
// float-float 256 (2^11 points, 16 particles: 128 / 256 threads 1076 / 929 us; shared instruction fetches).
__host__ __device__ constexpr int pass_b_target(int form) {
    return form == FCAS_PREC_FP32 ? 64 : form == FCAS_PREC_FP64 ? 128 : 256;
}
__host__ __device__ constexpr int pass_b_tb(int log_l, int form) {
    return imin_c(imin_c(16, imax_c(1, pass_b_target(form) / ((1 << log_l) / shape_v(log_l)))), (1 << log_l) / 2);
}
__host__ __device__ constexpr int pass_b_threads(int log_l, int form) {
    return pass_b_tb(log_l, form) * ((1 << log_l) / shape_v(log_l));
}
// Transforms per particle between the passes: the two network-weighted series.
constexpr int kSeries = 2;

// Smallest/largest supported transform lengths; each pass transforms at most 2^13 points.
constexpr int kMinLogN = 4;
constexpr int kMaxLogN = 24;
constexpr int kMaxLogPass = 13;
__host__ __device__ constexpr int split_log_n2_with(int log_n, int bias) {
    return imax_c(2, imax_c(log_n - kMaxLogPass, log_n / 2 - bias));
}

}  // namespace fcas
