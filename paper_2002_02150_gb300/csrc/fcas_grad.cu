// Adjoint of the coherent fitness at a fixed t_c (envelope theorem): d Gamma^2(theta, t*) / d theta
// for theta = (alpha, delta, tau0, tau1.5) at the argmax t* of a previous fitness evaluation.
//
// With Z_i = sum_k Q_i[k] e^{2 pi i k t*/N}, W = sum_i U^i Z_i and Gamma^2 = Re(W^H G^-1 W) (Sec. II.C),
//   d Gamma^2 = 2 Re(dW^H G^-1 W) - W^H (G^-1 dG G^-1) W,   dW = sum_i (dU^i Z_i + U^i dZ_i),
//   dG = sum_i sigma_i^2 (dU^i U^iT + U^i dU^iT),
// and, since Q_i[k] carries the phase 2 pi (psi(f_k)/2pi + k Delta^i df) (Sec. II.B, II.D),
//   dZ_i/d(alpha, delta) = 2 pi i (d(Delta^i df)/d(alpha, delta)) sum_k k Q_i e^{...},
//   dZ_i/d(tau0, tau1.5) = 2 pi i sum_j (dc_j/dtau) sum_k B_j(k) Q_i e^{...}
// with B_j = phi^-5/3, phi^-1, phi^-2/3, phi^-1/3. A reduction kernel forms the six sums per
// (particle, detector) over segments of the band; a per-particle kernel adds the segments and combines
// the sums in binary64.
#include <cmath>

#include "fcas_kernels.cuh"
#include "fcas_sums.cuh"

namespace fcas {

constexpr int kGradSums = 12;   // Z, F (= sum k Q), S_53, S_1, S_23, S_13: complex, as (re, im) doubles

template <typename Real> struct grad_sum { using type = double; };
template <> struct grad_sum<float> { using type = SumF; };

constexpr int kGradThreads = 256;
constexpr int kGradDet = 2;                        // detectors per CTA: they share a bin's chirp phase
constexpr int kGradVals = kGradDet * kGradSums;    // 24 sums per thread

// Sums of one warp's 24 values: the first three butterfly steps halve the values each lane carries (24 ->
// 12 -> 6 -> 3), the last two add whole lanes: 27 additions where a reduction value by value takes 120.
// Afterwards lane l holds in v[0..2] the totals of values 3 (l >> 2) .. + 2 in the order (l & 16) 12 +
// (l & 8) 6 + (l & 4) 3.
template <typename Acc>
__device__ __forceinline__ void warp_sums(Acc (&v)[kGradVals], int lane) {
#pragma unroll
    for (int step = 0; step < 3; ++step) {
        const int off = 16 >> step, half = kGradVals >> (step + 1);
        const bool up = lane & off;
#pragma unroll
        for (int i = 0; i < kGradVals / 2; ++i) {
            if (i < half) {
                const Acc mine = up ? v[i + half] : v[i], send = up ? v[i] : v[i + half];
                v[i] = sum_of(mine, sum_xor(send, off));
            }
        }
    }
#pragma unroll
    for (int off = 2; off > 0; off >>= 1)
#pragma unroll
        for (int i = 0; i < kGradVals / 8; ++i) v[i] = sum_of(v[i], sum_xor(v[i], off));
}

// Partial band sums of a particle: CTA (particle, detector pair, segment) adds the terms of its segment's
// column blocks (blks of them) at the rows k2 that hold band bins. The segments do not depend on the
// number of particles, so neither do the sums' bits. One CTA per (particle, detector) over the whole band
// left most SMs idle for a few particles and its twelve binary64 sums per bin held the binary64 unit: 8
// particles of the 60-min workload 42.9 -> 1.36 ms a call, and 1.32 -> 1.02 ms with each bin's loads one bin
// ahead; forward and backward of 40 particles on 64 s 799 -> 398 us. Bound now by FP32 issue (248
// instructions per bin and detector; 77 % of cycles issue).
template <typename Real>
__global__ void __launch_bounds__(kGradThreads, 2)
grad_sums_kernel(const cplx<Real>* __restrict__ y, bool y_ff, const Basis<Real>* __restrict__ basis,
                 const ParticleParams* params, const int64_t* __restrict__ tc, int n_det, int log_n,
                 int log_n1, int log_n2, int log_k1b, int k_lo, int k_hi, int nseg, int blks,
                 double* part) {
    using Acc = typename grad_sum<Real>::type;
    chain_wait();
    chain_go();
    __shared__ Acc red[kGradThreads / 32][kGradVals];
    const int pairs = (n_det + kGradDet - 1) / kGradDet;
    const int seg = blockIdx.x % nseg;
    const int i0 = (blockIdx.x / nseg) % pairs * kGradDet;
    const int64_t p = blockIdx.x / nseg / pairs;
    const int nd = n_det - i0 < kGradDet ? n_det - i0 : kGradDet;
    const ParticleParams& pp = params[p];
    const int64_t t = tc[p];
    const int k1b = 1 << log_k1b;
    const int64_t per_blk = (int64_t)1 << (log_n2 - 1 + log_k1b);
    const int k2_lo = k_lo >> log_n1, rows = (k_hi >> log_n1) - k2_lo + 1;
    const unsigned nmask = (1u << log_n) - 1u;
    Acc acc[kGradVals];
#pragma unroll
    for (int q = 0; q < kGradVals; ++q) sum_zero(acc[q]);
    if (pp.valid && t >= 0) {
        const unsigned tu = (unsigned)t;
        for (int blk = seg * blks; blk < (seg + 1) * blks; ++blk) {
            const Basis<Real>* bb = basis + blk * per_blk;
            const cplx<Real>* yb = y + ((int64_t)blk * n_det + i0) * per_blk;
            // FP32: the next bin's basis and spectrum are requested before this bin's arithmetic
            const int count = rows << log_k1b, e0 = k2_lo << log_k1b;
            Basis<Real> bn{};
            cplx<Real> yn[kGradDet] = {};
            auto request = [&](int r) {
                if (r >= count) return;
                bn = bb[e0 + r];
#pragma unroll
                for (int u = 0; u < kGradDet; ++u)
                    if (u < nd) yn[u] = yb[u * per_blk + e0 + r];
            };
            if constexpr (sizeof(Real) == 4) request(threadIdx.x);
            for (int r = threadIdx.x; r < count; r += kGradThreads) {
                const int e = r + e0;
                const int k = blk * k1b + (e & (k1b - 1)) + ((e >> log_k1b) << log_n1);
                Basis<Real> b;
                cplx<Real> yc[kGradDet];
                if constexpr (sizeof(Real) == 4) {
                    b = bn;
#pragma unroll
                    for (int u = 0; u < kGradDet; ++u) yc[u] = yn[u];
                    request(r + kGradThreads);
                }
                if (k < k_lo || k > k_hi) continue;
                if constexpr (sizeof(Real) != 4) b = bb[e];
                const unsigned m = ((unsigned)k * tu) & nmask;   // k t mod N (the low bits of the product)
                if constexpr (sizeof(Real) == 4) {
                    const float shift = (float)m * __int_as_float((127 - log_n) << 23);   // m / N, exact
                    const ChirpPowers cpw = chirp_powers(b);
                    float s = frac_mul_ff(pp.ch[0], pp.cl[0], cpw.b53.x, cpw.b53.y);
                    s += frac_mul_ff(pp.ch[1], pp.cl[1], cpw.b1.x, cpw.b1.y);
                    s += frac_mul_ff(pp.ch[2], pp.cl[2], cpw.b23.x, cpw.b23.y);
                    s += frac_mul_ff(pp.ch[3], pp.cl[3], cpw.b13.x, cpw.b13.y);
                    const float kk = (float)k;   // < 2^24: exact
#pragma unroll
                    for (int u = 0; u < kGradDet; ++u) {
                        if (u >= nd) break;
                        const float2 yv = yc[u];
                        float th = s + frac_mul_ff(kk, 0.0f, pp.dh[i0 + u], pp.dl[i0 + u]) + shift;
                        th -= rintf(th);
                        float sn, cs;
                        sincospif(2.0f * th, &sn, &cs);
                        const float qv[2] = {yv.x * cs - yv.y * sn, yv.x * sn + yv.y * cs};
#pragma unroll
                        for (int x = 0; x < 2; ++x) {
                            sum_add(acc[u * kGradSums + x], qv[x]);
                            sum_add_w(acc[u * kGradSums + 2 + x], kk, qv[x]);
                            sum_add_w(acc[u * kGradSums + 4 + x], cpw.b53, qv[x]);
                            sum_add_w(acc[u * kGradSums + 6 + x], cpw.b1, qv[x]);
                            sum_add_w(acc[u * kGradSums + 8 + x], cpw.b23, qv[x]);
                            sum_add_w(acc[u * kGradSums + 10 + x], cpw.b13, qv[x]);
                        }
                    }
                } else {
                    const double shift = (double)m * __hiloint2double((1023 - log_n) << 20, 0);   // m / N, exact
                    const double s = pp.c[0] * b.a.x + pp.c[1] * b.a.y + pp.c[2] * b.b.x + pp.c[3] * b.b.y;
                    const double kk = (double)k;
#pragma unroll
                    for (int u = 0; u < kGradDet; ++u) {
                        if (u >= nd) break;
                        double2 yv;
                        if (y_ff) {   // float-float layout (FCAS_PREC_FF contexts): hi/lo re, hi/lo im
                            const float4 q = reinterpret_cast<const float4*>(yb)[u * per_blk + e];
                            yv = make_double2((double)q.x + (double)q.y, (double)q.z + (double)q.w);
                        } else {
                            yv = yb[u * per_blk + e];
                        }
                        double th = s - rint(s);
                        const double kd = kk * pp.dturn[i0 + u];
                        th += kd - rint(kd) + shift;
                        th -= rint(th);
                        double sn, cs;
                        sincospi(2.0 * th, &sn, &cs);
                        const double qv[2] = {yv.x * cs - yv.y * sn, yv.x * sn + yv.y * cs};
#pragma unroll
                        for (int x = 0; x < 2; ++x) {
                            sum_add(acc[u * kGradSums + x], qv[x]);
                            sum_add_w(acc[u * kGradSums + 2 + x], kk, qv[x]);
                            sum_add_w(acc[u * kGradSums + 4 + x], b.a.x, qv[x]);
                            sum_add_w(acc[u * kGradSums + 6 + x], b.a.y, qv[x]);
                            sum_add_w(acc[u * kGradSums + 8 + x], b.b.x, qv[x]);
                            sum_add_w(acc[u * kGradSums + 10 + x], b.b.y, qv[x]);
                        }
                    }
                }
            }
        }
    }
#pragma unroll
    for (int q = 0; q < kGradVals; ++q) sum_normalise(acc[q]);
    const int lane = threadIdx.x & 31;
    warp_sums(acc, lane);
    if ((lane & 3) == 0) {
        const int v0 = (lane & 16 ? 12 : 0) + (lane & 8 ? 6 : 0) + (lane & 4 ? 3 : 0);
#pragma unroll
        for (int i = 0; i < 3; ++i) red[threadIdx.x >> 5][v0 + i] = acc[i];
    }
    __syncthreads();
    if (threadIdx.x < nd * kGradSums) {
        Acc v = red[0][threadIdx.x];
#pragma unroll
        for (int w = 1; w < kGradThreads / 32; ++w) v = sum_of(v, red[w][threadIdx.x]);
        const int u = threadIdx.x / kGradSums, q = threadIdx.x % kGradSums;
        part[((p * n_det + i0 + u) * nseg + seg) * kGradSums + q] = sum_value(v);
    }
}

// d c_j (turns) along (dt0, dt15) for the coefficients of the geometry kernel, by logarithmic derivatives:
// x ~ tau1.5 / tau0, eta ~ x^-2/3 / tau1.5, tau1 ~ P1(eta) / (eta x), tau2 ~ P2(eta) / (eta x^1/3) (one cube
// root where differentiating the powers term by term took four general powers: the kernel 28 -> 17 us).
__device__ void chirp_coeff_derivatives(double tau0, double tau15, double dt0, double dt15, double f_star, double dc[4]) {
    const double pi = 3.14159265358979323846;
    const double x = 5.0 * tau15 / (32.0 * pi * tau0);
    const double cx = cbrt(x);
    const double eta = 1.0 / (cx * cx * 8.0 * f_star * tau15);
    const double dl15 = dt15 / tau15;
    const double dlx = dl15 - dt0 / tau0;             // d ln x
    const double dle = -2.0 / 3.0 * dlx - dl15;       // d ln eta
    const double p1 = 743.0 / 336.0 + 11.0 / 4.0 * eta;
    const double p2 = 3058673.0 / 1016064.0 + (5429.0 / 1008.0 + 617.0 / 144.0 * eta) * eta;
    const double t1 = 5.0 / (192.0 * pi * f_star * eta * x), t2 = 5.0 / (128.0 * pi * f_star * eta * cx);
    dc[0] = 0.6 * f_star * dt0;
    dc[1] = f_star * t1 * (11.0 / 4.0 * eta * dle - p1 * (dle + dlx));
    dc[2] = -1.5 * f_star * dt15;
    dc[3] = 3.0 * f_star * t2 * ((5429.0 / 1008.0 + 617.0 / 72.0 * eta) * eta * dle - p2 * (dle + 1.0 / 3.0 * dlx));
}

// One CTA per particle: the segments' partial sums are added in order by all threads, the sky geometry
// (one lane per detector) and the chirp coefficients (one lane per chirp time) by two different warps,
// and four lanes combine them, one per component (one thread per particle did all of it serially in
// binary64, whose every dependent instruction waits tens of cycles).
constexpr int kFinalThreads = 128;
__global__ void __launch_bounds__(kFinalThreads)
grad_final_kernel(const double* __restrict__ theta, const int64_t* __restrict__ tc, const double* part,
                  int nseg, const double* __restrict__ det9, const double* __restrict__ s2, int n_det, double f_star,
                  double df, double* __restrict__ grad) {
    __shared__ double sp[FCAS_MAX_DET * kGradSums];   // Z_i, F_i, S_ij
    __shared__ double spart[kFinalThreads];
    __shared__ double u[FCAS_MAX_DET][3][2];          // U^i and its alpha / delta derivatives
    __shared__ double dd[FCAS_MAX_DET][3];            // delay in turns per bin and its derivatives
    __shared__ double dc[2][4];                       // d c_j / d tau0, d c_j / d tau1.5
    const int64_t p = blockIdx.x;
    const int tid = threadIdx.x;
    chain_wait();
    chain_go();
    const double nan = __longlong_as_double(0x7ff8000000000000LL);
    const double alpha = theta[4 * p], delta = theta[4 * p + 1], tau0 = theta[4 * p + 2], tau15 = theta[4 * p + 3];
    if (!(isfinite(alpha) && isfinite(delta) && tau0 > 0.0 && tau15 > 0.0 && tc[p] >= 0)) {
        if (tid < 4) grad[4 * p + tid] = nan;
        return;
    }
    // value v of the detectors' 12 n_det sums: groups of threads add every groups-th segment, then the
    // groups' totals in order
    const int vals = n_det * kGradSums, groups = kFinalThreads / vals;
    const int v = tid % vals, gr = tid / vals;
    double acc = 0.0;
    if (gr < groups)
        for (int seg = gr; seg < nseg; seg += groups)
            acc += part[((p * n_det + v / kGradSums) * nseg + seg) * kGradSums + v % kGradSums];
    spart[tid] = acc;
    if (tid >= 32 && tid < 34) {
        chirp_coeff_derivatives(tau0, tau15, tid == 32 ? 1.0 : 0.0, tid == 33 ? 1.0 : 0.0, f_star, dc[tid - 32]);
    }
    if (tid < 32) {
        // lane 0 takes sin and cos of alpha, lane 1 of delta
        double sn, cs;
        sincos(tid & 1 ? delta : alpha, &sn, &cs);
        const double sa = __shfl_sync(0xffffffffu, sn, 0), ca = __shfl_sync(0xffffffffu, cs, 0);
        const double sd = __shfl_sync(0xffffffffu, sn, 1), cd = __shfl_sync(0xffffffffu, cs, 1);
        if (tid < n_det) {
            // basis vectors and their derivatives: [0] value, [1] d/d alpha, [2] d/d delta
            const double nv[3][3] = {{cd * ca, cd * sa, sd}, {-cd * sa, cd * ca, 0.0}, {-sd * ca, -sd * sa, cd}};
            const double bx[3][3] = {{sa, -ca, 0.0}, {ca, sa, 0.0}, {0.0, 0.0, 0.0}};
            const double by[3][3] = {{-sd * ca, -sd * sa, cd}, {sd * sa, -sd * ca, 0.0}, {-cd * ca, -cd * sa, -sd}};
            const double* dv = det9 + 9 * tid;
            auto dot = [](const double* a, const double* b) { return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]; };
            const double xX = dot(dv + 3, bx[0]), xY = dot(dv + 3, by[0]), yX = dot(dv + 6, bx[0]),
                         yY = dot(dv + 6, by[0]);
            u[tid][0][0] = 0.5 * (xX * xX - xY * xY - yX * yX + yY * yY);
            u[tid][0][1] = xX * xY - yX * yY;
            for (int m = 1; m < 3; ++m) {
                const double dxX = dot(dv + 3, bx[m]), dxY = dot(dv + 3, by[m]), dyX = dot(dv + 6, bx[m]),
                             dyY = dot(dv + 6, by[m]);
                u[tid][m][0] = xX * dxX - xY * dxY - yX * dyX + yY * dyY;
                u[tid][m][1] = dxX * xY + xX * dxY - dyX * yY - yX * dyY;
            }
            for (int m = 0; m < 3; ++m) dd[tid][m] = -dot(dv, nv[m]) / kCLight * df;
        }
    }
    __syncthreads();
    if (tid < vals) {
        double total = spart[tid];
        for (int g = 1; g < groups; ++g) total += spart[g * vals + tid];
        sp[tid] = total;
    }
    __syncthreads();
    if (tid >= 4) return;
    const int m = tid;   // the component
    const double two_pi = 6.283185307179586476925286766559;
    double G[3] = {}, dG[3] = {};   // G entries (11, 12, 22) and their derivative for m = 0, 1
    const int md = m < 2 ? m + 1 : 0;
    for (int i = 0; i < n_det; ++i) {
        G[0] += s2[i] * u[i][0][0] * u[i][0][0];
        G[1] += s2[i] * u[i][0][0] * u[i][0][1];
        G[2] += s2[i] * u[i][0][1] * u[i][0][1];
        dG[0] += s2[i] * 2.0 * u[i][md][0] * u[i][0][0];
        dG[1] += s2[i] * (u[i][md][0] * u[i][0][1] + u[i][0][0] * u[i][md][1]);
        dG[2] += s2[i] * 2.0 * u[i][md][1] * u[i][0][1];
    }
    const double det = G[0] * G[2] - G[1] * G[1];
    const double tr = G[0] + G[2];
    if (det < kRank1Rtol * (0.5 * tr) * (0.5 * tr)) {   // rank-1 branch: no gradient (NaN)
        grad[4 * p + m] = nan;
        return;
    }
    const double gi[3] = {G[2] / det, -G[1] / det, G[0] / det};
    double Wr[2] = {0, 0}, Wi[2] = {0, 0};
    for (int i = 0; i < n_det; ++i)
        for (int a = 0; a < 2; ++a) {
            Wr[a] += u[i][0][a] * sp[12 * i + 0];
            Wi[a] += u[i][0][a] * sp[12 * i + 1];
        }
    auto quad_re = [&](const double* ar, const double* ai, const double* br, const double* bi, const double* g) {
        // Re(a^H Ginv b) with Ginv = [[g0, g1], [g1, g2]]
        const double r0 = g[0] * br[0] + g[1] * br[1], r1 = g[1] * br[0] + g[2] * br[1];
        const double i0 = g[0] * bi[0] + g[1] * bi[1], i1 = g[1] * bi[0] + g[2] * bi[1];
        return ar[0] * r0 + ar[1] * r1 + ai[0] * i0 + ai[1] * i1;
    };
    double dWr[2] = {0, 0}, dWi[2] = {0, 0};
    for (int i = 0; i < n_det; ++i) {
        const double* s = sp + 12 * i;
        // dZ_i = 2 pi i * X_i, X_i = (dd_i) F_i or sum_j dc_j S_ij
        double xr, xi;
        if (m < 2) {
            xr = dd[i][m + 1] * s[2];
            xi = dd[i][m + 1] * s[3];
        } else {
            const double* c = dc[m - 2];
            xr = c[0] * s[4] + c[1] * s[6] + c[2] * s[8] + c[3] * s[10];
            xi = c[0] * s[5] + c[1] * s[7] + c[2] * s[9] + c[3] * s[11];
        }
        const double dzr = -two_pi * xi, dzi = two_pi * xr;
        for (int a = 0; a < 2; ++a) {
            dWr[a] += u[i][0][a] * dzr;
            dWi[a] += u[i][0][a] * dzi;
            if (m < 2) {
                dWr[a] += u[i][m + 1][a] * s[0];
                dWi[a] += u[i][m + 1][a] * s[1];
            }
        }
    }
    double gsum = 2.0 * quad_re(dWr, dWi, Wr, Wi, gi);
    if (m < 2) {
        // - W^H Ginv dG Ginv W: Ginv W first, then the dG quadratic form
        const double ar[2] = {gi[0] * Wr[0] + gi[1] * Wr[1], gi[1] * Wr[0] + gi[2] * Wr[1]};
        const double ai[2] = {gi[0] * Wi[0] + gi[1] * Wi[1], gi[1] * Wi[0] + gi[2] * Wi[1]};
        gsum -= quad_re(ar, ai, ar, ai, dG);
    }
    grad[4 * p + m] = gsum;
}

// Segments of the band sums: ~2048 bins per CTA, at most 256 segments and one column block per segment
// (a power of two, as the number of column blocks is).
static int most_segments(int log_n) { return log_n > 12 ? imin_c(256, 1 << (log_n - 12)) : 1; }
static int grad_segments(const FitnessPlan& pl) {
    return imax_c(1, imin_c((1 << pl.log_n1) / pl.k1b, most_segments(pl.log_n)));
}

// (particle, segment) pairs of one launch, which bound the partial sums (12.6 MB with four detectors)
constexpr int64_t kGradPairs = 32768;

int64_t grad_launch_segments(int log_n, int64_t n) {
    const int64_t m = most_segments(log_n);
    return n < kGradPairs / m ? n * m : kGradPairs;
}

cudaError_t launch_gradient(const FitnessPlan& pl, int precision, int64_t k_lo, int64_t k_hi,
                            const ParticleParams* params, const double* theta, const int64_t* tc, int64_t n,
                            double* part, const double* det9, const double* s2, double f_star, double df, double* grad,
                            cudaStream_t s) {
    const int nseg = grad_segments(pl), pairs = (pl.n_det + kGradDet - 1) / kGradDet;
    const int blks = (1 << pl.log_n1) / pl.k1b / nseg;
    int log_k1b = 0;
    while ((1 << log_k1b) < pl.k1b) ++log_k1b;
    const int64_t chunk = kGradPairs / nseg;
    for (int64_t p0 = 0; p0 < n; p0 += chunk) {
        const int64_t np = n - p0 < chunk ? n - p0 : chunk;
        const unsigned ctas = (unsigned)(np * pairs * nseg);
        cudaError_t e;
        if (precision == FCAS_PREC_FP32)
            e = launch_chained(true, grad_sums_kernel<float>, dim3(ctas), dim3(kGradThreads), 0, s,
                               static_cast<const float2*>(pl.y), false, static_cast<const BasisF*>(pl.basis),
                               params + p0, tc + p0, pl.n_det, pl.log_n, pl.log_n1, pl.log_n2, log_k1b, (int)k_lo,
                               (int)k_hi, nseg, blks, part);
        else
            e = launch_chained(true, grad_sums_kernel<double>, dim3(ctas), dim3(kGradThreads), 0, s,
                               static_cast<const double2*>(pl.y), precision == FCAS_PREC_FF,
                               static_cast<const BasisD*>(pl.basis), params + p0, tc + p0, pl.n_det, pl.log_n,
                               pl.log_n1, pl.log_n2, log_k1b, (int)k_lo, (int)k_hi, nseg, blks, part);
        if (e == cudaSuccess)
            e = launch_chained(true, grad_final_kernel, dim3((unsigned)np), dim3(kFinalThreads), 0, s, theta + 4 * p0,
                               tc + p0, part, nseg, det9, s2, pl.n_det, f_star, df, grad + 4 * p0);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// ------------------------------------------------------------------------------------------
// Gradient polishing: ascent steps along the adjoint gradient, each halved until the fitness
// increases (the differentiation form's use of the adjoint; the paper itself only runs the swarm).
// Per particle, with s = scales (1, 1, tau0, tau1.5) (absolute for the angles, relative for the
// chirp times): direction d = s^2 g / |s g| (a step of length |s| in the metric of s, uphill),
// first trial step length 1, halved after every trial that does not raise the fitness.
// ------------------------------------------------------------------------------------------
__global__ void polish_direction_kernel(const double* __restrict__ theta, const double* __restrict__ grad,
                                        PolishScales sc, int64_t n, double* __restrict__ dir,
                                        double* __restrict__ step, int32_t* __restrict__ done) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    double sg[4], norm2 = 0.0;
    bool finite = true;
    for (int m = 0; m < 4; ++m) {
        const double s = sc.s[m] * (m < 2 ? 1.0 : theta[4 * p + m]);
        const double g = grad[4 * p + m];
        finite = finite && isfinite(g) && isfinite(s);
        sg[m] = s * g;
        dir[4 * p + m] = s * s * g;
        norm2 += sg[m] * sg[m];
    }
    const double norm = sqrt(norm2);
    const bool ok = finite && norm > 0.0;
    for (int m = 0; m < 4; ++m) dir[4 * p + m] = ok ? dir[4 * p + m] / norm : 0.0;
    step[p] = 1.0;
    done[p] = ok ? 0 : 1;
}

// the trial point of every particle still searching; NaN (not evaluated) for the others
__global__ void polish_candidate_kernel(const double* __restrict__ theta, const double* __restrict__ dir,
                                        const double* __restrict__ step, const int32_t* __restrict__ done, int64_t n,
                                        double* __restrict__ cand) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    for (int m = 0; m < 4; ++m)
        cand[4 * p + m] = done[p] ? __longlong_as_double(0x7ff8000000000000LL)
                                  : theta[4 * p + m] + step[p] * dir[4 * p + m];
}

// accept a trial that raises the fitness (a NaN trial never does); otherwise halve the step and count
// the particle as still searching
__global__ void polish_accept_kernel(double* __restrict__ theta, double* __restrict__ fit, int64_t* __restrict__ tc,
                                     const double* __restrict__ cand, const double* __restrict__ cfit,
                                     const int64_t* __restrict__ ctc, double* __restrict__ step,
                                     int32_t* __restrict__ done, int32_t* __restrict__ accepted, int64_t n,
                                     int32_t* __restrict__ searching) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n || done[p]) return;
    if (cfit[p] > fit[p]) {
        for (int m = 0; m < 4; ++m) theta[4 * p + m] = cand[4 * p + m];
        fit[p] = cfit[p];
        tc[p] = ctc[p];
        accepted[p] += 1;
        done[p] = 1;
    } else {
        step[p] *= 0.5;
        atomicAdd(searching, 1);
    }
}

cudaError_t launch_polish_direction(const double* theta, const double* grad, const PolishScales& sc, int64_t n,
                                    double* dir, double* step, int32_t* done, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    polish_direction_kernel<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(theta, grad, sc, n, dir, step, done);
    return cudaGetLastError();
}

cudaError_t launch_polish_candidate(const double* theta, const double* dir, const double* step, const int32_t* done,
                                    int64_t n, double* cand, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    polish_candidate_kernel<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(theta, dir, step, done, n, cand);
    return cudaGetLastError();
}

cudaError_t launch_polish_accept(double* theta, double* fit, int64_t* tc, const double* cand, const double* cfit,
                                 const int64_t* ctc, double* step, int32_t* done, int32_t* accepted, int64_t n,
                                 int32_t* searching, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    polish_accept_kernel<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(theta, fit, tc, cand, cfit, ctc, step, done,
                                                                     accepted, n, searching);
    return cudaGetLastError();
}

}  // namespace fcas
