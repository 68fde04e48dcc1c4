// Fitness path, per-particle and host-side parts: geometry, the final argmax, the shape helpers
// of the two passes, the per-stage twiddle tables, and the FP32 / binary64 instantiations of the
// passes (fcas_passes.cuh).
#include <cmath>

#include "fcas_passes.cuh"

namespace fcas {

// ------------------------------------------------------------------------------------------
// Geometry: Sec. II eq. detresponse (U = F(alpha, delta, 0), Delta^i), Sec. II.C/II.D
// (G = sum_i sigma_i^2 U^i U^i^T) and Sec. II.B (chirp times -> phase coefficients).
// ------------------------------------------------------------------------------------------
// Two warps per four particles, eight lanes of each per particle. The first warp takes the sky (one lane per
// detector), the second the chirp coefficients, so that their binary64 chains run beside each other: the
// kernel is bound by the latency of dependent binary64 instructions (a few particles) or by their number
// per SM (a large batch), and one thread per particle issued every detector's share serially (one
// particle on 64 s, host arrays: 89.5 -> 65.1 us a call; 40 particles 85.9 -> 62.6; the same results).
struct TaylorBound {
    double m[2][4];   // cm^3/6 |psi'''| <= sum_j |c_j| m[bit][j]; infinite where no anchor is allowed
};

// Remainder of psi(k + c) = psi(k) + c psi' + c^2 psi''/2 for c <= C (FP32 pass A, C + 1 adjacent columns
// per lane group, C = 3 or 7): at most C^3/6 max |psi'''| over the band, taken at k_b = f_*/df - 2 (C + 1)
// (the band's lowest bin, less the C by which an anchor bin may lie below it, with margin), where
// |psi'''| <= sum_m |c_m| e_m (e_m + 1) (e_m + 2) phi^-e_m / k^3.
static TaylorBound taylor_bound(double f_star, double df) {
    TaylorBound t;
    for (int bit = 0; bit < 2; ++bit) {
        const double cm = bit == 0 ? 3.0 : 7.0;
        const double kb = f_star / df - 2.0 * (cm + 1.0);
        if (kb < 1.0) {
            for (double& v : t.m[bit]) v = HUGE_VAL;
            continue;
        }
        const double r = f_star / (kb * df);   // phi^-1 at k_b
        const double r13 = std::cbrt(r);
        const double w = cm * cm * cm / 6.0 / (kb * kb * kb);
        t.m[bit][0] = w * (440.0 / 27.0) * r * r13 * r13;
        t.m[bit][1] = w * 6.0 * r;
        t.m[bit][2] = w * (80.0 / 27.0) * r13 * r13;
        t.m[bit][3] = w * (28.0 / 27.0) * r13;
    }
    return t;
}

constexpr int kGeomLanes = FCAS_MAX_DET;            // lanes per particle
constexpr int kGeomParticles = 32 / kGeomLanes;     // particles per warp

__global__ void __launch_bounds__(64)
geometry_kernel(const double* __restrict__ theta, int64_t n, ParticleParams* __restrict__ out,
                const double* __restrict__ det9, const double* __restrict__ s2, int n_det, double f_star, double df,
                int64_t kstep, bool wide, TaylorBound tb) {
    chain_go();
    const int lane = threadIdx.x & 31, sub = lane % kGeomLanes, lane0 = lane - sub;
    const int64_t p = (int64_t)blockIdx.x * kGeomParticles + lane / kGeomLanes;
    const bool have = p < n;
    const int64_t pc = have ? p : n - 1;   // lanes beyond the batch repeat its last particle, unwritten
    const double alpha = theta[4 * pc + 0], delta = theta[4 * pc + 1];
    const double tau0 = theta[4 * pc + 2], tau15 = theta[4 * pc + 3];
    const bool ok = isfinite(alpha) && isfinite(delta) && isfinite(tau0) && isfinite(tau15) && tau0 > 0.0 &&
                    tau15 > 0.0;
    ParticleParams* pp = out + pc;
    if (threadIdx.x >= 32) {
        // (tau0, tau1.5) -> x = pi M f_*, eta; then the 2PN chirp times: tau1 by even lanes, tau2 by odd ones
        const double pi = 0.5 * kTwoPi;
        const double x = 5.0 * tau15 / (32.0 * pi * tau0);
        const double cx = cbrt(x);
        const double eta = 1.0 / (cx * cx) / (8.0 * f_star * tau15);
        const bool odd = sub & 1;
        const double scale = 5.0 / ((odd ? 128.0 * pi : 192.0 * pi) * f_star * eta * (odd ? cx : x));
        const double tau = scale * (odd ? 3058673.0 / 1016064.0 + 5429.0 * eta / 1008.0 + 617.0 * eta * eta / 144.0
                                        : 743.0 / 336.0 + 11.0 * eta / 4.0);
        const double tau1 = __shfl_sync(0xffffffffu, tau, lane0), tau2 = __shfl_sync(0xffffffffu, tau, lane0 + 1);
        const double c[4] = {0.6 * f_star * tau0, f_star * tau1, -1.5 * f_star * tau15, 3.0 * f_star * tau2};
        int taylor = 0;
#pragma unroll
        for (int bit = 0; bit < 2; ++bit) {
            double rem = 0.0;
#pragma unroll
            for (int r = 0; r < 4; ++r) rem += fabs(c[r]) * tb.m[bit][r];
            if (rem < 1e-7) taylor |= 1 << bit;   // false for the infinite bound and for a NaN
        }
        if (!have) return;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            if (sub != r) continue;
            const double v = ok ? c[r] : 0.0;
            pp->c[r] = v;
            pp->ch[r] = (float)v;
            pp->cl[r] = (float)(v - (double)(float)v);
        }
        if (sub == 4) {
            pp->valid = ok;
            pp->taylor_ok = ok ? taylor : 0;
        }
        return;
    }
    // sky: sin and cos of alpha by even lanes, of delta by odd ones
    double sn, cs;
    sincos(sub & 1 ? delta : alpha, &sn, &cs);
    const double sa = __shfl_sync(0xffffffffu, sn, lane0), ca = __shfl_sync(0xffffffffu, cs, lane0);
    const double sd = __shfl_sync(0xffffffffu, sn, lane0 + 1), cd = __shfl_sync(0xffffffffu, cs, lane0 + 1);
    const double nx = cd * ca, ny = cd * sa, nz = sd;
    const double bx[3] = {sa, -ca, 0.0};             // -alpha_hat
    const double by[3] = {-sd * ca, -sd * sa, cd};   // delta_hat
    double dturn = 0.0, fp = 0.0, fx = 0.0, sfp = 0.0, sfx = 0.0;
    if (sub < n_det) {
        const double* d = det9 + 9 * sub;
        dturn = -(d[0] * nx + d[1] * ny + d[2] * nz) / kCLight * df;
        const double xX = d[3] * bx[0] + d[4] * bx[1] + d[5] * bx[2];
        const double xY = d[3] * by[0] + d[4] * by[1] + d[5] * by[2];
        const double yX = d[6] * bx[0] + d[7] * bx[1] + d[8] * bx[2];
        const double yY = d[6] * by[0] + d[7] * by[1] + d[8] * by[2];
        fp = 0.5 * (xX * xX - xY * xY - yX * yX + yY * yY);
        fx = xX * xY - yX * yY;
        sfp = s2[sub] * fp;
        sfx = s2[sub] * fx;
    }
    double g11 = 0.0, g12 = 0.0, g22 = 0.0;
    for (int i = 0; i < n_det; ++i) {
        const double fpi = __shfl_sync(0xffffffffu, fp, lane0 + i), fxi = __shfl_sync(0xffffffffu, fx, lane0 + i);
        const double spi = __shfl_sync(0xffffffffu, sfp, lane0 + i), sxi = __shfl_sync(0xffffffffu, sfx, lane0 + i);
        g11 += spi * fpi;
        g12 += spi * fxi;
        g22 += sxi * fxi;
    }
    const double det = g11 * g22 - g12 * g12;
    const double tr = g11 + g22;
    // G^-1: lane 0 divides for its first entry, lane 1 for its second, the others for its third
    const double quot = (sub == 0 ? g22 : sub == 1 ? -g12 : g11) / det;
    double ginv[3] = {__shfl_sync(0xffffffffu, quot, lane0), __shfl_sync(0xffffffffu, quot, lane0 + 1),
                      __shfl_sync(0xffffffffu, quot, lane0 + 2)};
    if (det < kRank1Rtol * (0.5 * tr) * (0.5 * tr)) {
        const double lam = 0.5 * tr + sqrt(0.25 * (g11 - g22) * (g11 - g22) + g12 * g12);
        double e1 = lam - g22, e2 = g12;
        double f1 = g12, f2 = lam - g11;
        if (f1 * f1 + f2 * f2 > e1 * e1 + e2 * e2) { e1 = f1; e2 = f2; }
        const double nrm = e1 * e1 + e2 * e2;
        ginv[0] = ginv[1] = ginv[2] = 0.0;
        if (lam > 0.0 && nrm > 0.0) {
            ginv[0] = e1 * e1 / nrm / lam;
            ginv[1] = e1 * e2 / nrm / lam;
            ginv[2] = e2 * e2 / nrm / lam;
        }
    }
    // Cholesky factor of G^-1 so that Gamma^2 = |l11 W+ + l21 Wx|^2 + |l22 Wx|^2 is a sum of
    // squares (no cancellation when F is ill-conditioned)
    double chol[3] = {0.0, 0.0, 0.0};
    if (ginv[0] > 0.0) {
        const double l11 = sqrt(ginv[0]);
        const double l21 = ginv[1] / l11;
        chol[0] = l11;
        chol[1] = l21;
        chol[2] = sqrt(fmax(0.0, ginv[2] - l21 * l21));
    } else {
        chol[2] = sqrt(fmax(0.0, ginv[2]));
    }
    const bool det_lane = ok && sub < n_det;
    const double w1 = det_lane ? chol[0] * fp + chol[1] * fx : 0.0;
    const double w2 = det_lane ? chol[2] * fx : 0.0;
    if (!det_lane) dturn = fp = fx = 0.0;
    double us = (double)kstep * dturn;   // |us| < 2^24 turns, exact to ~1e-9
    us -= rint(us);
    double su, cu;
    sincospi(2.0 * us, &su, &cu);
    if (wide) {
        const double d0 = __shfl_sync(0xffffffffu, dturn, lane0);
        const double rel = det_lane ? dturn - d0 : 0.0;
        double ur = (double)kstep * rel;
        ur -= rint(ur);
        double ur4 = 4.0 * ur;   // (exact, as kstep rel is: powers of two)
        ur4 -= rint(ur4);
        double sr, cr, s4, c4;
        sincospi(2.0 * ur, &sr, &cr);
        sincospi(2.0 * ur4, &s4, &c4);
        if (have) {
            pp->rturn[sub] = rel;
            pp->rstep[sub] = make_double2(cr, sr);
            pp->rstep4[sub] = make_double2(c4, s4);
        }
    }
    if (!have) return;
    pp->dturn[sub] = dturn;
    pp->u[sub][0] = fp;
    pp->u[sub][1] = fx;
    pp->w1[sub] = w1;
    pp->w2[sub] = w2;
    pp->dh[sub] = (float)dturn;
    pp->dl[sub] = (float)(dturn - (double)(float)dturn);
    pp->w1f[sub] = (float)w1;
    pp->w2f[sub] = (float)w2;
    pp->dstep[sub] = make_float2((float)cu, (float)su);
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        if (sub != r) continue;
        pp->ginv[r] = ok ? ginv[r] : 0.0;
        pp->chol[r] = ok ? chol[r] : 0.0;
    }
}

cudaError_t launch_geometry(const double* theta, int64_t n, ParticleParams* out, const double* det9,
                            const double* sigma2_scaled, int n_det, double f_star, double df, int64_t kstep,
                            int precision, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const int64_t blocks = (n + kGeomParticles - 1) / kGeomParticles;
    geometry_kernel<<<(unsigned)blocks, 64, 0, s>>>(theta, n, out, det9, sigma2_scaled, n_det, f_star, df, kstep,
                                                    precision != FCAS_PREC_FP32, taylor_bound(f_star, df));
    return cudaGetLastError();
}

__device__ __forceinline__ bool better(double v, int64_t t, double bv, int64_t bt) {
    return v > bv || (v == bv && t < bt);
}


__global__ void reduce_kernel(const Partial* partials, int64_t nb, const ParticleParams* params,
                              int64_t p0, double* __restrict__ fitness, int64_t* __restrict__ tc) {
    __shared__ double sv[32];
    __shared__ int64_t st[32];
    const int64_t p = blockIdx.x;
    chain_wait();
    chain_go();
    double best = -DBL_MAX;
    int64_t bt = INT64_MAX;
    for (int64_t b = threadIdx.x; b < nb; b += blockDim.x) {
        const Partial q = partials[p * nb + b];
        if (better(q.val, q.t, best, bt)) { best = q.val; bt = q.t; }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const double ov = __shfl_down_sync(0xffffffffu, best, off);
        const int64_t ot = __shfl_down_sync(0xffffffffu, bt, off);
        if (better(ov, ot, best, bt)) { best = ov; bt = ot; }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) { sv[warp] = best; st[warp] = bt; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x + 31) / 32; ++w)
            if (better(sv[w], st[w], best, bt)) { best = sv[w]; bt = st[w]; }
        const bool ok = params[p0 + p].valid != 0;
        fitness[p0 + p] = ok ? best : __longlong_as_double(0x7ff8000000000000LL);
        tc[p0 + p] = ok ? bt : -1;
    }
}

cudaError_t launch_reduce(const Partial* partials, int64_t nb, const ParticleParams* params, int64_t p0, int64_t np,
                          double* fitness, int64_t* tc, bool chained, cudaStream_t s) {
    if (np <= 0) return cudaSuccess;
    return launch_chained(chained, reduce_kernel, dim3((unsigned)np), dim3(256), 0, s, partials, nb, params, p0, fitness,
                          tc);
}

// ------------------------------------------------------------------------------------------
// shape helpers of the passes
// ------------------------------------------------------------------------------------------
int pass_b_blocks_per_particle(int log_n1, int log_n2, int precision) {
    if (log_n1 < 2 || log_n1 > kMaxLogPass) return -1;
    return (1 << log_n2) / pass_b_tb(log_n1, precision);
}

bool pass_a_radix8_available(int log_n2, int precision, int k1b) {
    if (precision == FCAS_PREC_FP32) return log_n2 >= 10 && ((log_n2 <= 11 && k1b == 4) || (log_n2 <= 12 && k1b == 2));
    return log_n2 >= 10 && log_n2 <= 12 && precision == FCAS_PREC_FF && k1b == 2;
}

int pass_a_default_radix_bits(int log_n2, int precision) {
    // float-float: radix 8 halves the registers per thread (16 resident warps per SM instead of 8)
    return precision == FCAS_PREC_FF && log_n2 == 11 ? 3 : 4;
}

int pass_a_k1b_variants(int log_n2, int precision, int* out) {
    if (log_n2 < 2 || log_n2 > kMaxLogPass) return 0;
    const int kd = pass_a_k1b(log_n2, precision);
    int n = 0;
    out[n++] = kd;
    if (log_n2 >= 8 && precision == FCAS_PREC_FP32) {
        if (x2_k1b_ok(log_n2, kd / 2)) out[n++] = kd / 2;
        if (x2_k1b_ok(log_n2, kd * 2)) out[n++] = kd * 2;
        if (x2_k1b_ok(log_n2, kd * 4)) out[n++] = kd * 4;
        if (log_n2 >= 10 && kd / 2 > 1) out[n++] = 1;
    }
    if (precision == FCAS_PREC_FP64 && fp64_k1b_double(log_n2)) out[n++] = kd * 2;
    return n;
}

template cudaError_t launch_pass_a<float>(const FitnessPlan&, const ParticleParams*, int64_t, int64_t, void*, cudaStream_t, int64_t*);
template cudaError_t launch_pass_a<double>(const FitnessPlan&, const ParticleParams*, int64_t, int64_t, void*, cudaStream_t, int64_t*);
template cudaError_t launch_pass_b<float>(const FitnessPlan&, const ParticleParams*, int64_t, int64_t, const void*,
                                          Partial*, cudaStream_t, int64_t*);
template cudaError_t launch_pass_b<double>(const FitnessPlan&, const ParticleParams*, int64_t, int64_t, const void*,
                                           Partial*, cudaStream_t, int64_t*);

// ------------------------------------------------------------------------------------------
// per-stage twiddle tables of the radix-16 transforms (create time)
// ------------------------------------------------------------------------------------------
// entry order: fft_tw_pos of transforms whose exchanges are local from bit cb on
// lf: (c, t) entries of the binary64 form's fused butterflies
__global__ void stage_table_kernel(int log_l, int maxrb, int cb, bool lf, double2* t64, float2* t32) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    const int l = 1 << log_l;
    if (m >= l) return;
    double2 val = make_double2(1.0, 0.0);
    // find the stage that owns entry m: (Ns - 1) <= m < Ns R - 1
    for (int done = 0; done < log_l; done += fftr_radix_bits(log_l, done, maxrb)) {
        const int ns = 1 << done;
        const int r_ = 1 << fftr_radix_bits(log_l, done, maxrb);
        if (ns > 1 && m >= ns - 1 && m < ns * r_ - 1) {
            const int off = m - (ns - 1);
            if (lf) {
                const int e = off / ns;
                if (e >= r_ / 2) continue;
                double sn, cs;
                sincospi(2.0 * (double)fft_lf_entry(e, off % ns, ns, r_) / (double)(ns * r_), &sn, &cs);
                if (cs == 0.0) cs = 8.673617379884035e-19;   // 2^-60
                val = make_double2(cs, sn / cs);
                continue;
            }
            const int r = off / ns + 1;
            // the inverse of fft_tw_pos on 0..ns-1
            const int pos = off % ns;
            const int b = ns < (1 << fft_log_g(log_l, maxrb)) ? ns : 1 << fft_log_g(log_l, maxrb), lo = pos & (b - 1);
            const int jm = cb == 0 || ns < (1 << cb) ? pos : pos - lo + lo / (b >> cb) + ((lo & ((b >> cb) - 1)) << cb);
            double sn, cs;
            // e^{2 pi i r jm / (Ns R)}, argument reduced exactly before sincospi
            const long long num = ((long long)r * jm) % ((long long)ns * r_);
            sincospi(2.0 * (double)num / (double)(ns * r_), &sn, &cs);
            val = make_double2(cs, sn);
        }
    }
    t64[m] = val;
    t32[m] = make_float2((float)val.x, (float)val.y);
}

unsigned int take_index_checks(cudaStream_t s) {
#ifdef FCAS_CHECKED
    unsigned int h = 0, zero = 0;
    if (cudaStreamSynchronize(s) != cudaSuccess) return 0;
    cudaMemcpyFromSymbol(&h, g_index_checks, sizeof(h));
    cudaMemcpyToSymbol(g_index_checks, &zero, sizeof(zero));
    return h;
#else
    (void)s;
    return 0;
#endif
}

cudaError_t launch_stage_tables(int log_l, int maxrb, int k, bool lf, double2* t64, float2* t32, cudaStream_t s) {
    const int l = 1 << log_l;
    stage_table_kernel<<<(l + 255) / 256, 256, 0, s>>>(log_l, maxrb, fft_local_bits(log_l, maxrb, k), lf, t64, t32);
    return cudaGetLastError();
}

}  // namespace fcas
