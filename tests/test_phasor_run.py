"""Accuracy of the accurate forms' phasor runs (CPU, the kernels' own source compiled for the host): against
the exact phasors, a run loses no more than products in a row by its step do, for steps from tiny to a full
turn, in binary64 and in float-float."""

import ctypes

import numpy as np
import pytest

from host_code import compile_host

SOURCE = r"""
#include "fcas_fft16.cuh"
#include "fcas_phasor.cuh"
using namespace fcas;
template <typename R> struct io;
template <> struct io<double> {
    static double2 get(const double* p) { return make_double2(p[0], p[1]); }
    static void put(double* p, double2 v) { p[0] = v.x; p[1] = v.y; p[2] = p[3] = 0.0; }
};
template <> struct io<ffloat> {
    static ff2 get(const double* p) {
        return ff2{ffloat((float)p[0], (float)p[2]), ffloat((float)p[1], (float)p[3])};
    }
    static void put(double* p, ff2 v) { p[0] = v.x.h; p[1] = v.y.h; p[2] = v.x.l; p[3] = v.y.l; }
};
// in [m][4 phasors: at q = 0, at the anchor, the step, four steps][re, im, their second words]; out [m][N][4]
template <typename R, int N> void go(int m, const double* in, double* run, double* row) {
    for (int i = 0; i < m; ++i, in += 16, run += 4 * N, row += 4 * N) {
        phasor_run<R, N>(io<R>::get(in + 4), io<R>::get(in + 8), io<R>::get(in + 12),
                         [&](int q, cplx<R> w) { io<R>::put(run + 4 * q, w); });
        cplx<R> w = io<R>::get(in);
        for (int q = 0; q < N; ++q, w = cmul(w, io<R>::get(in + 8))) io<R>::put(row + 4 * q, w);
    }
}
extern "C" int anchor(int n) { return phasor_anchor(n); }
extern "C" void runs(int ff, int n, int m, const double* in, double* run, double* row) {
    if (n == 1) ff ? go<ffloat, 1>(m, in, run, row) : go<double, 1>(m, in, run, row);
    if (n == 2) ff ? go<ffloat, 2>(m, in, run, row) : go<double, 2>(m, in, run, row);
    if (n == 4) ff ? go<ffloat, 4>(m, in, run, row) : go<double, 4>(m, in, run, row);
    if (n == 8) ff ? go<ffloat, 8>(m, in, run, row) : go<double, 8>(m, in, run, row);
    if (n == 16) ff ? go<ffloat, 16>(m, in, run, row) : go<double, 16>(m, in, run, row);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return compile_host(SOURCE, str(tmp_path_factory.mktemp("phasor")))


@pytest.mark.parametrize("top", [0.01, 0.39, 2.0 * np.pi])
@pytest.mark.parametrize("n", [1, 2, 4, 8, 16])
@pytest.mark.parametrize("form", ["fp64", "ff"])
def test_a_run_is_no_less_accurate_than_products_in_a_row(lib, form, n, top):
    m = 20000
    rng = np.random.default_rng(n)
    phi, theta = (rng.uniform(0.0, t, m).astype(np.longdouble) for t in (2.0 * np.pi, top))
    word = np.float64 if form == "fp64" else np.float32
    inputs = np.zeros((m, 4, 4))
    for s, angle in enumerate((phi, phi + lib.anchor(n) * theta, theta, 4 * theta)):
        for c, v in enumerate((np.cos(angle), np.sin(angle))):
            inputs[:, s, c] = v.astype(word)
            if form == "ff":
                inputs[:, s, 2 + c] = (v - inputs[:, s, c]).astype(word)
    out = np.zeros((2, m, n, 4))
    ptr = lambda a: a.ctypes.data_as(ctypes.POINTER(ctypes.c_double))
    lib.runs(int(form == "ff"), n, m, ptr(inputs), ptr(out[0]), ptr(out[1]))
    angle = phi[:, None] + np.arange(n) * theta[:, None]
    value = out[..., :2].astype(np.longdouble) + out[..., 2:]
    err = np.hypot(value[..., 0] - np.cos(angle), value[..., 1] - np.sin(angle)).astype(float)
    run, row = err[0].max(axis=1), err[1].max(axis=1)   # the worst of each run
    unit = 2.0 ** -53 if form == "fp64" else 2.0 ** -48
    text = f"{form} N = {n}: worst {run.max() / unit:.2f} / {row.max() / unit:.2f}, mean {run.mean() / unit:.2f} / {row.mean() / unit:.2f}"
    print(text)
    assert run.max() <= row.max() and run.mean() <= row.mean(), text
