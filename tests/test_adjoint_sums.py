"""The FP32 form's band sums (CPU, the kernel's own source compiled for the host): pairs of floats against exact
sums of the same terms, also where the terms cancel. u = 2^-24 throughout.

Bounds, with S the sum of the terms' sizes. A thread's n terms: the second word adds up n errors of at most u S
from the first word's additions, and n of the products' (u of each term), so it stays below (n + 1) u S; each of its
2 n additions and the products' own second roundings lose u of what they add: (n + 2)^2 u^2 S in all. A sum of
two pairs (one two-sum of the first words, the second words added to its error): at most 4 u^2 of their sizes,
12 of them on the way from a thread to the CTA's total (5 across a warp, 7 across the warps)."""

import ctypes
from fractions import Fraction

import numpy as np
import pytest

from host_code import compile_host

SOURCE = r"""
#include "fcas_sums.cuh"
using namespace fcas;
// sums of a CTA of 256 threads over n terms each: w [256][n][2], q [256][n]; kind 0: sum of q, 1: of w[0] q,
// 2: of (w[0] + w[1]) q. thread [256], total: the sums as doubles
extern "C" void cta_sums(int kind, int n, const float* w, const float* q, double* thread, double* total) {
    SumF t[256];
    for (int j = 0; j < 256; ++j) {
        sum_zero(t[j]);
        for (int i = 0; i < n; ++i) {
            const float* wi = w + 2 * (j * n + i);
            if (kind == 0) sum_add(t[j], q[j * n + i]);
            if (kind == 1) sum_add_w(t[j], wi[0], q[j * n + i]);
            if (kind == 2) sum_add_w(t[j], make_float2(wi[0], wi[1]), q[j * n + i]);
        }
        thread[j] = sum_value(t[j]);
        sum_normalise(t[j]);
    }
    for (int v = 0; v < 256; v += 32)
        for (int off = 16; off > 0; off >>= 1)
            for (int j = 0; j < off; ++j) t[v + j] = sum_of(t[v + j], t[v + j + off]);
    for (int v = 32; v < 256; v += 32) t[0] = sum_of(t[0], t[v]);
    *total = sum_value(t[0]);
}
"""
U = 2.0 ** -24


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return compile_host(SOURCE, str(tmp_path_factory.mktemp("sums")))


@pytest.mark.parametrize("cancelling", [False, True])
@pytest.mark.parametrize("n", [1, 2, 31, 128])   # 128: the terms of a thread at 2^24 points
@pytest.mark.parametrize("kind", [0, 1, 2])
def test_pairs_against_exact_sums(lib, kind, n, cancelling):
    rng = np.random.default_rng(100 * kind + n)
    q = rng.standard_normal((256, n)).astype(np.float32)
    q *= np.exp2(rng.integers(-6, 7, (256, n))).astype(np.float32)
    w = np.ones((256, n, 2), dtype=np.float32)
    if kind:
        hi = rng.uniform(0.01, 1.0, (256, n))
        w[..., 0] = hi
        w[..., 1] = np.float32(0) if kind == 1 else (hi - w[..., 0]).astype(np.float32)
    else:
        w[..., 1] = 0.0
    if cancelling and n > 1:   # the second half of a thread's terms takes the first half back
        h = n // 2
        q[:, h:2 * h], w[:, h:2 * h] = -q[:, :h], w[:, :h]
        q[:, 2 * h:] *= np.float32(2.0 ** -20)
    thread, total = np.zeros(256), np.zeros(1)
    f, d = (lambda a, t=t: a.ctypes.data_as(ctypes.POINTER(t)) for t in (ctypes.c_float, ctypes.c_double))
    lib.cta_sums(kind, n, f(w), f(q), d(thread), d(total))
    weight = [[Fraction(float(a)) + (Fraction(float(b)) if kind == 2 else 0) for a, b in row] for row in w]
    terms = [[x * Fraction(float(y)) for x, y in zip(wr, qr)] for wr, qr in zip(weight, q)]
    sizes = [float(sum(map(abs, row))) for row in terms]
    for j in range(256):
        assert abs(float(Fraction(thread[j]) - sum(terms[j]))) <= (n + 2) ** 2 * U * U * sizes[j] + 1e-300
    exact = sum(map(sum, terms))
    assert abs(float(Fraction(total[0]) - exact)) <= ((n + 2) ** 2 + 12 * 4) * U * U * sum(sizes)
    # and far below the rounding that the FP32 terms themselves carry
    assert abs(float(Fraction(total[0]) - exact)) <= U * sum(sizes) / 512
