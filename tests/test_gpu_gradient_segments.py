"""Segmented band sums of the adjoint: transform lengths from one column block to several segments,
detector counts that leave a pair half filled, ragged bands and every layout width, against the
oracle's gradient; and the same bits whatever the batch (across the launch chunk's boundary too)."""

import dataclasses

import numpy as np
import pytest

import synthdata as sd
from parity_util import make_ctx, oracle_setup
from test_gpu_gradient import _check, _gpu_grad

pytestmark = pytest.mark.gpu


def _case(n_fft, n_samples, fs, f_low, f_high, n_det):
    return dataclasses.replace(sd.SMALL, n_fft=n_fft, n_samples=n_samples, fs=fs, f_low=f_low, f_high=f_high,
                               detectors=("H1", "L1", "V1", "K1")[:n_det], arrival_s=0.3 * n_samples / fs)


# (n_fft, n_samples, fs, f_low, f_high, detectors): 16 points (one column block, one bin row), one
# segment, two, an odd detector count, a band of few rows at the top of the spectrum, 16 segments
CASES = [(16, 16, 1024.0, 80.0, 400.0, 4), (256, 200, 128.0, 12.0, 60.0, 3), (8192, 6001, 512.0, 60.0, 250.0, 2),
         (8192, 8192, 512.0, 200.0, 201.0, 4), (65536, 40001, 1024.0, 60.0, 470.0, 3)]


@pytest.mark.parametrize("case", CASES, ids=[f"N{c[0]}-D{c[5]}" for c in CASES])
@pytest.mark.parametrize("precision", ["fp32", "fp64", "ff"])
def test_segments_match_the_oracle(case, precision):
    w = _case(*case)
    data = sd.make_dataset(w, 5)
    theta = sd.make_particles(w, 3, seed=5)
    with make_ctx(w, data, precision) as ctx:
        f, tc, g = _gpu_grad(ctx, theta)
    _check(oracle_setup(w, data), theta, tc, g, precision, f"N={w.n_fft}")


def test_same_bits_in_any_batch_and_layout():
    import paper_2002_02150_gb300 as fc
    w = _case(65536, 65536, 1024.0, 60.0, 500.0, 4)
    data = sd.make_dataset(w, 5)
    few = sd.make_particles(w, 5, seed=5)
    with make_ctx(w, data, "fp32") as ctx:
        f, tc, g = _gpu_grad(ctx, few)
        # a batch larger than one launch takes (2^15 particle-segments at 16 segments)
        many, tcs = np.tile(few, (500, 1)), np.tile(tc, 500)
        np.testing.assert_array_equal(fc.fcas_gradient(ctx, many, tcs), np.tile(g, (500, 1)))
        for j in range(5):
            np.testing.assert_array_equal(fc.fcas_gradient(ctx, few[j:j + 1], tc[j:j + 1]), g[j:j + 1])
        # other layouts add the same terms in another order: binary64-class agreement
        for k1b in (8, 16):
            fc.fcas_set_shape(ctx, 0, k1b, 8, 4)
            g2 = fc.fcas_gradient(ctx, few, tc)
            assert np.all(np.abs(g2 - g) <= 1e-9 * np.abs(g).max(axis=1, keepdims=True))
