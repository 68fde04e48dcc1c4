"""The geometry kernel takes eight lanes per particle and four particles per warp: batches that leave a
group of lanes empty, detector counts from one to eight, and invalid particles beside valid ones give
each particle what it gets alone, and the oracle's value."""

import numpy as np
import pytest

import synthdata as sd
from oracle import fcas_oracle as o
from parity_util import assert_parity, gpu_fitness

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_det", [1, 2, 7, 8])
def test_ragged_batches_and_invalid_neighbours(n_det):
    import paper_2002_02150_gb300 as fc
    w = sd.SMALL
    base = sd.make_dataset(w, 11)
    pick = np.arange(n_det) % 4
    det, psd, data = base["det"][pick].copy(), base["psd"][pick], base["data"][pick]
    det[4:, 0:3] *= 0.9       # repeated sites moved, so that their delays differ
    theta = sd.make_particles(w, 9, seed=11)
    bad = theta.copy()
    bad[[1, 4, 8]] = [[np.nan, 0.1, 3.0, 0.3], [1.0, 0.1, -1.0, 0.3], [1.0, 0.1, 3.0, np.inf]]
    with fc.fcas_create(det, psd, data, w.n_fft, w.fs, w.f_low, w.f_high, precision="fp64") as ctx:
        alone = [gpu_fitness(ctx, theta[j:j + 1]) for j in range(9)]
        for n in (1, 3, 4, 5, 9):
            f, t = gpu_fitness(ctx, theta[:n])
            np.testing.assert_array_equal(f, [alone[j][0][0] for j in range(n)])
            np.testing.assert_array_equal(t, [alone[j][1][0] for j in range(n)])
        f, t = gpu_fitness(ctx, bad)
        for j in range(9):
            if j in (1, 4, 8):
                assert np.isnan(f[j]) and t[j] == -1
            else:
                assert (f[j], t[j]) == (alone[j][0][0], alone[j][1][0])
    setup = o.OracleSetup(det, psd, data, w.n_fft, w.fs, w.f_low, w.f_high)
    assert_parity(setup, theta, np.array([a[0][0] for a in alone]), np.array([a[1][0] for a in alone]), "fp64")
