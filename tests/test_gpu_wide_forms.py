"""Binary64 and float-float passes at the sizes where their phasor runs and constant staging change:
columns of 4 to 64 points (2 to 8 bins per thread), more detectors than a CTA has threads, one
detector (no relative delays), and delays of many turns, against the oracle."""

import numpy as np
import pytest

import synthdata as sd
from oracle import fcas_oracle as o
from parity_util import assert_parity, gpu_fitness

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "ff"])
@pytest.mark.parametrize("log_n,n_det,stretch", [(4, 8, 1.0), (4, 1, 1.0), (6, 5, 1.0), (7, 8, 1.0), (12, 1, 1.0),
                                                 (12, 8, 30.0)])
def test_short_columns_many_detectors_long_delays(precision, log_n, n_det, stretch):
    import paper_2002_02150_gb300 as fc
    n, fs, f_low, f_high = 1 << log_n, 1024.0, 80.0, 400.0
    rng = np.random.default_rng(log_n + n_det)
    pick = np.arange(n_det) % 4
    det = sd.detector_geometry()[pick].copy()
    det[:, 0:3] *= stretch * (1.0 + 0.1 * np.arange(n_det))[:, None]   # 30: delays of up to ~0.6 s
    psd = sd.psd_on_grid(1, n, fs)[np.zeros(n_det, dtype=int)]
    data = rng.standard_normal((n_det, n)) * 1e-22
    w = sd.SMALL
    theta = sd.make_particles(w, 5, seed=3, f_star=f_low)
    with fc.fcas_create(det, psd, data, n, fs, f_low, f_high, precision=precision) as ctx:
        f, t = gpu_fitness(ctx, theta)
    assert_parity(o.OracleSetup(det, psd, data, n, fs, f_low, f_high), theta, f, t, precision, f"N=2^{log_n}")
