"""The FP32 form's transforms exchange data within a warp wherever a residue class or a whole transform
fits one, with their own order of rows and twiddles: every pass length from 2^8 to 2^12 points on either
side, with every compiled column width and stage radix, against the oracle."""

import dataclasses

import numpy as np
import pytest

import synthdata as sd
from oracle import fcas_oracle as o
from parity_util import RTOL, TIE_RTOL, gpu_fitness, make_ctx, oracle_setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log_n", [17, 18, 19, 20, 21])
def test_pass_lengths_and_widths_match_the_oracle(log_n):
    import paper_2002_02150_gb300 as fc
    n = 1 << log_n
    w = dataclasses.replace(sd.C1, n_fft=n, n_samples=n - n // 9 - 1, f_low=60.0 * (65536 / n) ** 0.375)
    data = sd.make_dataset(w, 4)
    theta = sd.make_particles(w, 3, seed=4, f_star=w.f_low)
    setup = oracle_setup(w, data)
    curves = [o.fitness_curve(setup, th)[: w.n_samples] for th in theta]
    with make_ctx(w, data, "fp32", max_batch=2) as ctx:
        tried = 0
        for bias in (0, 1):
            for k1b in (1, 2, 4, 8, 16):
                for radix_bits in (4, 3):
                    try:
                        fc.fcas_set_shape(ctx, bias, k1b, 16, radix_bits)
                    except fc.FcasError:
                        continue
                    tried += 1
                    f, t = gpu_fitness(ctx, theta)
                    for j, c in enumerate(curves):
                        best = float(c.max())
                        context = f"2^{log_n} bias {bias} k1b {k1b} radix bits {radix_bits} particle {j}"
                        assert abs(f[j] - best) <= RTOL["fp32"] * best, context
                        assert t[j] == int(np.argmax(c)) or abs(c[t[j]] - best) <= TIE_RTOL * best, context
        assert tried >= 4
