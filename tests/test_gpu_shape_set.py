"""Every launch shape of pass A, form by form: exactly the (width, radix) pairs of the rules below are accepted for a
column length, everything else is refused as invalid, and every accepted one matches the oracle. The FP32 form's
2^10- to 2^12-point columns (2^22 to 2^24 points) with all their widths and both radices, the binary64 and
float-float forms' 2^7- to 2^11-point columns."""

import dataclasses

import numpy as np
import pytest

import synthdata as sd
from oracle import fcas_oracle as o
from parity_util import RTOL, TIE_RTOL, gpu_fitness, make_ctx, oracle_setup

pytestmark = pytest.mark.gpu

# columns per CTA by log2 of the column length, with radix-16 and with radix-8 stages
WIDTHS = {("fp32", 4): {8: {4, 8, 16}, 9: {2, 4, 8, 16}, 10: {1, 2, 4, 8}, 11: {1, 2, 4}, 12: {1, 2}},
          ("fp32", 3): {10: {2, 4}, 11: {2, 4}, 12: {2}},
          ("fp64", 4): {7: {16}, 8: {8, 16}, 9: {4, 8}, 10: {2, 4}, 11: {1, 2}}, ("fp64", 3): {},
          ("ff", 4): {7: {16}, 8: {16}, 9: {8}, 10: {4}, 11: {2}}, ("ff", 3): {10: {2}, 11: {2}}}


def workload(log_n):
    n = 1 << log_n
    if log_n < 22:
        return dataclasses.replace(sd.C1, n_fft=n, n_samples=n - n // 9 - 1, f_low=60.0 * (65536 / n) ** 0.375)
    return dataclasses.replace(sd.C2, detectors=("H1", "L1"), n_fft=n, n_samples=n - 12345)


@pytest.mark.parametrize("precision,log_n", [("fp32", 22), ("fp32", 23), ("fp32", 24), ("fp64", 17), ("fp64", 19),
                                             ("fp64", 21), ("fp64", 23), ("ff", 17), ("ff", 19), ("ff", 21), ("ff", 23)])
def test_the_shapes_of_the_rules_and_no_others(precision, log_n):
    import paper_2002_02150_gb300 as fc
    w = workload(log_n)
    data = sd.make_dataset(w, 4)
    theta = sd.make_particles(w, 2, seed=4, f_star=w.f_low)
    setup = oracle_setup(w, data)
    curves = [o.fitness_curve(setup, th)[: w.n_samples] for th in theta]
    with make_ctx(w, data, precision, max_batch=2) as ctx:
        for bias in (0, 1):
            log_l = max(2, log_n - 13, log_n // 2 - bias)
            accepted = set()
            for k1b in (1, 2, 4, 8, 16):
                for radix_bits in (4, 3):
                    try:
                        fc.fcas_set_shape(ctx, bias, k1b, 16, radix_bits)
                    except fc.FcasError as e:
                        assert e.code == -1
                        continue
                    accepted.add((k1b, radix_bits))
                    f, t = gpu_fitness(ctx, theta)
                    for j, c in enumerate(curves):
                        best = float(c.max())
                        context = f"{precision} 2^{log_n} bias {bias} k1b {k1b} radix bits {radix_bits} particle {j}"
                        assert abs(f[j] - best) <= RTOL[precision] * best, context
                        assert t[j] == int(np.argmax(c)) or abs(c[t[j]] - best) <= TIE_RTOL * best, context
            assert accepted == {(k, rb) for rb in (4, 3) for k in WIDTHS[precision, rb].get(log_l, ())}
