"""Launch shapes of the shortest transforms: a split either is refused, and leaves the context as it was, or
evaluates; and the autotuner ends with one that evaluates. 2^4 to 2^10 points, every form, against the oracle."""

import dataclasses

import pytest

import synthdata as sd
from parity_util import assert_parity, gpu_fitness, make_ctx, oracle_setup

pytestmark = pytest.mark.gpu

SIZES = [(16, 16, 16.0, 1.5, 6.0), (32, 27, 32.0, 2.2, 12.0), (64, 50, 64.0, 5.0, 28.0),
         (128, 128, 128.0, 10.0, 50.0), (256, 200, 128.0, 12.0, 60.0), (512, 511, 256.0, 30.0, 120.0),
         (1024, 900, 256.0, 30.0, 120.0)]


@pytest.mark.parametrize("precision", ["fp32", "fp64", "ff"])
@pytest.mark.parametrize("n_fft,n_samples,fs,f_low,f_high", SIZES)
def test_every_accepted_shape_and_the_tuned_one_evaluate(precision, n_fft, n_samples, fs, f_low, f_high):
    import paper_2002_02150_gb300 as fc
    w = dataclasses.replace(sd.SMALL, n_fft=n_fft, n_samples=n_samples, fs=fs, f_low=f_low, f_high=f_high,
                            arrival_s=0.3 * n_samples / fs)
    data = sd.make_dataset(w, 3)
    theta = sd.make_particles(w, 5, seed=3, f_star=f_low)
    setup = oracle_setup(w, data)
    shape = lambda info: tuple(info[k] for k in ("split_bias", "k1b", "sub", "radix_bits_a"))

    def check(ctx, context):
        f, t = gpu_fitness(ctx, theta)
        assert_parity(setup, theta, f, t, precision, context)

    with make_ctx(w, data, precision) as ctx:
        for bias in (0, 1):
            before = shape(fc.fcas_get_info(ctx))
            try:
                fc.fcas_set_shape(ctx, bias, 0, 16, 0)
            except fc.FcasError as e:
                assert e.code == -1 and bias == 1      # FCAS_ERR_INVALID; the balanced split always exists
                assert shape(fc.fcas_get_info(ctx)) == before
            check(ctx, f"N={n_fft} bias {bias}")
        info = fc.fcas_autotune(ctx, 8)
        assert info["tuned_ms_per_particle"] > 0
        check(ctx, f"N={n_fft} tuned {shape(info)}")


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("w", [sd.SMALL, sd.C1], ids=["small", "64s"])
def test_the_binding_s_default_shape_is_the_one_at_creation(w, precision):
    import paper_2002_02150_gb300 as fc
    with make_ctx(w, sd.make_dataset(w, 3), precision) as ctx:
        created = fc.fcas_get_info(ctx)
        fc.fcas_set_shape(ctx, sub=1)
        again = fc.fcas_set_shape(ctx)
    assert again == created
