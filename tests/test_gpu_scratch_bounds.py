"""Device memory that contexts and groups hold against what fcas.h says of it."""

import numpy as np
import pytest

import synthdata as sd
from parity_util import make_ctx

pytestmark = pytest.mark.gpu

SLACK = 6 << 20      # allocations come in pages of 2 MB; the other arrays of these short segments are far smaller


def held(make):
    """What make() returns, and the bytes of device memory it holds."""
    import torch
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    thing = make()
    torch.cuda.synchronize()
    return thing, free - torch.cuda.mem_get_info()[0]


def search_config(w, runs, iterations):
    import paper_2002_02150_gb300 as fc
    return fc.pso_config(n_runs=runs, n_particles=40, n_iter=iterations, seed=2,
                         box=(0.0, 2.0 * np.pi, -0.5 * np.pi, 0.5 * np.pi) + sd.chirp_time_box(w.f_low))


def test_an_automatic_group_holds_scratch_for_at_most_64_particles():
    import paper_2002_02150_gb300 as fc
    w = sd.C1
    per_particle = 2 * w.n_fft * 8
    data = sd.make_dataset(w, 12)
    ctxs = [fc.fcas_create(data["det"], data["psd"], data["data"], w.n_fft, w.fs, w.f_low, w.f_high,
                           flags=fc.FCAS_SETUP_LAZY_SCRATCH) for _ in range(2)]
    cfg = search_config(w, 8, 20)
    warm = fc.fcas_group_create(ctxs, max_batch=3)       # what the first search loads stays out of the count
    expect = warm.search(cfg)
    warm.close()

    def make():
        g = fc.fcas_group_create(ctxs)
        assert g.search(cfg) == expect
        return g
    group, size = held(make)
    assert size <= 64 * per_particle + SLACK      # (the search has given its larger chunks back)
    group.close()
    for c in ctxs:
        c.close()


@pytest.mark.parametrize("log_n", [12, 16])
def test_an_automatic_context_holds_scratch_for_the_batches_it_is_given(log_n):
    import torch
    import paper_2002_02150_gb300 as fc
    w = sd.SMALL if log_n == 12 else sd.C1
    per_particle = 2 * w.n_fft * 8
    data = sd.make_dataset(w, 13)
    theta = torch.tensor(sd.make_particles(w, 640, seed=13), device="cuda:0")
    with make_ctx(w, data, "fp32", max_batch=8) as ctx:     # what the first calls load stays out of the count
        expect = [x.cpu().numpy() for x in fc.fcas_fitness(ctx, theta)]
    f, t = torch.empty(640, dtype=torch.float64, device="cuda:0"), torch.empty(640, dtype=torch.int64, device="cuda:0")

    def check(ctx, n):
        fc.fcas_fitness(ctx, theta[:n], fitness=f[:n], tc=t[:n])
        np.testing.assert_array_equal(f[:n].cpu().numpy(), expect[0][:n])
        np.testing.assert_array_equal(t[:n].cpu().numpy(), expect[1][:n])

    def make(n):
        ctx = make_ctx(w, data, "fp32")
        if n:
            check(ctx, n)
        return ctx
    bare, rest = held(lambda: fc.fcas_create(data["det"], data["psd"], data["data"], w.n_fft, w.fs, w.f_low, w.f_high,
                                             flags=fc.FCAS_SETUP_LAZY_SCRATCH))     # everything but the scratch
    bare.close()
    sizes = {}
    for n in (0, 64, 640):
        ctx, size = held(lambda: make(n))
        sizes[n] = size - rest
        assert fc.fcas_get_info(ctx)["chunk"] == (64 if n <= 64 else min(n, (128 << 20) // per_particle))
        check(ctx, 64)
        check(ctx, 640)
        ctx.close()
    assert sizes[0] <= 64 * per_particle + SLACK
    assert sizes[64] <= 64 * per_particle + SLACK
    assert sizes[640] <= 64 * per_particle + min(640 * per_particle, 128 << 20) + SLACK


def test_searches_take_larger_chunks_once_these_pay_and_find_the_same():
    import paper_2002_02150_gb300 as fc
    w = sd.C1
    data = sd.make_dataset(w, 14)
    short, long = search_config(w, 8, 2), search_config(w, 8, 40)
    with make_ctx(w, data, "fp32", max_batch=64) as ctx:    # the caller's bound is kept
        expect = [fc.fcas_search(ctx, cfg) for cfg in (short, long)]
        again, size = held(lambda: fc.fcas_search(ctx, long))
        assert again == expect[1] and size <= SLACK
    with make_ctx(w, data, "fp32") as ctx:
        for cfg, ref, top in ((short, expect[0], 0), (long, expect[1], 512 << 20), (long, expect[1], 0)):
            got, size = held(lambda: fc.fcas_search(ctx, cfg))
            assert got == ref and size <= top + SLACK
