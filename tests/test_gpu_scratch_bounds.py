"""Device memory that contexts and groups hold against what fcas.h says of it."""

import numpy as np
import pytest

import synthdata as sd
from parity_util import make_ctx

pytestmark = pytest.mark.gpu

SLACK = 6 << 20      # allocations come in pages of 2 MB; the other arrays of these short segments are far smaller


def held(make):
    """Bytes of device memory held by what make() returns (and what a second call of it returns)."""
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
    assert size <= 64 * per_particle + SLACK
    group.close()
    for c in ctxs:
        c.close()
