"""Overlapped launches: the kernels of a call start while their predecessors drain. Many calls with
different particles enqueued without a wait between them, in one chunk and in several, give the bits of
the same calls made one at a time."""

import numpy as np
import pytest

import synthdata as sd
from parity_util import make_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64", "ff"])
@pytest.mark.parametrize("max_batch", [0, 1, 3])
def test_calls_in_flight_equal_calls_alone(precision, max_batch):
    import torch
    import paper_2002_02150_gb300 as fc
    w = sd.SMALL
    data = sd.make_dataset(w, 8)
    sets = [torch.tensor(sd.make_particles(w, 10, seed=s), device="cuda:0") for s in range(6)]
    sets[2][4, 2] = float("nan")
    with make_ctx(w, data, precision) as ctx:
        alone = []
        for th in sets:
            f, t = fc.fcas_fitness(ctx, th)
            g = fc.fcas_gradient(ctx, th, t)
            torch.cuda.synchronize()
            alone.append([x.cpu().numpy() for x in (f, t, g)])
    with make_ctx(w, data, precision, max_batch=max_batch) as ctx:
        got = []
        for r in range(40):
            f, t = fc.fcas_fitness(ctx, sets[r % 6])
            got.append((f, t, fc.fcas_gradient(ctx, sets[r % 6], t)))
        torch.cuda.synchronize()
        for r, res in enumerate(got):
            for x, ref in zip(res, alone[r % 6]):
                np.testing.assert_array_equal(x.cpu().numpy(), ref)
