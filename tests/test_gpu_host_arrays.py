"""Host arrays of fcas_fitness: small batches go through pinned memory that the kernels read and write,
larger ones through copies; both, and calls that mix host and device arrays, give the device arrays' bits."""

import numpy as np
import pytest

import synthdata as sd
from parity_util import make_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 7, 1024, 1025])
def test_host_and_mixed_arrays_equal_device_arrays(n):
    import torch
    import paper_2002_02150_gb300 as fc
    w = sd.SMALL
    data = sd.make_dataset(w, 9)
    theta = sd.make_particles(w, n, seed=9)
    with make_ctx(w, data, "fp32") as ctx:
        dev = torch.tensor(theta, device="cuda:0")
        f, t = (x.cpu().numpy() for x in fc.fcas_fitness(ctx, dev))
        for _ in range(2):
            hf, ht = fc.fcas_fitness(ctx, theta)
            np.testing.assert_array_equal(hf, f)
            np.testing.assert_array_equal(ht, t)
        other = fc.fcas_fitness(ctx, theta[::-1].copy())       # the staging holds other particles now
        np.testing.assert_array_equal(other[0], f[::-1])
        np.testing.assert_array_equal(hf, f)                   # results already returned stay
        out = torch.empty(n, dtype=torch.float64, device="cuda:0")
        lag = np.empty(n, dtype=np.int64)
        fc.fcas_fitness(ctx, theta, fitness=out, tc=lag)       # host in, one output on each side
        np.testing.assert_array_equal(out.cpu().numpy(), f)
        np.testing.assert_array_equal(lag, t)
        hf, lag = np.empty(n), torch.empty(n, dtype=torch.int64, device="cuda:0")
        fc.fcas_fitness(ctx, dev, fitness=hf, tc=lag)          # device in
        np.testing.assert_array_equal(hf, f)
        np.testing.assert_array_equal(lag.cpu().numpy(), t)
