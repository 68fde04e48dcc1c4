"""Calls on device arrays captured in a CUDA graph stay valid while the context is used for other things: a
replay reads and writes the arrays that the capture saw, so nothing the context owned then may be replaced."""

import numpy as np
import pytest

import synthdata as sd
from parity_util import make_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("captured", [40, 320])
def test_a_search_leaves_a_captured_fitness_valid(captured):
    # 320 rows on 2^16 points for 12 iterations: the search takes larger chunks than the context's
    import torch
    import paper_2002_02150_gb300 as fc
    w = sd.C1
    data = sd.make_dataset(w, 10)
    sets = [torch.tensor(sd.make_particles(w, captured, seed=s), device="cuda:0") for s in (1, 2)]
    cfg = fc.pso_config(n_runs=8, n_particles=40, n_iter=12, seed=3,
                        box=(0.0, 2.0 * np.pi, -0.5 * np.pi, 0.5 * np.pi) + sd.chirp_time_box(w.f_low))
    with make_ctx(w, data, "fp32") as ctx:
        expect = [[x.cpu().numpy() for x in fc.fcas_fitness(ctx, th)] for th in sets]
        theta = sets[0].clone()
        fit = torch.zeros(captured, dtype=torch.float64, device="cuda:0")
        tc = torch.zeros(captured, dtype=torch.int64, device="cuda:0")
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            fc.fcas_fitness(ctx, theta, fitness=fit, tc=tc)
        chunk = fc.fcas_get_info(ctx)["chunk"]
        first = fc.fcas_search(ctx, cfg)
        assert fc.fcas_get_info(ctx)["chunk"] == chunk
        for th, (f, t) in zip(sets, expect):
            theta.copy_(th)
            graph.replay()
            torch.cuda.synchronize()
            np.testing.assert_array_equal(fit.cpu().numpy(), f)
            np.testing.assert_array_equal(tc.cpu().numpy(), t)
        assert fc.fcas_search(ctx, cfg) == first


def test_a_change_of_shape_and_back_leaves_a_captured_gradient_valid():
    # 2^18 points: sixteen columns per CTA split the band into fewer segments than the default width does
    import dataclasses

    import torch
    import paper_2002_02150_gb300 as fc
    w = dataclasses.replace(sd.C1, n_fft=1 << 18, n_samples=200001, f_low=40.0)
    data = sd.make_dataset(w, 11)
    sets = [torch.tensor(sd.make_particles(w, 6, seed=s, f_star=w.f_low), device="cuda:0") for s in (1, 2)]
    with make_ctx(w, data, "fp32") as ctx:
        fc.fcas_set_shape(ctx, 0, 16, 16, 4)
        lags = [fc.fcas_fitness(ctx, th)[1] for th in sets]
        expect = [fc.fcas_gradient(ctx, th, t).cpu().numpy() for th, t in zip(sets, lags)]
        theta, tc, grad = sets[0].clone(), lags[0].clone(), torch.zeros_like(sets[0])
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            fc.fcas_gradient(ctx, theta, tc, grad=grad)
        fc.fcas_set_shape(ctx, 0, 0, 16, 0)
        fc.fcas_gradient(ctx, theta, tc)
        torch.cuda.synchronize()
        fc.fcas_set_shape(ctx, 0, 16, 16, 4)
        for th, t, g in zip(sets, lags, expect):
            theta.copy_(th)
            tc.copy_(t)
            graph.replay()
            torch.cuda.synchronize()
            np.testing.assert_array_equal(grad.cpu().numpy(), g)


def test_larger_chunks_leave_a_captured_fitness_valid():
    # the gradient call has made the particle records large enough: the larger evaluation replaces nothing
    import torch
    import paper_2002_02150_gb300 as fc
    w = sd.SMALL
    data = sd.make_dataset(w, 12)
    many = torch.tensor(sd.make_particles(w, 320, seed=1), device="cuda:0")
    sets = [many[:40].clone(), many[40:80].clone()]
    with make_ctx(w, data, "fp32") as ctx:
        fc.fcas_gradient(ctx, many, torch.zeros(320, dtype=torch.int64, device="cuda:0"))
        expect = [[x.cpu().numpy() for x in fc.fcas_fitness(ctx, th)] for th in sets]
        theta = sets[0].clone()
        fit = torch.zeros(40, dtype=torch.float64, device="cuda:0")
        tc = torch.zeros(40, dtype=torch.int64, device="cuda:0")
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            fc.fcas_fitness(ctx, theta, fitness=fit, tc=tc)
        chunk = fc.fcas_get_info(ctx)["chunk"]
        fc.fcas_fitness(ctx, many)
        assert fc.fcas_get_info(ctx)["chunk"] > chunk
        for th, (f, t) in zip(sets, expect):
            theta.copy_(th)
            graph.replay()
            torch.cuda.synchronize()
            np.testing.assert_array_equal(fit.cpu().numpy(), f)
            np.testing.assert_array_equal(tc.cpu().numpy(), t)
