"""The allocation-free binding's short check takes exactly what its long check takes (CPU, with a library and
tensors that stand in for the device's)."""

import pytest
import torch

from paper_2002_02150_gb300 import fcas as binding


class _Claims:
    """What a CUDA tensor of the current device says of itself."""
    is_cuda = property(lambda self: True)
    device = property(lambda self: torch.device("cuda", 0))

    def get_device(self):
        return 0


class ForeignTensor(_Claims, torch.Tensor):
    """A subclass from a module that is not torch's."""


class OwnTensor(_Claims, torch.Tensor):
    __module__ = "torch.stand_in"


class _Library:
    def __init__(self):
        self.calls = []

    def fcas_fitness_noalloc(self, handle, n, theta, fitness, tc, stream):
        self.calls.append((n, stream.value))
        return 0


class _Context:
    handle = None


def arrays(kind):
    make = lambda shape, dtype: torch.zeros(shape, dtype=dtype).as_subclass(kind)
    return make((5, 4), torch.float64), make((5,), torch.float64), make((5,), torch.int64)


@pytest.fixture
def library(monkeypatch):
    lib = _Library()
    monkeypatch.setattr(binding, "load_library", lambda: lib)
    monkeypatch.setattr(binding, "_current_stream", lambda: 1234)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    return lib


@pytest.mark.parametrize("foreign", [(0, 1, 2), (0,), (1,), (2,)])
def test_a_tensor_the_long_check_refuses_never_reaches_the_library(library, foreign):
    own, other = arrays(OwnTensor), arrays(ForeignTensor)
    args = [other[i] if i in foreign else own[i] for i in range(3)]
    with pytest.raises(TypeError):
        binding.fcas_fitness_noalloc(_Context(), *args)
    assert not library.calls


def test_a_tensor_that_passes_runs_on_the_current_stream(library):
    binding.fcas_fitness_noalloc(_Context(), *arrays(OwnTensor))
    assert library.calls == [(5, 1234)]
