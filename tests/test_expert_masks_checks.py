"""The Python call for expert masks refuses, before anything reaches the device, a layer outside `out` and an `out`
that is smaller than what the kernel writes (the C call gets addresses only and cannot check them)."""
import pytest
import torch

from paper_2608_15018_b200 import binding


class _Library:
    """Records the calls that would have reached the device."""

    def __init__(self):
        self.calls = []

    def s2moe_expert_masks(self, *args):
        self.calls.append(args)
        return binding.OK


@pytest.fixture
def library(monkeypatch):
    lib = _Library()
    monkeypatch.setattr(binding, "load_library", lambda: lib)
    monkeypatch.setattr(binding, "_dptr", lambda t: t.data_ptr())
    monkeypatch.setattr(binding, "_stream_handle", lambda stream: 0)
    return lib


@pytest.mark.parametrize("layer", [-1, 3, 4, 1 << 40])
def test_layer_outside_out(library, layer):
    with pytest.raises(ValueError, match="layer"):
        binding.expert_masks(torch.zeros((5, 2), dtype=torch.int32), 130, torch.zeros((5, 3, 3), dtype=torch.int64), layer)
    assert not library.calls


@pytest.mark.parametrize("shape,dtype", [((4, 3, 3), torch.int64), ((5, 3, 2), torch.int64), ((5, 3, 3), torch.int32)])
def test_out_smaller_than_what_is_written(library, shape, dtype):
    with pytest.raises(ValueError, match="out"):
        binding.expert_masks(torch.zeros((5, 2), dtype=torch.int32), 130, torch.zeros(shape, dtype=dtype), 0)
    assert not library.calls


def test_every_layer_has_its_own_address(library):
    out = torch.zeros((6, 3, 3), dtype=torch.int64)          # (a row more than there are tokens is no fault)
    for layer in range(3):
        assert binding.expert_masks(torch.zeros((5, 2), dtype=torch.int32), 130, out, layer) is out
    assert [c[4] - out.data_ptr() for c in library.calls] == [0, 24, 48] and all(c[5] == 9 for c in library.calls)
