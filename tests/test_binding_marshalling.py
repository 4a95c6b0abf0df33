"""Argument marshalling of the binding that needs no GPU: the shapes and devices `empty` takes."""
from types import SimpleNamespace

import numpy as np
import pytest
import torch

from paper_2512_18345_gb300 import binding


@pytest.fixture
def made(monkeypatch):
    calls = []
    fake = SimpleNamespace(int32=torch.int32, device=torch.device,
                           empty=lambda shape, dtype, device: calls.append((shape, device)))
    monkeypatch.setattr(binding, "_cuda", lambda: fake)
    monkeypatch.setattr(binding, "_devices", {})
    return calls


@pytest.mark.parametrize("shape", [(2, 3), [2, 3], torch.Size((2, 3)), np.array([2, 3]), map(int, "23")])
def test_any_sequence_is_a_shape(made, shape):
    binding.empty(shape)
    assert type(made[0][0]) is tuple and made[0][0] == (2, 3)


@pytest.mark.parametrize("device", [1, np.int64(1), "1"])
def test_device_index_of_any_integer_kind(made, device):
    binding.empty((1,), device)
    assert made[0][1] == torch.device("cuda", 1)
