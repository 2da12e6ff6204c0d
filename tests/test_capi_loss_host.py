"""gabm_cumulative_mse takes device memory only: arrays that are not all CUDA tensors are refused
before the library (here a stand-in) sees a pointer."""
from types import SimpleNamespace

import numpy as np
import pytest
import torch

from paper_2207_09714_gb300 import capi


class OnDevice(torch.Tensor):
    """A host tensor that says it is a CUDA one."""
    is_cuda = True


def on_device(shape=(2, 5)):
    return torch.rand(shape, dtype=torch.float64).as_subclass(OnDevice)


@pytest.mark.parametrize("D,y", [(on_device(), np.zeros((2, 5))), (on_device(), torch.zeros((2, 5), dtype=torch.float64)),
                                 (torch.zeros((2, 5), dtype=torch.float64), on_device()),
                                 (np.zeros((2, 5)), np.zeros((2, 5))),
                                 (torch.zeros((2, 5), dtype=torch.float64), torch.zeros((2, 5), dtype=torch.float64))],
                         ids=["host array target", "host tensor target", "host deaths", "host arrays", "host tensors"])
def test_host_operands_are_refused(monkeypatch, D, y):
    calls = []
    library = SimpleNamespace(gabm_cumulative_mse=lambda *a: calls.append(a) or 0)
    monkeypatch.setattr(capi, "load_library", lambda: library)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda device=None: SimpleNamespace(cuda_stream=0))
    with pytest.raises(ValueError):
        capi.gabm_cumulative_mse(D, y)
    assert not calls
    capi.gabm_cumulative_mse(on_device(), on_device())
    assert len(calls) == 1
