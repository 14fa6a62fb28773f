"""The binding's check of a tensor's device while torch.cuda is not initialised.

Native code can make a CUDA tensor without the Python side having initialised
CUDA. Such a tensor is taken when it is on the current device and refused for
what is wrong with it otherwise. Tensors that report a CUDA device stand in for
it here.
"""
import pytest
import torch

import paper_2510_11683_gb300 as bg


class _OnGpu(torch.Tensor):
    """A CPU tensor that says it is on cuda:`index`."""
    index = 0

    @property
    def is_cuda(self):
        return True

    @property
    def device(self):
        return torch.device("cuda", self.index)

    def get_device(self):
        return self.index


def _on_gpu(t, index=0):
    t = t.as_subclass(_OnGpu)
    t.index = index
    return t


@pytest.fixture(autouse=True)
def _uninitialised(monkeypatch):
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: False)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)


def test_a_tensor_of_the_current_device_is_taken():
    t = torch.zeros(4)
    assert bg._current_device() == -1
    assert bg._ptr(_on_gpu(t), torch.float32, "ell") == t.data_ptr()
    assert bg._ptr(_on_gpu(t), torch.float32, "ell", bg._current_device()) == t.data_ptr()


@pytest.mark.parametrize("tensor,error,text", [
    (lambda: torch.zeros(4), ValueError, "must be a CUDA tensor"),
    (lambda: _on_gpu(torch.zeros(4), 1), ValueError, "is on cuda:1"),
    (lambda: _on_gpu(torch.zeros(4, dtype=torch.float64)), TypeError, "must be torch.float32"),
    (lambda: _on_gpu(torch.zeros(4, 4)[:, 1]), ValueError, "must be contiguous"),
    (lambda: [0.0], TypeError, "must be a torch.Tensor"),
])
def test_what_is_wrong_with_another_is_named(tensor, error, text):
    with pytest.raises(error, match=text):
        bg._ptr(tensor(), torch.float32, "ell")
