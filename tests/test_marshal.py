"""What the marshalling extension takes and refuses: the same objects, and the same exceptions, as the ctypes calls of the
other entry points."""
import pytest
import torch

from paper_1909_04823_b200 import binding as D


@pytest.fixture(scope="module")
def native():
    return D.native()


@pytest.mark.parametrize("shape", [(6,), (2, 3, 4)])
def test_cross_takes_matrices_only(shape):
    x, w = torch.zeros(shape), torch.zeros(shape[-1])
    with pytest.raises(ValueError):
        D.cross_forward(x, x, w, w, 1)
    with pytest.raises(ValueError):
        D.cross_backward(x, x, w, torch.zeros(shape[0]), x)
