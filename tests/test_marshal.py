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


@pytest.mark.gpu
def test_out_of_memory_keeps_its_type():
    """Result arrays of 2^45 bytes: the allocator refuses, as for torch.empty."""
    N, lib = D.native()
    with pytest.raises(torch.OutOfMemoryError):
        torch.empty(1 << 43, device="cuda")
    with pytest.raises(torch.OutOfMemoryError):
        N.dense1_get(lib, None, 1 << 22, 1 << 21)


class _Pointer:
    """Memory that is no tensor: all a call needs is the address (and the length)."""

    def __init__(self, t):
        self.t = t

    def data_ptr(self):
        return self.t.data_ptr()

    def numel(self):
        return self.t.numel()


@pytest.mark.gpu
def test_objects_with_an_address(native):
    N, lib = native
    t = torch.zeros(8, dtype=torch.int32)
    assert N.write_rows(lib, None, _Pointer(t), None, None, None, None) == 1          # a closed table: INVALID_ARG
    assert N.write_rows(lib, None, t, _Pointer(t), t.untyped_storage(), None, None) == 1
    with pytest.raises(AttributeError):
        N.write_rows(lib, None, t, object(), None, None, None)
