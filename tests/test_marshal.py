"""What the marshalling extension takes and refuses: the same objects, and the same exceptions, as the ctypes calls of the
other entry points."""
import ctypes as C

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


class _Own(D.DeviceBatch):
    """A batch that builds its own struct."""
    made = 0

    def c(self):
        self.made += 1
        return super().c()


class _Bare:
    def __init__(self, db):
        self.db = db

    def c(self):
        return self.db.c()


@pytest.mark.gpu
def test_batches_that_build_their_own_struct(native):
    N, lib = native
    off, ids = torch.zeros(4, dtype=torch.int32), torch.zeros(3, dtype=torch.int64)
    db = _Own(off, ids, None, 1, device="cpu")
    assert N.find_or_insert(lib, None, db, True) == 1 and db.made == 1
    assert N.find_or_insert(lib, None, _Bare(db), True) == 1 and db.made == 2
    assert N.find_or_insert(lib, None, D.DeviceBatch(off, ids, None, 1, device="cpu"), True) == 1


@pytest.mark.gpu
def test_batch_struct_is_read_as_c():
    """The same step from a batch of the class itself and from one that builds its own struct."""
    res = []
    for cls in (D.DeviceBatch, _Own):
        t = D.Table(2, 3, 8, max_rows=1000, seed=1, max_nnz=64, max_batch=8)
        try:
            off = torch.arange(0, 13, dtype=torch.int32)
            db = cls(off, torch.arange(12) % 7 + 1, torch.arange(12) + 0.5, 4)
            t.find_or_insert(db)
            out = torch.zeros(4, 12, device="cuda")
            t.forward_fused(D.OP_LR | D.OP_FM, db, out_small=out)
            res.append((db.rows.clone(), db.uidx.clone(), db.n_uniq.clone(), out))
        finally:
            t.close()
    assert all(torch.equal(a, b) for a, b in zip(*res))


@pytest.mark.gpu
def test_head_converts_its_numbers(native):
    t = object.__new__(D.Table)
    t.N, t._lib = native
    t.h = C.c_void_p()
    for b in (4, 4.0, torch.tensor(4)):
        with pytest.raises(D.DesError) as e:                # a closed table, not a TypeError
            t.head(D.OP_LR, b, dict(b0="0.5", c_lr=torch.tensor(1.0), c_fm=1, u=None, b1=None, q=None, d=None))
        assert e.value.code == 1
