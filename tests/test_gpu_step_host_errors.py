"""A host step that is refused leaves the caller's buffers alone: nothing is copied into them behind the error, and the next
step of the same slot is right."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


# out_small of 32 KB (read back on the caller's stream) and of 512 KB (beside the backward)
@pytest.mark.parametrize("B", [256, 4096])
@pytest.mark.parametrize("submit", [False, True])
@pytest.mark.parametrize("missing", ["gL", "gF", "gE", "d_pooled", "ops"])
def test_refused_step_touches_nothing(B, submit, missing):
    from paper_1909_04823_b200 import binding as D
    F, k = 4, 28
    rng = np.random.default_rng(B)
    ops = D.OP_LR | D.OP_FM | D.OP_POOL
    t = D.Table(3, F, k, optimizer=D.OPT_SGD, max_rows=4000, seed=5, init_scale=0.05, max_nnz=B * F, max_batch=B)
    try:
        off = torch.arange(B * F + 1, dtype=torch.int32).pin_memory()
        ids = torch.from_numpy(rng.integers(1, 500, B * F)).pin_memory()
        out = torch.full((B, k + 4), 7.0).pin_memory()
        kw = dict(d_pooled=torch.zeros(B, F * k, device="cuda"), gL=torch.zeros(B, device="cuda"), gF=torch.zeros(B, device="cuda"),
                  gE=torch.zeros(B, F * k, device="cuda"))
        call = t.step_host_submit if submit else t.step_host
        torch.cuda.synchronize()
        with pytest.raises(D.DesError) as e:
            if missing == "ops":
                call(16 | ops, B, B * F, off, ids, None, out, **kw)
            else:
                call(ops, B, B * F, off, ids, None, out, **dict(kw, **{missing: None}))
        assert e.value.code == 1
        torch.cuda.synchronize()
        assert bool((out == 7.0).all())
        ticket = call(ops, B, B * F, off, ids, None, out, **kw)      # zero gradients: the weights stay what they were
        if submit:
            t.step_host_wait(ticket)
        db = D.DeviceBatch(off, ids, None, B)
        t.find_or_insert(db, insert=False)
        ref = torch.zeros(B, k + 4, device="cuda")
        t.forward_fused(ops | D.FUSED_SHARD_ORDER, db, pooled=kw["d_pooled"], out_small=ref)
        # (the update writes each row's cached squared norm anew: one rounding of a sum of 28 squares below 0.0025)
        assert torch.allclose(out, ref.cpu(), rtol=1e-6, atol=1e-6)
        assert t.status() == 0
    finally:
        t.close()
