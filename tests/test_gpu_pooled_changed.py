"""Between des_forward_partials and des_aggregate the pooled block is the caller's: the first layer's product is of what it holds
then (a dropout mask, a sum over processes), in an eager call and in a captured one."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _product(pooled, W1):
    """(operands rounded to bfloat16, in double; the sum of the terms' sizes)"""
    a, w = pooled.bfloat16().double(), W1.bfloat16().double()
    return a @ w, a.abs() @ w.abs()


# HASH (pool_kernel), FIELD in one kernel per sample, FIELD with samples too large for that, extents the tensor cores do not take
@pytest.mark.parametrize("partition,F,k,H", [(0, 6, 16, 64), (1, 6, 16, 64), (1, 200, 64, 64), (0, 5, 12, 20)])
@pytest.mark.parametrize("captured", [False, True])
def test_product_of_the_changed_block(partition, F, k, H, captured):
    from paper_1909_04823_b200 import binding as D
    g = torch.Generator(device="cuda").manual_seed(F + k)
    B, n, S = 130, 2, 3
    t = D.Table(S, F, k, H, partition, max_rows=60 * F + 200, rows_per_shard=[60 * F + 200] * S, seed=2, init_scale=0.5,
                max_nnz=B * F * n, max_batch=B)
    try:
        W1 = torch.randn(F * k, H, generator=g, device="cuda")
        t.dense1_set(W1)
        ids = torch.randint(0, 50, (B * F * n,), generator=g, device="cuda") + torch.arange(B * F * n, device="cuda") // n % F * 1000 + 1
        db = D.DeviceBatch(torch.arange(B * F + 1, device="cuda") * n, ids, None, B)
        t.find_or_insert(db)
        ops = D.OP_LR | D.OP_POOL | D.OP_DENSE1
        part, pooled = torch.zeros(S, B, k + 4, device="cuda"), torch.zeros(B, F * k, device="cuda")
        out, Z = torch.zeros(B, k + 4, device="cuda"), torch.zeros(B, H, device="cuda")
        aggregate = lambda: t.aggregate(ops, db, part, pooled, out_small=out, Z=Z)
        aggregate()                                        # (allocations and attributes of a first call)
        t.forward_partials(ops, db, part, pooled)
        gr = torch.cuda.CUDAGraph()
        if captured:
            torch.cuda.synchronize()
            with torch.cuda.graph(gr):
                aggregate()
        for step in range(2):
            pooled.mul_((torch.rand(B, F * k, generator=g, device="cuda") < 0.5) * 2.0)
            gr.replay() if captured else aggregate()
            ref, size = _product(pooled, W1)
            assert bool(((Z.double() - ref).abs() <= 1e-5 * size + 1e-6).all()), step      # float32 sums of up to 12800 products
            t.forward_partials(ops, db, part, pooled)
        # and the fused form, whose product follows in the same call
        t.forward_fused(ops, db, pooled=pooled, out_small=out, Z=Z)
        ref, size = _product(pooled, W1)
        assert bool(((Z.double() - ref).abs() <= 1e-5 * size + 1e-6).all())
        assert t.status() == 0
    finally:
        t.close()
