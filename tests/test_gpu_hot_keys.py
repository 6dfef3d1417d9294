"""Keys that own a large part of a batch: the counts (whole batch, one occurrence in four, a sample), the replica rows, their
sums in the update or in a kernel of their own, and the keys counted instead of scattered.  Against sums in double."""
import pytest
import torch

pytestmark = pytest.mark.gpu


# (samples, fields, occurrences per bag, k, feature values): below and above the sizes at which the counting, the
# look-up of gradient rows and the replica sums change hands (2^17, 2^19, 2^20 occurrences; 8 per bag)
@pytest.mark.parametrize("B,F,n,k,vals", [(100, 3, 1, 8, False), (4000, 8, 4, 20, True), (8192, 16, 1, 16, False), (8193, 16, 1, 64, True),
                                          (9000, 30, 2, 32, False), (20000, 30, 2, 4, False), (3000, 40, 10, 64, False),
                                          (3000, 40, 10, 64, True), (2000, 100, 11, 60, False)])
def test_gradient_of_hot_keys(B, F, n, k, vals):
    from paper_1909_04823_b200 import binding as D
    g = torch.Generator(device="cuda").manual_seed(B + n)
    nnz = B * F * n
    t = D.Table(4, F, k, optimizer=D.OPT_SGD, lr=1.0, max_rows=nnz + 5000, seed=3, init_scale=0.0, max_nnz=nnz, max_batch=B)
    try:
        u = torch.rand(nnz, generator=g, device="cuda", dtype=torch.float64)
        ids = (u.pow(-1.5)).clamp(max=1e6).long() + 7          # a heavy head: the first key owns a quarter of the batch
        x = torch.rand(nnz, generator=g, device="cuda") + 0.5 if vals else None
        db = D.DeviceBatch(torch.arange(B * F + 1, device="cuda") * n, ids, x, B)
        t.find_or_insert(db)
        U = int(db.n_uniq)
        ops = D.OP_LR | D.OP_FM | D.OP_POOL
        out = torch.randn(B, k + 4, generator=g, device="cuda")
        gL, gF = torch.randn(B, generator=g, device="cuda"), torch.randn(B, generator=g, device="cuda")
        gE = torch.randn(B, F * k, generator=g, device="cuda")
        for again in range(2):      # the second backward over the same batch starts from clean buffers and kept counts
            rows = db.uniq_rows[:U].clone()
            zero = torch.zeros(U, k, device="cuda")
            t.write_rows(rows, zero, zero[:, 0].contiguous())
            t.backward_update(ops, db, out, torch.empty(B, F * k, device="cuda"), None, gL, gF, gE)
            got = t.read_rows(rows)
            # v = 0 and w = 0 before the step, lr = 1: the row is minus the summed gradient
            bag = torch.arange(B * F, device="cuda").repeat_interleave(n)
            xx = torch.ones(nnz, device="cuda", dtype=torch.float64) if x is None else x.double()
            c = (gF[:, None] * out[:, :k])[:, None, :].double() + gE.view(B, F, k).double()
            idx = db.uidx[:nnz].long()
            G = torch.zeros(U, k, dtype=torch.float64, device="cuda")
            S = torch.zeros(U, k, dtype=torch.float64, device="cuda")
            cb = c.reshape(B * F, k)
            for lo in range(0, nnz, 1 << 18):
                sl = slice(lo, lo + (1 << 18))
                term = cb[bag[sl]] * xx[sl, None]
                G.index_add_(0, idx[sl], term)
                S.index_add_(0, idx[sl], term.abs())
            Gw = torch.zeros(U, dtype=torch.float64, device="cuda").index_add_(0, idx, gL.double()[bag // F] * xx)
            Sw = torch.zeros(U, dtype=torch.float64, device="cuda").index_add_(0, idx, (gL.double()[bag // F] * xx).abs())
            # float32 chains of a few hundred terms at most, combined in double: the bound of the parity harness
            for got_, ref, absum, what in ((got["emb"], -G, S, "v"), (got["lin"], -Gw, Sw, "w")):
                err = (got_.double() - ref).abs()
                assert bool((err <= 1e-5 * ref.abs() + 1e-6 + 2e-7 * absum).all()), (what, float((err / (1e-6 + absum)).max()))
        assert t.status() == 0
    finally:
        t.close()
