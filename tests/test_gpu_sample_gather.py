"""The gather that keeps a sample's bags together (fused forward; FIELD partition with per-shard partials): one to eight warps
per sample, more fields than lane groups, empty bags, missing keys, feature values, samples too large for shared
memory.  Against sums in double of the rows the table holds."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _setup(D, B, F, k, S, partition, mean, vals, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    lens = torch.poisson(torch.full((B * F,), float(mean), device="cuda"), generator=g).long()
    off = torch.zeros(B * F + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(lens, 0)
    nnz = int(off[-1])
    bag = torch.repeat_interleave(torch.arange(B * F, device="cuda"), lens)
    ids = torch.randint(0, 500, (nnz,), generator=g, device="cuda") + (bag % F + 1) * 1000
    x = torch.rand(nnz, generator=g, device="cuda") + 0.5 if vals else None
    known = ids[torch.rand(nnz, generator=g, device="cuda") < 0.9]       # the others look up as "no row"
    t = D.Table(S, F, k, partition=partition, max_rows=500 * F + 1000, rows_per_shard=[500 * F + 8] * S, seed=3,
                init_scale=0.1, max_nnz=nnz + 64, max_batch=B)
    db = D.DeviceBatch(off, ids, x, B)
    keep = torch.isin(ids, known)
    lens2 = torch.zeros(B * F, dtype=torch.int64, device="cuda").index_add_(0, bag, keep.long())
    off2 = torch.zeros(B * F + 1, dtype=torch.int64, device="cuda")
    off2[1:] = torch.cumsum(lens2, 0)
    first = D.DeviceBatch(off2, ids[keep], None, B)
    t.find_or_insert(first)
    base = torch.tensor(t.row_base(), device="cuda")
    n = int(first.n_uniq)
    t.write_rows(first.uniq_rows[:n], lin=torch.randn(n, generator=g, device="cuda"))
    t.find_or_insert(db, insert=False)
    found = db.rows[:nnz] != -1
    rows = torch.where(found, base[db.shards[:nnz].long()] + db.rows[:nnz].long(), -1).to(torch.int32)
    r = t.read_rows(rows)
    xx = torch.ones(nnz, device="cuda", dtype=torch.float64) if x is None else x.double()
    v, w = r["emb"].double() * xx[:, None], r["lin"].double() * xx
    return t, db, bag, v, w, nnz


@pytest.mark.parametrize("B,F,k,S,partition,mean,vals", [
    (1, 1, 4, 1, 1, 1, False), (48, 39, 32, 16, 1, 1, False), (700, 8, 8, 4, 0, 2, True), (1300, 39, 16, 5, 1, 1, True),
    (2500, 40, 20, 7, 1, 1, False), (5000, 26, 16, 8, 1, 1, False), (33, 100, 64, 64, 0, 20, False), (5000, 3, 64, 3, 0, 12, True),
    (20, 400, 64, 9, 1, 1, False),
    # about the largest sample whose pooled vectors a block holds, and the sizes behind it
    *[(20, F, 64, 9, 1, 1, False) for F in (182, 183, 185, 186, 187)], (20, 360, 32, 7, 1, 1, True), (20, 361, 32, 7, 1, 1, False),
    (20, 682, 16, 5, 1, 1, False),
    # long bags under FIELD: a warp per bag
    (300, 20, 64, 7, 1, 12, False), (40, 30, 16, 4, 1, 20, True), (2500, 8, 32, 8, 1, 10, True)])
def test_sums_of_a_sample(B, F, k, S, partition, mean, vals):
    from paper_1909_04823_b200 import binding as D
    t, db, bag, v, w, nnz = _setup(D, B, F, k, S, partition, mean, vals, B + F)
    try:
        ops = D.OP_LR | D.OP_FM | D.OP_POOL
        samp = bag // F
        z = lambda *s: torch.zeros(*s, dtype=torch.float64, device="cuda")
        pooled = z(B * F, k).index_add_(0, bag, v)
        pabs = z(B * F, k).index_add_(0, bag, v.abs())
        A, Aabs = z(B, k).index_add_(0, samp, v), z(B, k).index_add_(0, samp, v.abs())
        R, Rabs = z(B).index_add_(0, samp, w), z(B).index_add_(0, samp, w.abs())
        Q = z(B).index_add_(0, samp, (v * v).sum(1))

        def close(got, ref, absum, what):             # float32 sums of a few dozen terms at most per accumulator
            err = (got.double() - ref).abs()
            assert bool((err <= 1e-6 * ref.abs() + 2e-6 * absum + 1e-12).all()), (what, float(err.max()))

        for form in ("fused", "two"):
            out, pl = torch.full((B, k + 4), 9.0, device="cuda"), torch.full((B, F * k), 9.0, device="cuda")
            if form == "fused":
                t.forward_fused(ops, db, pooled=pl, out_small=out)
            else:
                part = torch.full((S, B, k + 4), 9.0, device="cuda")
                t.forward_partials(ops, db, part, pl)
                t.aggregate(ops, db, part, pl, out_small=out)
            close(pl.view(B * F, k), pooled, pabs, "pooled")
            close(out[:, :k], A, Aabs, "A")
            close(out[:, k], R, Rabs, "R")
            close(out[:, k + 2], Q, Q, "Q")
            close(out[:, k + 1], 0.5 * (A * A).sum(1) - 0.5 * Q, (A.abs() * Aabs).sum(1) + Q, "F")
            assert bool((out[:, k + 3] == 0).all())
        if partition == 1:
            f = bag % F
            for s in range(min(S, F)):
                m = f % S == s
                ref = z(B, k).index_add_(0, samp[m], v[m])
                close(part[s][:, :k], ref, z(B, k).index_add_(0, samp[m], v[m].abs()), ("M_1", s))
        out2, part2 = torch.zeros_like(out), torch.zeros_like(part)
        t.forward_fused(ops, db, part2, pooled=pl, out_small=out2)          # both at once: the two-call path's bits
        assert torch.equal(part2, part) and torch.equal(out2, out)
        assert t.status() == 0
    finally:
        t.close()
