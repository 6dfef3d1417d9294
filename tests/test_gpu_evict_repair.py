"""Eviction repairs the runs of occupied slots in place: crowded regions (load 0.9), wrap-around, one shard and many, and
a region without a single empty slot (filled up by inserts that found no row), which is rebuilt instead."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _batch(D, ids):
    n = ids.numel()
    return D.DeviceBatch(torch.arange(n + 1, device="cuda"), ids, None, n)


def _contents(D, t, ids):
    """(found mask, latent vector) of each id."""
    db = _batch(D, ids)
    t.find_or_insert(db, insert=False)
    base = torch.tensor(t.row_base(), device="cuda")
    found = db.rows[:ids.numel()] != -1
    rows = torch.where(found, base[db.shards[:ids.numel()].long()] + db.rows[:ids.numel()].long(), -1).to(torch.int32)
    return found, t.read_rows(rows)["emb"], rows


@pytest.mark.parametrize("shards", [1, 3, 64])
@pytest.mark.parametrize("n", [5, 400, 5000])
@pytest.mark.parametrize("share", [0.02, 0.5, 1.0])
def test_runs_are_repaired(shards, n, share):
    from paper_1909_04823_b200 import binding as D
    per = [int(n / shards * 1.3) + 8] * shards
    t = D.Table(shards, 1, 8, optimizer=D.OPT_SGD, max_rows=sum(per), rows_per_shard=per, max_load=0.9, seed=7, max_nnz=8192,
                max_batch=8192)
    try:
        g = torch.Generator(device="cuda").manual_seed(n + shards)
        ids = torch.randint(-2 ** 62, 2 ** 62, (n,), generator=g, device="cuda")
        t.find_or_insert(_batch(D, ids))
        assert t.status() in (0, 3)
        found0, emb0, _ = _contents(D, t, ids)
        order = torch.randperm(n, generator=g, device="cuda")
        gone = ids[order[:max(1, int(n * share))]]
        twice = torch.cat([gone, gone[:gone.numel() // 2], torch.tensor([12345], device="cuda")])
        before = sum(t.size())
        mask = torch.zeros(n, dtype=torch.bool, device="cuda")
        mask[order[:gone.numel()]] = True
        assert t.evict_keys(twice) == int((mask & found0).sum())
        assert sum(t.size()) == before - int((mask & found0).sum())
        found, emb, rows = _contents(D, t, ids)
        assert torch.equal(found, found0 & ~mask)
        assert torch.equal(emb[found], emb0[found])
        # rows of a shard are still 0 .. n_s - 1, each once
        base = t.row_base()
        for s, m in enumerate(t.size()):
            mine = rows[found][(rows[found] >= base[s]) & (rows[found] < base[s + 1])] - base[s]
            assert torch.equal(torch.sort(mine).values, torch.arange(m, device="cuda", dtype=mine.dtype))
        # and again, by age: everything that is left was inserted at clock 1
        left = sum(t.size())
        assert t.evict_stale(2) == left and sum(t.size()) == 0
        assert not _contents(D, t, ids)[0].any()
    finally:
        t.close()


@pytest.mark.parametrize("gone", [1, 7])
def test_full_region_is_rebuilt(gone):
    from paper_1909_04823_b200 import binding as D
    t = D.Table(1, 1, 8, optimizer=D.OPT_SGD, max_rows=100, rows_per_shard=[100], max_load=0.9, seed=7, max_nnz=1024, max_batch=1024)
    try:
        g = torch.Generator(device="cuda").manual_seed(3)
        ids = torch.randint(-2 ** 62, 2 ** 62, (300,), generator=g, device="cuda")
        t.find_or_insert(_batch(D, ids))                   # 100 rows, 112 slots: the rest finds no row or no slot
        assert t.status() == 3 and t.size() == [100]
        found0, emb0, _ = _contents(D, t, ids)
        assert int(found0.sum()) == 100
        out = ids[found0][:gone]
        assert t.evict_keys(out) == gone and t.size() == [100 - gone]
        found, emb, _ = _contents(D, t, ids)
        assert not found[found0][:gone].any() and found[found0][gone:].all() and int(found.sum()) == 100 - gone
        assert torch.equal(emb[found], emb0[found])
        t.find_or_insert(_batch(D, out))                   # there is room again
        assert t.size() == [100] and _contents(D, t, out)[0].all()
    finally:
        t.close()
