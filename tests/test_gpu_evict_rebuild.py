"""Evictions whose shards are rebuilt instead of repaired run by run: runs of occupied slots too long for one thread, keys without
a row (their insert met a full shard), and a rebuild whose memory is not to be had."""
import pytest
import torch

from test_gpu_evict_repair import _batch, _contents

pytestmark = pytest.mark.gpu


def _table(D, shards, rows, load, most):
    return D.Table(shards, 1, 8, optimizer=D.OPT_ADAGRAD, init_acc=0.5, max_rows=rows * shards, rows_per_shard=[rows] * shards,
                   max_load=load, seed=7, max_nnz=most, max_batch=most)


def _some_ids(seed, n):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randint(-2 ** 62, 2 ** 62, (n,), generator=g, device="cuda")


def _check(D, t, ids, gone, found0, emb0):
    """The keys of mask `gone` are out, the others are what they were, rows are 0 .. n_s - 1."""
    found, emb, rows = _contents(D, t, ids)
    assert torch.equal(found, found0 & ~gone)
    assert torch.equal(emb[found], emb0[found])
    base = t.row_base()
    for s, m in enumerate(t.size()):
        mine = rows[found][(rows[found] >= base[s]) & (rows[found] < base[s + 1])] - base[s]
        assert torch.equal(torch.sort(mine).values, torch.arange(m, device="cuda", dtype=mine.dtype))


# full at load 0.9 a region of 200 k slots has runs of a thousand and more, one of 2 k some of hundreds.  In the checking build a
# run of 64 slots is a long one: all shards of the first cases are rebuilt, some of the last one
@pytest.mark.parametrize("shards,rows,load", [(1, 200_000, 0.9), (3, 60_000, 0.9), (8, 1800, 0.9), (40, 1500, 0.6)])
@pytest.mark.parametrize("share", [0.0005, 0.2])
@pytest.mark.parametrize("checking", [False, True])
def test_long_runs(shards, rows, load, share, checking):
    from paper_1909_04823_b200 import binding as D
    n = shards * rows
    prev = D.use_debug_library(checking)
    try:
        t = _table(D, shards, rows, load, n)
    finally:
        D.use_debug_library(prev)
    try:
        ids = _some_ids(n, n - 3 * shards * int(rows ** 0.5) if shards > 1 else n)
        t.find_or_insert(_batch(D, ids))
        assert t.status() == 0
        found0, emb0, _ = _contents(D, t, ids)
        assert bool(found0.all())
        gone = torch.zeros(ids.numel(), dtype=torch.bool, device="cuda")
        gone[torch.randperm(ids.numel(), device="cuda")[:max(1, int(ids.numel() * share))]] = True
        assert t.evict_keys(ids[gone]) == int(gone.sum())
        _check(D, t, ids, gone, found0, emb0)
        t.find_or_insert(_batch(D, ids))                   # back in, as new keys
        assert t.status() == 0 and bool(_contents(D, t, ids)[0].all())
    finally:
        t.close()


@pytest.mark.parametrize("seed", range(6))
def test_keys_without_a_row_are_dropped(seed):
    from paper_1909_04823_b200 import binding as D
    t = _table(D, 1, 200, 0.5, 1024)                       # 401 slots
    try:
        ids = _some_ids(seed, 600)
        t.find_or_insert(_batch(D, ids[:200]))
        t.find_or_insert(_batch(D, ids[200:390]))          # no rows left: 190 keys that hold a slot and nothing else
        assert t.status() == 3 and t.size() == [200]
        found0, emb0, _ = _contents(D, t, ids[:200])
        gone = torch.zeros(200, dtype=torch.bool, device="cuda")
        gone[17] = True
        assert t.evict_keys(ids[17:18]) == 1
        _check(D, t, ids[:200], gone, found0, emb0)
        t.find_or_insert(_batch(D, ids[390:590]))          # 200 keys find a slot each, and the first of them the row
        assert t.size() == [200]
        found, _, rows = _contents(D, t, ids[390:590])
        assert bool(found[0]) and int(found.sum()) == 1 and int(rows[0]) == 199
    finally:
        t.close()


def test_no_memory_for_a_rebuild_changes_nothing(monkeypatch):
    from paper_1909_04823_b200 import binding as D
    prev = D.use_debug_library(True)
    try:
        t = _table(D, 2, 300, 0.5, 2048)
        try:
            ids = _some_ids(1, 900)
            t.find_or_insert(_batch(D, ids))               # about 450 keys a shard for 300 rows
            assert t.status() == 3 and t.size() == [300, 300]
            found0, emb0, rows0 = _contents(D, t, ids)
            gone = torch.zeros(900, dtype=torch.bool, device="cuda")
            gone[torch.nonzero(found0)[::3, 0]] = True
            monkeypatch.setenv("DES_DEBUG_EVICT_NO_MEMORY", "1")
            with pytest.raises(D.DesError):
                t.evict_keys(ids[gone])
            found, emb, rows = _contents(D, t, ids)
            assert torch.equal(found, found0) and torch.equal(emb, emb0) and torch.equal(rows, rows0) and t.size() == [300, 300]
            monkeypatch.delenv("DES_DEBUG_EVICT_NO_MEMORY")
            assert t.evict_keys(ids[gone]) == int(gone.sum())
            _check(D, t, ids, gone, found0, emb0)
        finally:
            t.close()
    finally:
        D.use_debug_library(prev)
