"""Evictions whose shards are rebuilt instead of repaired run by run: keys without a row (their insert met a full shard)."""
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
