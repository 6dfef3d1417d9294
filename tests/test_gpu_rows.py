"""Rows in and out of the table (des_table_read_rows / des_table_write_rows): every column group, ragged counts, dense
arrays that are not 16-byte aligned, repeated and missing rows.  Copies: the bits come back."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [4, 8, 12, 20, 32, 64])
@pytest.mark.parametrize("n", [1, 33, 127, 1025])
@pytest.mark.parametrize("shift", [0, 1])
def test_rows_round_trip(k, n, shift):
    from paper_1909_04823_b200 import binding as D
    t = D.Table(3, 2, k, optimizer=D.OPT_ADAGRAD, max_rows=3000, max_nnz=4096, max_batch=2048)
    try:
        ids = torch.arange(1, n + 1, dtype=torch.int64, device="cuda")
        off = (torch.arange(2 * n + 1, dtype=torch.int64, device="cuda") + 1) // 2      # one id per sample
        db = D.DeviceBatch(off, ids, None, n)
        t.find_or_insert(db)
        rows = db.uniq_rows[:n].clone()
        g = torch.Generator(device="cuda").manual_seed(k * 1000 + n)

        def dense(*shape):                      # `shift` floats past an allocation's start
            m = int(np.prod(shape))
            return torch.randn(m + shift, generator=g, device="cuda")[shift:].view(*shape)

        emb, lin, ae, al = dense(n, k), dense(n), dense(n, k), dense(n)
        t.write_rows(rows, emb, lin, ae, al)
        got = t.read_rows(rows)
        for name, want in (("emb", emb), ("lin", lin), ("acc_emb", ae), ("acc_lin", al)):
            assert torch.equal(got[name], want), name
        # the squared norm cached with a row is that of the row written: LR + FM of one-id samples
        part = torch.zeros(3, n, k + 4, device="cuda")
        t.forward_partials(D.OP_LR | D.OP_FM, db, part)
        m2 = part[:, :, k + 1].sum(0).double()
        assert torch.allclose(m2, (emb.double() ** 2).sum(1), rtol=1e-6, atol=0)     # k additions: k * 2^-24
        # repeated rows and "no row"
        pick = torch.randint(0, n, (n,), generator=g, device="cuda")
        some = rows[pick].clone()
        some[::3] = -1
        got = t.read_rows(some)
        want = emb[pick].clone()
        want[::3] = 0
        assert torch.equal(got["emb"], want) and t.status() == 0
    finally:
        t.close()
