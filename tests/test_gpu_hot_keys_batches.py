"""The hot-key counts belong to the batch whose backward is running, whatever the table has seen in between: a captured backward
replayed after another batch, a captured step replayed before an eager backward, and index arrays put back into
buffers that held another batch.  Against sums in double."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _ids(g, nnz, most):
    u = torch.rand(nnz, generator=g, device="cuda", dtype=torch.float64)
    return u.pow(-1.5).clamp(max=most).long() + 7           # a heavy head: the first key owns a quarter of the batch


class _Step:
    """A batch with its own buffers and upstream gradients, and the sums its backward has to arrive at."""

    def __init__(self, D, t, g, B, F, n, k, most):
        self.t, self.shape = t, (B, F, n, k)
        self.db = D.DeviceBatch(torch.arange(B * F + 1, device="cuda") * n, _ids(g, B * F * n, most), None, B)
        self.ops = D.OP_LR | D.OP_FM | D.OP_POOL
        self.out = torch.randn(B, k + 4, generator=g, device="cuda")
        self.gL, self.gF = torch.randn(B, generator=g, device="cuda"), torch.randn(B, generator=g, device="cuda")
        self.gE = torch.randn(B, F * k, generator=g, device="cuda")
        self.pooled = torch.empty(B, F * k, device="cuda")

    def insert(self):
        self.t.find_or_insert(self.db)

    def backward(self):
        self.t.backward_update(self.ops, self.db, self.out, self.pooled, None, self.gL, self.gF, self.gE)

    def clear(self):
        """v = 0 and w = 0 before the step, lr = 1: afterwards the rows are minus the summed gradients."""
        self.U = int(self.db.n_uniq)
        self.rows = self.db.uniq_rows[:self.U].clone()
        zero = torch.zeros(self.U, self.shape[3], device="cuda")
        self.t.write_rows(self.rows, zero, zero[:, 0].contiguous())

    def check(self, what):
        B, F, n, k = self.shape
        got = self.t.read_rows(self.rows)
        idx = self.db.uidx[:B * F * n].long()
        bag = torch.arange(B * F, device="cuda").repeat_interleave(n)
        c = ((self.gF[:, None] * self.out[:, :k])[:, None, :].double() + self.gE.view(B, F, k).double()).reshape(B * F, k)
        z = lambda *s: torch.zeros(*s, dtype=torch.float64, device="cuda")
        G, S = z(self.U, k).index_add_(0, idx, c[bag]), z(self.U, k).index_add_(0, idx, c[bag].abs())
        w = self.gL.double()[bag // F]
        Gw, Sw = z(self.U).index_add_(0, idx, w), z(self.U).index_add_(0, idx, w.abs())
        # float32 chains of a few hundred terms at most, combined in double: the bound of the parity harness
        for a, ref, absum, name in ((got["emb"], -G, S, "v"), (got["lin"], -Gw, Sw, "w")):
            err = (a.double() - ref).abs()
            assert bool((err <= 1e-5 * ref.abs() + 1e-6 + 2e-7 * absum).all()), (what, name, float((err / (1e-6 + absum)).max()))


@pytest.mark.parametrize("B,F,n,k", [(3000, 8, 4, 20), (9000, 30, 2, 32)])   # below and above 2^19 occurrences
@pytest.mark.parametrize("how", ["captured backward", "captured step", "arrays put back"])
def test_counts_of_the_running_batch(B, F, n, k, how):
    from paper_1909_04823_b200 import binding as D
    g = torch.Generator(device="cuda").manual_seed(B + k)
    t = D.Table(4, F, k, optimizer=D.OPT_SGD, lr=1.0, max_rows=B * F * n + 5000, seed=3, init_scale=0.0, max_nnz=B * F * n, max_batch=B)
    try:
        a = _Step(D, t, g, B, F, n, k, 1e6)
        b = _Step(D, t, g, B, F, n, k, 40)                  # the other batch: few keys, nearly all of them hot
        a.insert(); b.insert()                              # (all keys of both have rows)
        gr = torch.cuda.CUDAGraph()
        if how == "captured backward":
            a.insert()
            torch.cuda.synchronize()
            with torch.cuda.graph(gr):
                a.backward()
            for other in (b, a):                            # the graph after the other batch, then after its own
                other.insert()
                a.clear()
                gr.replay()
                a.check((how, other is b))
        elif how == "captured step":
            torch.cuda.synchronize()
            with torch.cuda.graph(gr):
                b.insert(); b.backward()
            a.insert()
            gr.replay()
            a.clear()
            a.backward()
            a.check(how)
        else:
            a.insert()
            held = ("rows", "shards", "uidx", "uniq_rows", "n_uniq", "ids")
            save = {x: getattr(a.db, x).clone() for x in held}
            a.db.ids.copy_(b.db.ids)
            a.insert()                                      # the same buffers, another batch
            for x in held:
                getattr(a.db, x).copy_(save[x])
            a.clear()
            a.backward()
            a.check(how)
        for s in (b, a):                                    # and nothing is left behind for later steps
            s.insert(); s.clear(); s.backward(); s.check((how, "after"))
        assert t.status() == 0
    finally:
        t.close()
