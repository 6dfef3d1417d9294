"""The backward with a first layer, part of which runs beside the rest on a stream of the table's own: the same results as with its
launches one after the other (as they run while they are being timed), step after step, and replayed from a captured graph."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,F,k,H,optimizer", [(64, 5, 8, 16, "adam"), (777, 39, 32, 400, "adagrad"), (14000, 39, 16, 136, "sgd"),
                                               (3000, 11, 12, 20, "adam")])   # (the last: H not a multiple of 8)
def test_same_as_in_order(B, F, k, H, optimizer):
    from paper_1909_04823_b200 import binding as D
    opt = {"adam": D.OPT_ADAM, "adagrad": D.OPT_ADAGRAD, "sgd": D.OPT_SGD}[optimizer]
    g = torch.Generator(device="cuda").manual_seed(B)
    rn = lambda *s: torch.randn(*s, generator=g, device="cuda")
    ids = [torch.rand(B * F, generator=g, device="cuda").pow(4).mul(3000).long() * F + torch.arange(F, device="cuda").repeat(B) for _ in range(4)]
    W1, off = rn(F * k, H) / 8, torch.arange(B * F + 1, device="cuda")
    grads = [(rn(B), rn(B), rn(B, F * k), rn(B, H)) for _ in range(4)]
    ops = D.OP_LR | D.OP_FM | D.OP_POOL | D.OP_DENSE1
    got = {}
    for how in ("in order", "beside", "captured"):
        t = D.Table(3, F, k, hidden=H, partition=D.PART_FIELD, optimizer=opt, max_rows=3100 * F, rows_per_shard=[3100 * F] * 3, seed=3,
                    init_acc=0.1, max_nnz=B * F, max_batch=B)
        try:
            t.dense1_set(W1)
            t.profile_enable(how == "in order")
            bufs = dict(pooled=torch.zeros(B, F * k, device="cuda"), out_small=torch.zeros(B, k + 4, device="cuda"), Z=torch.zeros(B, H, device="cuda"))
            work = torch.zeros(B, F * k, device="cuda")
            db = D.DeviceBatch(off, ids[0].clone(), None, B)
            cur = [x.clone() for x in grads[0]]

            def step():
                t.find_or_insert(db)
                t.forward_fused(ops, db, **bufs)
                t.backward_update(ops, db, bufs["out_small"], bufs["pooled"], bufs["Z"], *cur, work)

            graph, works = None, []
            for i in range(4):
                db.ids.copy_(ids[i])
                for a, b in zip(cur, grads[i]):
                    a.copy_(b)
                if how == "captured" and i == 1:
                    torch.cuda.synchronize()
                    graph = torch.cuda.CUDAGraph()
                    with torch.cuda.graph(graph):
                        step()
                graph.replay() if graph else step()
                works.append(work.clone())
            n = int(db.n_uniq)
            got[how] = dict(t.read_rows(db.uniq_rows[:n]), W1=t.dense1_get(), work=torch.stack(works))
            assert t.status() == 0
        finally:
            t.close()
    for how in ("beside", "captured"):
        for name, a in got["in order"].items():
            b = got[how][name]
            # (float32 atomics in another order; the step of a rounding-sized gradient under Adagrad / Adam; bfloat16 weights one bit apart)
            err = float((a - b).double().norm() / (a.double().norm() + 1e-30))
            assert err < 2e-3, (how, name, err)
