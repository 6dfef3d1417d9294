"""Performance cases: what a user of the library has it do, through its public entry points.

A case is a plain dict.  `listed()` names the fixed ones, `draw(rng)` makes one more of the same ranges,
`prepare(case, seed)` builds what a program holds before the call (table, batch, upstream gradients, buffers),
`run(state)` is one pass, `work(case)` the bytes and operations of a pass, `tolerance(case)` how far two correct
implementations may differ.

Kinds of pass:
  step     one training step: find-or-insert, per-shard partials, aggregation, (read-out and loss,) backward and
           update, then the pull of the batch's updated rows that a program makes to publish or store them.  With
           `fused` the forward is the one-call form.
  stream   a training step on a table that grows: a share of the ids was never seen before, and the same number
           of keys is evicted afterwards, which is what keeps such a table inside its memory.
  serve    prediction with a trained table: look-up without insertion, fused forward.
  host     two training steps whose batches start in pinned host memory, both in flight, results read back.
  cross    the DCN cross layer, forward and backward.

Ids follow a Zipf law (by rank, inverse of the continuous hat), as click logs do; bag lengths, field counts,
dimensions, shard counts and optimizers are those of the workloads in `paper_1909_04823_b200.synth`, with tables
scaled so that several fit one GPU.  Tables are populated before the pass: training meets mostly known keys."""
import math

import numpy as np
import torch

from paper_1909_04823_b200 import binding as D

LR, FM, POOL, DENSE1 = D.OP_LR, D.OP_FM, D.OP_POOL, D.OP_DENSE1
OPS = {"lr+fm": LR | FM, "lr+pool+dense1": LR | POOL | DENSE1, "lr+fm+pool": LR | FM | POOL,
       "lr+fm+pool+dense1": LR | FM | POOL | DENSE1}
OPTIMIZERS = {"sgd": D.OPT_SGD, "adagrad": D.OPT_ADAGRAD, "adam": D.OPT_ADAM}
MAX_LEN = 100                     # cap of the geometric bag lengths


def _case(kind, batch, fields, dim, shards, ops, **kw):
    c = dict(kind=kind, batch=batch, fields=fields, dim=dim, shards=shards, ops=ops, partition="hash", optimizer="adagrad",
             ftrl=False, hidden=0, law="onehot", mean=1.0, zipf=1.1, keys=100_000, buckets=0, vals=False, head=False,
             fused=False)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest training step: a toy LR + FM model, bags of 1-4 ids, plain SGD (latency and launches)
        _case("step", 512, 8, 8, 4, "lr+fm", name="tiny_lr_fm", optimizer="sgd", law="uniform", mean=2.5, keys=100_000),
        # Wide & Deep on Criteo-like one-hot fields, closed loop: read-out and log loss supply the gradients
        _case("step", 8192, 26, 16, 8, "lr+pool+dense1", name="wide_deep_loop", partition="field", hidden=256, zipf=1.05,
              keys=26_000_000, head=True),
        # DeepFM on 13 bucketised + 26 categorical fields, gradients from the rest of the model
        _case("step", 16384, 39, 32, 16, "lr+fm+pool+dense1", name="deepfm", partition="field", hidden=400, buckets=13,
              keys=26_000_000),
        # a small online-learning step of the same model, odd batch, read-out in the loop, one-call forward
        _case("step", 777, 39, 32, 16, "lr+fm+pool+dense1", name="deepfm_online", partition="field", hidden=400, buckets=13,
              keys=2_600_000, head=True, fused=True),
        # ragged bags with feature values, odd sizes, lazy Adam and FTRL for the linear weights
        _case("step", 3001, 17, 20, 7, "lr+fm+pool", name="ragged_adam_ftrl", optimizer="adam", ftrl=True, law="poisson",
              mean=4.0, keys=1_500_000, vals=True),
        # the large multi-hot workload: about 20 ids per bag, 100 fields, per-shard partials materialised
        _case("step", 16384, 100, 64, 64, "lr+fm+pool", name="multihot_large", law="geometric", mean=20.0, zipf=1.2,
              keys=40_000_000),
        # the same model at an ordinary batch, with the one-call forward
        _case("step", 1500, 100, 64, 64, "lr+fm+pool", name="multihot_fused", law="geometric", mean=20.0, zipf=1.2,
              keys=20_000_000, fused=True),
        # streaming features: 1/16 of the occurrences are new keys, evicted again when the step is over
        _case("stream", 32768, 30, 64, 32, "lr+fm+pool", name="streaming_evict", law="poisson", mean=4.0, keys=1_000_000),
        # prediction: a request of a few dozen candidates, and a large scoring batch
        _case("serve", 48, 39, 32, 16, "lr+fm+pool+dense1", name="serve_request", partition="field", hidden=400, buckets=13,
              keys=2_600_000, optimizer="sgd"),
        _case("serve", 4096, 100, 64, 64, "lr+fm+pool", name="serve_multihot", law="geometric", mean=20.0, zipf=1.2,
              keys=20_000_000, optimizer="sgd"),
        # batches that arrive in host memory
        _case("host", 16384, 30, 64, 32, "lr+fm+pool", name="host_steps", law="poisson", mean=4.0, keys=4_000_000),
        # DCN cross layer over the pooled vectors of the DeepFM fields
        dict(kind="cross", name="cross_layer", batch=16384, dim=1248, shards=16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "serve", "serve", "stream", "host", "cross"])
    if kind == "cross":
        return dict(kind="cross", batch=_log_int(rng, 64, 16384), dim=_log_int(rng, 64, 2048), shards=rng.randint(1, 32))
    criteo = kind in ("step", "serve") and rng.random() < 0.5      # one-hot fields with a first dense layer
    if criteo:
        buckets = rng.choice([0, 13])
        fields = buckets + rng.randint(20, 40)
        batch, dim = _log_int(rng, 32, 16384), 8 * rng.randint(1, 4)
        c = _case(kind, batch, fields, dim, rng.randint(2, 20), rng.choice(["lr+pool+dense1", "lr+fm+pool+dense1"]),
                  partition="field", hidden=8 * rng.randint(16, 50), buckets=buckets, zipf=round(rng.uniform(1.05, 1.2), 3))
    else:
        fields = _log_int(rng, 4, 100)
        law, mean = rng.choice([("uniform", 2.5), ("poisson", 4.0), ("geometric", 20.0)])
        batch = _log_int(rng, 64, 16384)
        batch = max(32, min(batch, int(8e6 / (fields * mean))))
        dim = 4 * rng.randint(2, 16)
        ops = rng.choice(["lr+fm", "lr+fm+pool"]) if kind != "stream" else "lr+fm+pool"
        c = _case(kind, batch, fields, dim, rng.randint(1, 64), ops, law=law, mean=mean, zipf=round(rng.uniform(1.05, 1.25), 3),
                  vals=kind in ("step", "serve") and law != "geometric" and rng.random() < 0.3)
    if kind == "serve":
        c["optimizer"] = "sgd"
    elif rng.random() < 0.3:
        c["optimizer"], c["ftrl"] = rng.choice([("sgd", False), ("adam", True), ("adagrad", True), ("adam", False)])
    c["head"] = kind == "step" and rng.random() < 0.3
    c["fused"] = kind == "step" and rng.random() < 0.3
    per_call = c["batch"] * c["fields"]
    top = min(1_000_000 if kind == "stream" else 10_000_000, 300 * per_call)
    c["keys"] = max(64 * c["fields"], _log_int(rng, max(1000, top // 50), max(2000, top)))
    return c


# ---- inputs -----------------------------------------------------------------------------------------------------
def _i64(v):
    return v - (1 << 64) if v >= 1 << 63 else v


def _fmix64(x):
    """Ranks to ids: a bijective 64-bit finaliser (int64 tensors; the shifts are logical)."""
    for mult in (0xFF51AFD7ED558CCD, 0xC4CEB9FE1A85EC53):
        x = x ^ ((x >> 33) & 0x7FFFFFFF)
        x = x * _i64(mult)
    return x ^ ((x >> 33) & 0x7FFFFFFF)


def _zipf_ranks(g, s, n, size):
    """`size` ranks 0..n-1 with P(r) about (r + 1)^-s: the continuous hat inverted and rounded."""
    a = 1.0 - s
    lo, hi = 0.5 ** a, (n + 0.5) ** a
    u = torch.rand(size, generator=g, device="cuda", dtype=torch.float64)
    return (lo + u * (hi - lo)).pow_(1.0 / a).add_(0.5).floor_().clamp_(1, n).to(torch.int64) - 1


def _lengths(c, g, nbags):
    """Bag lengths: the same multiset for every seed (a case's outputs have one shape), in the seed's own order."""
    law, mean = c["law"], c["mean"]
    if law == "onehot":
        return torch.ones(nbags, dtype=torch.int64, device="cuda")
    fixed = torch.Generator(device="cuda").manual_seed(17)
    if law == "uniform":
        lens = torch.randint(1, int(2 * mean), (nbags,), generator=fixed, device="cuda")
    elif law == "poisson":
        lens = torch.poisson(torch.full((nbags,), mean - 1.0, device="cuda"), generator=fixed).to(torch.int64) + 1
    else:
        u = torch.rand(nbags, generator=fixed, device="cuda", dtype=torch.float64)
        lens = (torch.log1p(-u) / math.log1p(-1.0 / mean)).floor().to(torch.int64).add_(1).clamp_(1, MAX_LEN)
    return lens[torch.randperm(nbags, generator=g, device="cuda")]


def _vocab(c):
    """Ids a field can draw, per field under FIELD (one vocabulary for all fields under HASH)."""
    return max(64, c["keys"] // (c["fields"] - c["buckets"])) if c["partition"] == "field" else c["keys"]


def _max_nnz(c):
    nbags = c["batch"] * c["fields"]
    return nbags if c["law"] == "onehot" else int(nbags * c["mean"] * (1.6 if c["law"] == "uniform" else 1.15)) + 8192


def _room_for_distinct(c):
    """Entries of the list of a batch's distinct keys that a program provides for (unused ones say "no row")."""
    u = _sizes(c)[1]
    return min(int(1.05 * u + 6.0 * math.sqrt(u)) + 16, _max_nnz(c))


def _batch(c, g, first_new=0):
    """(offsets, ids, vals, fresh) on the GPU; `fresh` = the ids of a stream batch that the table has not seen."""
    B, F = c["batch"], c["fields"]
    lens = _lengths(c, g, B * F)
    off = torch.zeros(B * F + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=off[1:])
    nnz = int(off[-1])
    # a served request meets some ids that training never saw
    vocab = int(_vocab(c) * 1.05) if c["kind"] == "serve" else _vocab(c)
    ranks = _zipf_ranks(g, c["zipf"], vocab, nnz)
    fresh = None
    if c["partition"] == "field":
        field = torch.repeat_interleave(torch.arange(F, device="cuda").repeat(B), lens)
        if c["buckets"]:
            x = torch.randn(nnz, generator=g, device="cuda")
            ranks = torch.where(field < c["buckets"], ((x + 4.0) * 8.0).floor().clamp_(0, 63).to(torch.int64), ranks)
        ids = _fmix64(((field + 1) << 40) | ranks)
    else:
        if c["kind"] == "stream":
            new = torch.rand(nnz, generator=g, device="cuda") < 1.0 / 16.0
            n = int(new.sum())
            ranks[new] = first_new + torch.arange(n, device="cuda")
            fresh = _fmix64(first_new + torch.arange(n, device="cuda"))
        ids = _fmix64(ranks)
    vals = torch.rand(nnz, generator=g, device="cuda") + 0.5 if c["vals"] else None
    return off.to(torch.int32), ids, vals, fresh


def _table(c):
    """The table a program of this case creates, populated with the vocabulary."""
    B, F, S, n = c["batch"], c["fields"], c["shards"], c["keys"]
    max_nnz = _max_nnz(c)
    room = n + (max_nnz // 12 if c["kind"] == "stream" else 0)
    per_shard = None
    if c["partition"] == "field":
        per_shard = [256 + sum(64 if f < c["buckets"] else _vocab(c) + 1 for f in range(s, F, S)) for s in range(S)]
        room = sum(per_shard)
    t = D.Table(S, F, c["dim"], c["hidden"], D.PART_FIELD if c["partition"] == "field" else D.PART_HASH,
                OPTIMIZERS[c["optimizer"]], max_rows=room, rows_per_shard=per_shard, seed=11, init_scale=0.01,
                init_acc=1e-8 if c["head"] else 0.1, max_nnz=max_nnz, max_batch=B,
                max_uniq=min(max_nnz, int(1.5 * _sizes(c)[1]) + 4096), lin_optimizer=D.LIN_FTRL if c["ftrl"] else D.LIN_SAME)
    if c["partition"] == "field":
        for lo in range(0, _vocab(c), B):
            m = min(B, _vocab(c) - lo)
            rank = torch.arange(lo, lo + m, device="cuda")[:, None].expand(m, F)
            if c["buckets"]:
                rank = torch.where(torch.arange(F, device="cuda") < c["buckets"], rank % 64, rank)
            ids = _fmix64(((torch.arange(F, device="cuda") + 1) << 40) | rank).reshape(-1)
            t.find_or_insert(D.DeviceBatch(torch.arange(m * F + 1, device="cuda"), ids, None, m))
    else:
        chunk = min(max_nnz, B * F)
        for lo in range(0, n, chunk):
            m = min(chunk, n - lo)
            off = torch.arange(B * F + 1, device="cuda").clamp_(max=m)
            t.find_or_insert(D.DeviceBatch(off, _fmix64(torch.arange(lo, lo + m, device="cuda")), None, B))
    if c["hidden"]:
        g = torch.Generator(device="cuda").manual_seed(3)
        t.dense1_set(torch.randn(F * c["dim"], c["hidden"], generator=g, device="cuda") / math.sqrt(F * c["dim"]))
    return t


def _randomise_linear(t, g):
    """Linear weights of a trained table (a new row starts at 0)."""
    base = t.row_base()
    for s, n in enumerate(t.size()):
        rows = torch.arange(base[s], base[s] + n, device="cuda").to(torch.int32)
        t.write_rows(rows, lin=torch.randn(n, generator=g, device="cuda") * 0.01)


def _earlier_step(s, db, normal):
    """One training step with other gradients: Adam's moments are those of a table in training (at its very first
    step a weight moves by the sign of its gradient)."""
    like = [None if x is None else normal(*x.shape) * float(x.std()) for x in (s.gL, s.gF, s.gE, s.gZ)]
    s.t.find_or_insert(db)
    s.t.forward_fused(s.ops, db, pooled=s.pooled, out_small=s.out_small, Z=s.Z)
    s.t.backward_update(s.ops, db, s.out_small, s.pooled, s.Z, *like, s.gE_work)


class _State:
    pass


def prepare(case, seed):
    c = case
    g = torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 62))
    s = _State()
    s.case, B = c, c["batch"]

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda")

    if c["kind"] == "cross":
        d = c["dim"]
        s.x0, s.x, s.gY = normal(B, d), normal(B, d), normal(B, d)
        s.w, s.b = normal(d) / math.sqrt(d), normal(d) * 0.1
        return s

    F, k, S, H = c["fields"], c["dim"], c["shards"], c["hidden"]
    s.ops = OPS[c["ops"]]
    s.t = _table(c)
    s.out_small = torch.zeros(B, k + 4, device="cuda")
    s.pooled = torch.zeros(B, F * k, device="cuda") if s.ops & POOL else None
    s.Z = torch.zeros(B, H, device="cuda") if H else None
    if c["kind"] == "serve":
        _randomise_linear(s.t, g)
        off, ids, vals, _ = _batch(c, g)
        s.db = D.DeviceBatch(off, ids, vals, B)
        return s

    # upstream gradients: unit normal (of a mean loss where nothing normalises them: plain SGD), or from the
    # read-out of the step itself
    scale = 1.0 / B if c["optimizer"] == "sgd" or c["head"] else 1.0
    s.gL = normal(B) * scale if s.ops & LR else None
    s.gF = normal(B) * scale if s.ops & FM else None
    s.gE = normal(B, F * k) * scale if s.ops & POOL else None
    s.gZ = normal(B, H) * scale if H else None
    s.gE_work = torch.zeros(B, F * k, device="cuda") if H else None
    if c["head"]:
        s.y = (torch.rand(B, generator=g, device="cuda") < 0.25).float()
        s.xdense = normal(B, 13)
        s.logit, s.loss = torch.zeros(B, device="cuda"), torch.zeros(B, device="cuda")
        s.hc = dict(b0=-1.0, c_lr=1.0, c_fm=0.5, u=normal(H) / math.sqrt(H) if H else None, b1=0.1 * normal(H) if H else None,
                    q=None if H or s.pooled is None else normal(F * k) / math.sqrt(F * k), d=normal(13) / math.sqrt(13))
        if H:
            s.gE = None               # pooled feeds the first layer only
    if c["kind"] == "host":
        s.batches = []
        for _ in range(2):
            off, ids, vals, _ = _batch(c, g)
            s.batches.append((off.cpu().pin_memory(), ids.cpu().pin_memory(), int(ids.numel()),
                              torch.zeros(B, k + 4).pin_memory()))
        # global rows of the second batch's keys (all of them are in the table)
        db = D.DeviceBatch(off, ids, vals, B)
        s.t.find_or_insert(db, False)
        if c["optimizer"] == "adam":
            _earlier_step(s, db, normal)
        base = torch.tensor(s.t.row_base(), device="cuda")
        rows = torch.unique(base[db.shards.long()] + db.rows.long()).to(torch.int32)
        s.rows = torch.full((_room_for_distinct(c),), -1, dtype=torch.int32, device="cuda")
        s.rows[:rows.numel()] = rows
        return s
    off, ids, vals, s.fresh = _batch(c, g, first_new=c["keys"])
    s.db = D.DeviceBatch(off, ids, vals, B)
    s.U = _room_for_distinct(c)
    s.db.uniq_rows = torch.full((max(s.U, s.db.nnz),), -1, dtype=torch.int32, device="cuda")
    if c["optimizer"] == "adam":
        _earlier_step(s, s.db, normal)
    s.part_small = None if c["fused"] else torch.zeros(S, B, k + 4, device="cuda")
    return s


# ---- one pass ---------------------------------------------------------------------------------------------------
def run(s):
    c = s.case
    B = c["batch"]
    if c["kind"] == "cross":
        y, P, _ = D.cross_forward(s.x0, s.x, s.w, s.b, c["shards"])
        gx0, gx, gw, gb = D.cross_backward(s.x0, s.x, s.w, P, s.gY)
        return dict(y=y, P=P, gx0=gx0, gx=gx, gw=gw, gb=gb)
    t, ops = s.t, s.ops
    if c["kind"] == "serve":
        t.find_or_insert(s.db, insert=False)
        t.forward_fused(ops, s.db, pooled=s.pooled, out_small=s.out_small, Z=s.Z)
        return dict(rows=s.db.rows, shards=s.db.shards, out_small=s.out_small, pooled=s.pooled, Z=s.Z)
    if c["kind"] == "host":
        tickets = [t.step_host_submit(ops, B, nnz, off, ids, None, out, d_pooled=s.pooled, gL=s.gL, gF=s.gF, gE=s.gE)
                   for off, ids, nnz, out in s.batches]
        for ticket in tickets:
            t.step_host_wait(ticket)
        r = t.read_rows(s.rows)
        return dict(r, out0=s.batches[0][3], out1=s.batches[1][3], pooled=s.pooled)

    db = s.db
    t.find_or_insert(db)
    if c["fused"]:
        t.forward_fused(ops, db, pooled=s.pooled, out_small=s.out_small, Z=s.Z)
    else:
        t.forward_partials(ops, db, s.part_small, s.pooled)
        t.aggregate(ops, db, s.part_small, s.pooled, out_small=s.out_small, Z=s.Z)
    if c["head"]:
        t.head(ops, B, s.hc, s.out_small, s.pooled, s.Z, s.xdense, s.y, s.logit, s.loss, s.gL, s.gF, s.gE, s.gZ)
    t.backward_update(ops, db, s.out_small, s.pooled, s.Z, s.gL, s.gF, s.gE, s.gZ, s.gE_work)
    out = t.read_rows(db.uniq_rows[:s.U])
    out.update(rows=db.rows, shards=db.shards, uidx=db.uidx, uniq_rows=db.uniq_rows[:s.U], n_uniq=db.n_uniq,
               part_small=s.part_small, out_small=s.out_small, pooled=s.pooled, Z=s.Z)
    if c["hidden"]:
        out.update(gE_work=s.gE_work, W1=t.dense1_get())
    if c["head"]:
        out.update(logit=s.logit, loss=s.loss, gL=s.gL, gF=s.gF, gE=s.gE, gZ=s.gZ)
    if c["kind"] == "stream":
        out["evicted"] = t.evict_keys(s.fresh)
    return out


# ---- what a pass cannot do without --------------------------------------------------------------------------------
def _distinct(n, s, vocab):
    """Expected number of distinct values among n draws of the Zipf law over `vocab` ranks."""
    edge = np.unique(np.concatenate([np.arange(0, min(vocab, 4096)), np.geomspace(min(vocab, 4096), vocab, 400)]).astype(np.int64))
    edge = np.append(edge[edge < vocab], vocab)
    a = 1.0 - s
    cdf = ((edge + 0.5) ** a - 0.5 ** a) / ((vocab + 0.5) ** a - 0.5 ** a)
    width = np.diff(edge).astype(np.float64)
    return float((width * -np.expm1(-n * np.diff(cdf) / width)).sum())


def _sizes(c):
    """(occurrences, distinct keys) of a batch, expected."""
    B, F = c["batch"], c["fields"]
    nnz = B * F * c["mean"]
    if c["partition"] == "field":
        return nnz, (F - c["buckets"]) * _distinct(B, c["zipf"], _vocab(c)) + 64.0 * c["buckets"] * -math.expm1(-B / 64.0)
    if c["kind"] == "stream":
        return nnz, _distinct(nnz * 15 / 16, c["zipf"], c["keys"]) + nnz / 16
    return nnz, _distinct(nnz, c["zipf"], _vocab(c))


def work(case):
    """Each input read once, each output written once; a key's row counts once per pass for reading and once for
    writing, however often the key occurs."""
    c = case
    B = c["batch"]
    if c["kind"] == "cross":
        d = c["dim"]
        return dict(bytes=4.0 * (6 * B * d + B + 4 * d), flops=B * d * 13.0)
    F, k, S, H = c["fields"], c["dim"], c["shards"], c["hidden"]
    ops = OPS[c["ops"]]
    nnz, U = _sizes(c)
    train = c["kind"] != "serve"
    row = 4.0 * (k + 2)                                       # latent vector, linear weight, cached norm
    state = {"sgd": 0.0, "adagrad": 1.0, "adam": 2.0}[c["optimizer"]] * 4.0 * (k + 1) + (8.0 if c["ftrl"] else 0.0)
    pooled = 4.0 * B * F * k if ops & POOL else 0.0
    b = 8.0 * nnz + (4.0 * nnz if c["vals"] else 0.0) + 4.0 * B * F + 16.0 * U        # ids, values, offsets, slots
    b += 5.0 * nnz + U * row + 4.0 * B * (k + 4) + pooled + 4.0 * B * H               # rows and shards, gather, outputs
    flops = nnz * (2.0 * k + 4) + 2.0 * B * F * k * H
    if H:
        b += 4.0 * F * k * H
    if train:
        b += 4.0 * nnz + 4.0 * U                                                       # uidx, uniq_rows
        b += U * (row + 2 * state)                                                     # update in place
        b += 8.0 * B + (0.0 if c["head"] and H else pooled) + 4.0 * B * H              # upstream gradients
        b += U * (4.0 + 8.0 * (k + 1)) if c["kind"] != "host" else 0.0                 # pull of the updated rows
        flops += nnz * 2.0 * k + U * k * 6.0 + 4.0 * B * F * k * H
        if H:
            b += pooled + 4.0 * F * k * H * (3.0 + 2.0 * {"sgd": 0, "adagrad": 1, "adam": 2}[c["optimizer"]])
        if not c["fused"] and c["kind"] != "host":
            b += 4.0 * S * B * (k + 4)
        if c["kind"] == "stream":
            b += nnz / 16 * (8.0 + 16.0)                                               # ids to evict, their slots
    if c["kind"] == "host":
        b, flops = 2 * b + U * 8.0 * (k + 1), 2 * flops
    return dict(bytes=b, flops=flops)


def tolerance(case):
    """float32 sums in another order; with a first dense layer its operands are bfloat16, and so is all that follows
    from it.  Integers are the same.  `max` leaves room for single sums that cancel."""
    if case["kind"] != "cross" and case["hidden"]:
        return {"rel": 1e-2, "max": 0.4}
    return {"rel": 1e-5, "max": 1e-2}
