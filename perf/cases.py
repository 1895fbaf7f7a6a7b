"""Performance cases of the library: what a user of it has it do, through the public binding, over the sizes in use.

Five kinds of pass (``kind``):

``train``     restore both tables, ``epochs`` epochs with the objective read after each ``loss_every`` of them, fetch both tables
``job``       the whole job from page-locked host buffers: upload of the matrix and of both tables, epochs, both tables back
``fold``      embeddings of new rows from their entries, host arrays in and out
``topk``      Top-K of device-resident queries over a resident item table
``serve``     a request: fold in a few new rows, and the Top-K of as many known ones without the items they already have
``evaluate``  the held-out protocol on folded-in rows: Top-K without the kept links, Recall@K against the held-out ones

Matrices are long-tailed in both directions: row lengths follow a capped rank-size law, the columns of a row follow a popularity
law or stay near the row's own id (``law``).  Tables of a trained model have a decaying spectrum; training starts from small
normal tables and, where ``warm`` is set, from the tables that many epochs later (a run that is resumed).
"""
import math

import numpy as np
import torch

from paper_2112_02194_b200.binding import ALX_COLS, ALX_ROWS, Alx


def _train(name, n, m, nnz, d, storage, law, epochs, loss_every, warm=0, labels=False, solver=0, s=1.1, lam=0.02, alpha=0.001):
    return dict(name=name, kind="train", n=n, m=m, nnz=nnz, d=d, storage=storage, law=law, s=s, epochs=epochs,
                loss_every=loss_every, warm=warm, labels=labels, solver=solver, lam=lam, alpha=alpha)


def listed():
    return [
        # the smallest model: a whole training run of 16 epochs, objective watched after each; launches and latency count
        _train("train_f32_d16_tiny", 2000, 1500, 40_000, 16, "f32", "uniform", 16, 1, lam=0.1, alpha=0.01, s=0.6),
        # ratings of an ordinary size with labels, fp32 tables of 32 features, odd sizes
        _train("train_f32_d32_labels", 138_493, 26_747, 10_000_003, 32, "f32", "popular", 2, 1, labels=True, s=0.7, lam=0.05, alpha=0.01),
        # the mid-size fp32 graph: 1M x 1M, 5e7 entries, 64 features, resumed after three epochs
        _train("train_f32_d64", 1_000_000, 1_000_000, 50_000_000, 64, "f32", "popular", 1, 1, warm=3, s=1.2, lam=0.05),
        # bfloat16 tables of 64 features, ragged sizes, more rows than columns
        _train("train_bf16_d64", 301_117, 90_001, 6_000_011, 64, "bf16", "popular", 2, 2, s=0.9),
        # 128 features in fp32 (no reduced storage), labels
        _train("train_f32_d128_labels", 60_013, 24_989, 2_000_003, 128, "f32", "popular", 1, 1, labels=True, s=0.8),
        # a small graph on the bfloat16 path: three epochs from fresh tables
        _train("train_bf16_d128_small", 200_000, 200_000, 10_000_000, 128, "bf16", "local", 3, 3, lam=0.01),
        # the headline workload: 10M x 10M, 1e9 entries, 128 features, bfloat16 tables, one more epoch of a run under way
        _train("train_bf16_d128_large", 10_000_000, 10_000_000, 1_000_000_000, 128, "bf16", "local", 1, 1, warm=3, lam=0.01),
        # a nightly job that starts and ends in host memory
        dict(name="job_bf16_d128", kind="job", n=400_000, m=250_007, nnz=20_000_000, d=128, storage="bf16", law="popular", s=1.0,
             epochs=2, labels=False, lam=0.01, alpha=0.001),
        # one online request: three new users to embed, three known ones to give 20 items each out of a million
        dict(name="serve_bf16_d128_few", kind="serve", m=1_000_000, d=128, storage="bf16", new=3, mean=40, k=20),
        # a day's new users in one batch
        dict(name="fold_f32_d64_batch", kind="fold", m=200_003, d=64, storage="f32", new=50_021, mean=30, labels=True),
        # related items for a page of queries, fp32 tables
        dict(name="topk_f32_d64", kind="topk", m=300_007, d=64, storage="f32", queries=300, k=50),
        # the retrieval half of the held-out protocol on a block of test rows
        dict(name="evaluate_bf16_d128", kind="evaluate", m=1_000_000, d=128, storage="bf16", new=2048, mean=40, k=50),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["train", "train", "train", "train", "job", "fold", "topk", "serve", "evaluate"])
    d, storage = rng.choice([(16, "f32"), (32, "f32"), (64, "f32"), (128, "f32"), (16, "bf16"), (32, "bf16"), (64, "bf16"),
                             (128, "bf16"), (128, "bf16"), (128, "bf16")])
    if kind in ("train", "job"):
        nnz = _log(rng, 30_000, 30_000_000 if d * (2 if storage == "bf16" else 4) <= 256 else 8_000_000)
        n = max(500, int(nnz / math.exp(rng.uniform(math.log(8), math.log(120)))))
        m = max(500, int(n * math.exp(rng.uniform(math.log(0.2), math.log(2.0)))))
        c = dict(kind=kind, n=n, m=m, nnz=nnz, d=d, storage=storage, law=rng.choice(["uniform", "popular", "local"]),
                 s=round(rng.uniform(0.6, 1.2), 2), epochs=rng.randint(1, 3), labels=rng.random() < 0.4,
                 lam=round(rng.uniform(0.01, 0.1), 3), alpha=rng.choice([0.0005, 0.001, 0.01]))
        if kind == "train":
            c.update(loss_every=1, warm=rng.choice([0, 2]), solver=int(rng.random() < 0.2))
        return c
    m = _log(rng, 5_000, 1_500_000)
    if kind == "fold":
        return dict(kind=kind, m=m, d=d, storage=storage, new=_log(rng, 1, 60_000), mean=rng.randint(4, 80), labels=rng.random() < 0.5)
    if kind == "topk":
        return dict(kind=kind, m=m, d=d, storage=storage, queries=_log(rng, 1, 2048), k=rng.choice([1, 10, 20, 50, 100]))
    return dict(kind=kind, m=m, d=d, storage=storage, new=_log(rng, 1, 64) if kind == "serve" else _log(rng, 100, 4000),
                mean=rng.randint(10, 60), k=rng.choice([10, 20, 50]))


# ------------------------------------------------------------------------------------------------------------------ inputs
def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed((seed * 1_000_003 + stream) & ((1 << 62) - 1))
    return g


def _degrees(n, nnz, s, cap, gen):
    """int64[n]: capped rank-size law of exponent s with the given sum (up to the cap), scattered over the rows."""
    base = torch.arange(1, n + 1, dtype=torch.float64, device="cuda").pow_(-s)
    lo, hi = 0.0, 2.0 * cap * n ** s
    for _ in range(50):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if float((base * mid).clamp_(1, cap).sum()) < nnz else (lo, mid)
    deg = (base * hi).clamp_(1, cap).floor_().to(torch.int64)
    left = nnz - int(deg.sum())                        # what the floor took: one each for the first rows that have room
    if left > 0:
        deg[(deg < cap).nonzero().flatten()[:left]] += 1
    return deg[torch.randperm(n, generator=gen, device="cuda")]


def _matrix(n, m, nnz, law, s, seed):
    """(rowptr int64, colidx int32) on the GPU; ascending, distinct columns in each row."""
    gen = _gen(seed, 1)
    deg = _degrees(n, nnz, s, max(1, min(m // 2, 1_000_000)), gen)
    ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(deg, 0, out=ptr[1:])
    total = int(ptr[-1])
    col = torch.empty(total, dtype=torch.int32, device="cuda")
    width = max(m // 50, 16)                           # law "local": four entries in five within 1 % of the row's place
    piece = 1 << 26
    for e0 in range(0, total, piece):
        e1 = min(total, e0 + piece)
        e = torch.arange(e0, e1, dtype=torch.int64, device="cuda")
        row = torch.searchsorted(ptr, e, right=True) - 1
        k = deg[row]
        j = e - ptr[row]
        t = (j + torch.rand(e1 - e0, generator=gen, dtype=torch.float64, device="cuda")) / k
        if law == "popular":
            g = t.pow_(2.5)
        elif law == "local":
            a = ((row.to(torch.float64) * (m / n) - width / 2).clamp_(0, max(m - width, 0))) / m
            b = a + min(width, m) / m
            left = 0.2 * a / (1 - b + a).clamp_(min=1e-9)  # share of the entries before the window
            g = torch.where(t < left, t * (a / left.clamp(min=1e-12)),
                            torch.where(t < left + 0.8, a + (t - left) * ((b - a) / 0.8),
                                        b + (t - left - 0.8) * ((1 - b) / (0.2 - left).clamp(min=1e-12))))
            g = g.clamp_(0, 1 - 1e-12)
        else:
            g = t
        col[e0:e1] = (torch.floor(g * (m - k)).to(torch.int64) + j).to(torch.int32)
    return ptr, col


def _dtype(storage):
    return torch.bfloat16 if storage == "bf16" else torch.float32


def _normal(n, d, storage, seed, stream, sigma):
    return torch.empty(n, d, dtype=_dtype(storage), device="cuda").normal_(0.0, sigma, generator=_gen(seed, stream))


def _trained(n, d, storage, seed, stream):
    """A table with the decaying spectrum of a trained model."""
    z = torch.randn(d, d, generator=_gen(seed, stream + 1), device="cuda")
    mix = torch.linalg.qr(z)[0] * torch.arange(1, d + 1, device="cuda", dtype=torch.float32).pow(-0.5)[:, None]
    return (torch.randn(n, d, generator=_gen(seed, stream), device="cuda") @ mix * 0.5).to(_dtype(storage))


def _labels(count, seed):
    return torch.rand(count, generator=_gen(seed, 5), device="cuda") * 1.5 + 0.5


def _pinned(t):
    out = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    out.copy_(t)
    return out


def _bits(t):
    """The numpy array the host calls take: float32, or the bit patterns of bfloat16."""
    return t.view(torch.int16).numpy().view(np.uint16) if t.dtype == torch.bfloat16 else t.numpy()


def _state_train(c, seed):
    ptr, col = _matrix(c["n"], c["m"], c["nnz"], c["law"], c["s"], seed)
    val = _labels(col.numel(), seed) if c["labels"] else None
    a = Alx(c["n"], c["m"], c["d"], c["lam"], c["alpha"], storage=c["storage"], solver=c.get("solver", 0))
    sigma = 0.1 / math.sqrt(c["d"])
    W = _normal(c["n"], c["d"], c["storage"], seed, 2, sigma)
    H = _normal(c["m"], c["d"], c["storage"], seed, 3, sigma)
    if c["kind"] == "job":
        return dict(a=a, ptr=_pinned(ptr), col=_pinned(col), val=None if val is None else _pinned(val), W=_pinned(W), H=_pinned(H),
                    W_out=_pinned(W), H_out=_pinned(H))
    a.set_csr(ptr, col, val)
    del ptr, col, val
    if c["warm"]:
        a.set_embeddings(ALX_ROWS, W)
        a.set_embeddings(ALX_COLS, H)
        for _ in range(c["warm"]):
            a.epoch()
        a.get_embeddings(ALX_ROWS, out=W)
        a.get_embeddings(ALX_COLS, out=H)
    return dict(a=a, W=W, H=H, W_out=torch.empty_like(W), H_out=torch.empty_like(H))


def _state_model(c, seed):
    """A trained model in hand: the item table resident, new rows or queries beside it."""
    m, d = c["m"], c["d"]
    a = Alx(1000, m, d, 0.05, 0.001, storage=c["storage"])
    a.set_embeddings(ALX_COLS, _trained(m, d, c["storage"], seed, 10))
    st = dict(a=a)
    if c["kind"] == "topk":
        q = c["queries"]
        st.update(q=_trained(q, d, "f32", seed, 20), ids=torch.empty(q, c["k"], dtype=torch.int32, device="cuda"),
                  scores=torch.empty(q, c["k"], dtype=torch.float32, device="cuda"))
        return st
    ptr, col = _matrix(c["new"], m, c["new"] * c["mean"], "popular", 0.5, seed)      # entries of the rows the pass is about
    if c["kind"] == "evaluate":
        # a quarter of each row's links is held out (every fourth), the rest is kept
        deg = ptr[1:] - ptr[:-1]
        row = torch.repeat_interleave(torch.arange(c["new"], device="cuda"), deg)
        held = (torch.arange(col.numel(), device="cuda") - ptr[row]) % 4 == 3
        zero = torch.zeros(1, dtype=torch.int64, device="cuda")
        for name, mask in (("truth", held), ("kept", ~held)):
            n_of = torch.bincount(row[mask], minlength=c["new"])
            st[name] = (torch.cat([zero, torch.cumsum(n_of, 0)]).cpu().numpy(), col[mask].cpu().numpy())
    else:
        st["kept"] = (ptr.cpu().numpy(), col.cpu().numpy())
    st["val"] = _labels(col.numel(), seed).cpu().numpy() if c.get("labels") else None
    if c["kind"] != "fold":
        st["q"] = _trained(c["new"], d, "f32", seed, 20).cpu().numpy()
    return st


def prepare(case, seed):
    st = _state_train(case, seed) if case["kind"] in ("train", "job") else _state_model(case, seed)
    st["case"] = case
    return st


# -------------------------------------------------------------------------------------------------------------------- passes
def run(st):
    c, a = st["case"], st["a"]
    if c["kind"] == "train":
        a.set_embeddings(ALX_ROWS, st["W"])
        a.set_embeddings(ALX_COLS, st["H"])
        losses = []
        for e in range(1, c["epochs"] + 1):
            a.epoch()
            if e % c["loss_every"] == 0:
                losses.append(a.loss()[0])
        return dict(W=a.get_embeddings(ALX_ROWS, out=st["W_out"]), H=a.get_embeddings(ALX_COLS, out=st["H_out"]),
                    losses=np.array(losses))
    if c["kind"] == "job":
        a.load_host(st["ptr"].numpy(), st["col"].numpy(), None if st["val"] is None else st["val"].numpy(), _bits(st["W"]), _bits(st["H"]))
        for _ in range(c["epochs"] - 1):
            a.epoch()
        a.epoch_to_host(_bits(st["W_out"]), _bits(st["H_out"]))
        return dict(W=st["W_out"], H=st["H_out"])
    if c["kind"] == "topk":
        a.topk_device(ALX_COLS, st["q"], c["k"], st["ids"], st["scores"])
        return dict(ids=st["ids"], scores=st["scores"])
    if c["kind"] == "fold":
        return a.fold_in(*st["kept"], st["val"])
    out = dict(x=a.fold_in(*st["kept"])) if c["kind"] == "serve" else {}
    out["ids"], out["scores"] = a.topk(ALX_COLS, st["q"], c["k"], exclude=st["kept"])
    if c["kind"] == "evaluate":
        out["recall"] = a.recall_at_k(out["ids"], c["k"], *st["truth"])[0]
    return out


# ---------------------------------------------------------------------------------------------------- floors and tolerances
def work(case):
    """Inputs read once, outputs written once; products of Eq. 4 with symmetric sums and one factorisation per row (rows of fewer
    than d entries through their own, smaller system)."""
    c, d = case, case["d"]
    e = 2 if c["storage"] == "bf16" else 4

    def solve(rows, entries, fixed):
        k = entries / max(1, rows)
        per = k * d * (d + 1.0) + d ** 3 / 3.0 if k >= d else min(k * d * (d + 1.0) + d ** 3 / 3.0, 2.0 * k * d * (k + 2.0) + k ** 3 / 3.0)
        return rows * per + fixed * d * (d + 1.0)

    if c["kind"] in ("train", "job"):
        n, m, nnz = c["n"], c["m"], c["nnz"]
        index = nnz * (4 + (4 if c["labels"] else 0))
        epoch = 2 * index + (n + m) * (8 + 3 * d * e)
        once = 2 * (n + m) * d * e
        if c["kind"] == "train":
            reads = c["epochs"] // c["loss_every"]
            return dict(bytes=c["epochs"] * epoch + 2 * once + reads * (index + (n + m) * d * e),
                        flops=c["epochs"] * (solve(n, nnz, m) + solve(m, nnz, n)) + reads * 2.0 * nnz * d)
        return dict(bytes=c["epochs"] * epoch + once + 3 * index, flops=c["epochs"] * (solve(n, nnz, m) + solve(m, nnz, n)))
    m = c["m"]
    if c["kind"] == "topk":
        return dict(bytes=m * d * e + c["queries"] * (4 * d + 8 * c["k"]), flops=2.0 * m * d * c["queries"])
    new, entries = c["new"], c["new"] * c["mean"]
    b, f = 0.0, 0.0
    if c["kind"] != "evaluate":
        b += m * d * e + new * (8 + 4 * d) + entries * (8 if c.get("labels") else 4)
        f += solve(new, entries, m)
    if c["kind"] != "fold":
        b += m * d * e + new * (4 * d + 8 * c["k"]) + entries * 4
        f += 2.0 * m * d * new
    return dict(bytes=b, flops=f)


def tolerance(case):
    """fp32 tables: iterative solves stopped at a relative residual of 1e-6 on systems of condition up to about 10^3 in single rows.
    bfloat16 tables: each value is rounded to 2^-9.  Ids: two items whose scores differ by less than fp32 rounding may swap."""
    if case["kind"] in ("topk", "evaluate"):
        return dict(rel=1e-5, max=1e-4, differ=1e-3)
    t = dict(rel=1e-4, max=1e-2) if case["storage"] == "f32" else dict(rel=1e-2, max=0.3)
    return dict(t, differ=1e-3) if case["kind"] == "serve" else t
