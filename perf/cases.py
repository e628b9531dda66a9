"""Timed cases of the parameter manager, through the methods of `adapm.ParameterManager`.

A pass of a clock case is one clock of a data-parallel job (App. C of the paper): every worker slot signals the
intent of the batch `lookahead` clocks ahead, uses its current batch (pull + push, or a fused training step) and
advances its clock; one sync merges the clock's updates; then the job reads back the rows that the clock's
batches touched.  A pass of an access case reads and writes without any intent: pull, push, read back.

Outputs: the rows every worker pulled (clock and access cases), the batch losses (training steps) and the touched
rows after the pass, whole.  Sizes are those of the five workloads that the benchmark and the tests name, and
sizes between them.
"""
import math

import numpy as np
import torch

from paper_2206_00470_gb300 import adapm

DEV = "cuda"


def listed():
    return [
        # --- the smallest calls: latency and launches -----------------------------------------------------------
        # the tiny factorisation configuration: a few hundred cells per worker and clock
        mf("tiny_mf", rows=1000, cols=500, rank=16, adagrad=False, workers=4, batch=256, lookahead=2, s=0.0),
        # a latency-critical reader and writer of a thousand rows, no intents, no allocation in the push
        access("online_1k", keys=1_000_000, dim=64, batch=1000, s=1.1, noalloc=True),
        # the smallest batch of the access microbenchmark
        clock("clock_16k", keys=10_000_000, dim=64, workers=8, batch=1 << 14, s=1.1, span=1, lookahead=1),
        # --- ordinary sizes --------------------------------------------------------------------------------------
        # moderate skew, replicas held for several clocks (overlapping windows)
        clock("clock_128k_span4", keys=20_000_000, dim=64, workers=8, batch=1 << 17, s=0.8, span=4, lookahead=1),
        # a few hot keys take most rows; ragged rows (9 vectors), an odd batch, an odd number of workers
        clock("clock_hot_odd", keys=10_000_000, dim=36, workers=5, batch=300_007, s=1.4, span=2, lookahead=2),
        # relocation instead of replication for keys with one active worker
        clock("clock_relocate", keys=20_000_000, dim=64, workers=8, batch=1 << 18, s=0.8, span=1, lookahead=1,
              relocate=True),
        # the benchmark's factorisation: rank 100 + AdaGrad
        mf("mf_65k", rows=10_000_000, cols=1_000_000, rank=100, adagrad=True, workers=8, batch=65_536, lookahead=4,
           s=1.1),
        # the same job fed by a data loader: pinned host batches, odd batch size
        mf("mf_host_odd", rows=2_000_000, cols=200_000, rank=100, adagrad=True, workers=4, batch=29_989, lookahead=4,
           s=1.1, host=True),
        # --- the largest -----------------------------------------------------------------------------------------
        # bulk reads and updates without intent: uniform keys, an odd count, rows of 50 vectors
        access("bulk_1m", keys=11_000_000, dim=200, batch=999_983, s=0.0, noalloc=False),
        # the access microbenchmark at 100M keys
        clock("clock_1m", keys=100_000_000, dim=64, workers=8, batch=1 << 20, s=1.1, span=1, lookahead=1),
        # knowledge-graph embeddings: 103 rows of 512 floats per triple
        kge("complex_4k", entities=5_000_000, relations=800, half=128, workers=8, batch=4096, negs=100, lookahead=2),
        # word vectors: 261 rows of 300 floats per centre
        sgns("sgns_8k", vocab=700_000, dim=300, workers=8, batch=8192, window=5, negs=25, lookahead=3),
    ]


def clock(name, keys, dim, workers, batch, s, span, lookahead, relocate=False, refresh=False, timing="start"):
    return {"name": name, "kind": "clock", "keys": keys, "dim": dim, "workers": workers, "batch": batch, "s": s,
            "span": span, "lookahead": lookahead, "relocate": relocate, "refresh": refresh, "timing": timing,
            "host": False}


def access(name, keys, dim, batch, s, noalloc):
    return {"name": name, "kind": "access", "keys": keys, "dim": dim, "workers": 1, "batch": batch, "s": s,
            "noalloc": noalloc}


def mf(name, rows, cols, rank, adagrad, workers, batch, lookahead, s, host=False, relocate=False):
    return {"name": name, "kind": "mf", "rows": rows, "cols": cols, "keys": rows + cols, "rank": rank,
            "adagrad": adagrad, "dim": rank * (2 if adagrad else 1), "workers": workers, "batch": batch, "s": s,
            "span": 1, "lookahead": lookahead, "host": host, "relocate": relocate, "refresh": False,
            "timing": "start"}


def kge(name, entities, relations, half, workers, batch, negs, lookahead):
    return {"name": name, "kind": "complex", "entities": entities, "relations": relations,
            "keys": entities + relations, "half": half, "dim": 4 * half, "workers": workers, "batch": batch,
            "negs": negs, "span": 1, "lookahead": lookahead, "host": False, "relocate": False, "refresh": False,
            "timing": "start"}


def sgns(name, vocab, dim, workers, batch, window, negs, lookahead):
    return {"name": name, "kind": "sgns", "vocab": vocab, "keys": 2 * vocab, "dim": dim, "workers": workers,
            "batch": batch, "window": window, "negs": negs, "span": 1, "lookahead": lookahead, "host": False,
            "relocate": False, "refresh": False, "timing": "start"}


# ---------------------------------------------------------------------------
# drawn cases
# ---------------------------------------------------------------------------
def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["clock"] * 5 + ["access"] * 2 + ["mf"] * 2 + ["complex", "sgns"])
    if kind == "clock":
        dim = rng.choice([16, 20, 36, 64, 100, 128, 200, 256])
        workers, span = rng.randint(1, 8), rng.choice([1, 1, 1, 2, 4, 8])
        # no more row floats than the largest batch of 8 workers, no more than 24 GB of replica pool
        most = min(1 << 20, (8 << 26) // (workers * dim), 24_000_000_000 // (workers * (span + 4) * 8 * dim))
        batch = _log(rng, 256, most)
        keys = _log(rng, 20_000, min(100_000_000, 24_000_000_000 // (4 * dim)))
        opt = rng.choice(["", "", "", "", "relocate", "relocate", "refresh", "adaptive"])
        c = clock("", keys, dim, workers, batch, rng.choice([0.0, 0.8, 1.1, 1.4]), span, rng.randint(1, 3),
                  opt == "relocate", opt == "refresh", "adaptive" if opt == "adaptive" else "start")
    elif kind == "access":
        dim = rng.choice([16, 36, 64, 100, 200, 300, 512])
        batch = _log(rng, 100, min(1_000_000, 200_000_000 // dim))
        keys = _log(rng, 20_000, min(50_000_000, 10_000_000_000 // (4 * dim)))
        c = access("", keys, dim, batch, rng.choice([0.0, 0.8, 1.1, 1.4]),
                   batch <= 300_000 and rng.random() < 0.3)
    elif kind == "mf":
        rank = rng.choice([16, 32, 64, 100, 128])
        rows = _log(rng, 1000, 10_000_000)
        c = mf("", rows, max(500, rows // 10), rank, rng.random() < 0.7, rng.randint(1, 8), _log(rng, 200, 65_536),
               rng.randint(1, 4), rng.choice([0.0, 1.1, 1.1]), rng.random() < 0.3, rng.random() < 0.2)
    elif kind == "complex":
        c = kge("", _log(rng, 20_000, 4_000_000), rng.choice([50, 800]), rng.choice([32, 64, 100, 128]),
                rng.randint(1, 4), _log(rng, 100, 4096), rng.choice([10, 33, 100]), rng.randint(1, 2))
    else:
        c = sgns("", _log(rng, 5_000, 700_000), rng.choice([64, 100, 200, 300]), rng.randint(1, 4),
                 _log(rng, 100, 8192), rng.choice([2, 5]), rng.choice([5, 10, 25]), rng.randint(1, 3))
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
DELTA_STD, INIT_STD, LR, EPS = 1e-3, 0.1, 0.05, 1e-8


def _ranks(n, size, s, g):
    """n ranks in [0, size), P(rank) falling as (rank + 1)^-s (the bounded power law, rounded down)."""
    u = torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    if s == 0.0:
        x = u * size
    elif s == 1.0:
        x = torch.exp(u * math.log(size + 1.0)) - 1.0
    else:
        x = torch.pow(u * ((size + 1.0) ** (1.0 - s) - 1.0) + 1.0, 1.0 / (1.0 - s)) - 1.0
    return x.to(torch.int64).clamp_(0, size - 1)


def _spread(ranks, size, salt):
    """Ranks to keys by a fixed bijection of [0, size), so that hot keys are not neighbours."""
    a = max(1, int(size * (0.6180339887 + 0.01 * salt))) | 1
    while math.gcd(a, size) != 1:
        a += 2
    return (ranks * a + 12345 + salt) % size


def _store(c, g):
    """Initial rows: parameters N(0, 0.1); AdaGrad accumulators as after some training."""
    K, D = c["keys"], c["dim"]
    init = torch.empty((K, D), device=DEV)
    if c["kind"] == "complex" or c.get("adagrad"):
        init[:, :D // 2].normal_(0.0, INIT_STD, generator=g)
        init[:, D // 2:].uniform_(0.05, 1.0, generator=g)
    else:
        init.normal_(0.0, INIT_STD, generator=g)
    return init


def _batch(c, w, g):
    """One worker's batch: the arguments of its access or step, and "keys", the keys its intent names."""
    B = c["batch"]
    if c["kind"] in ("clock", "access"):
        return {"keys": _spread(_ranks(B, c["keys"], c["s"], g), c["keys"], 0)}
    if c["kind"] == "mf":
        W = c["workers"]
        share = c["rows"] // W   # rows are partitioned over the workers
        r = _spread(_ranks(B, share, c["s"], g), share, 1) * W + w
        k = _spread(_ranks(B, c["cols"], c["s"], g), c["cols"], 2) + c["rows"]
        v = torch.randn(B, generator=g, device=DEV)
        return {"rows": r, "cols": k, "vals": v, "keys": torch.cat([r, k])}
    if c["kind"] == "complex":
        E = c["entities"]
        h, t = (_spread(_ranks(B, E, 1.0, g), E, 1) for _ in range(2))
        r = _spread(_ranks(B, c["relations"], 1.2, g), c["relations"], 2) + E
        n = torch.randint(0, E, (B * c["negs"],), generator=g, device=DEV)
        return {"heads": h, "rels": r, "tails": t, "negs": n, "keys": torch.cat([h, r, t, n])}
    V, ww = c["vocab"], c["window"]
    stream = _spread(_ranks(B + 2 * ww, V, 1.0, g), V, 1)
    offs = torch.tensor([o for o in range(-ww, ww + 1) if o], device=DEV)
    at = torch.arange(B, device=DEV).view(-1, 1) + ww + offs
    ctx = stream[at]
    if w == 0:   # the first worker's shard begins here: its first tokens miss contexts
        ctx = torch.where(at < ww, torch.full_like(ctx, 0xFFFFFFFF), ctx)
    neg = _spread(_ranks(B * 2 * ww * c["negs"], V, 0.75, g), V, 1).view(B, 2 * ww, c["negs"])
    cen = stream[ww:ww + B]
    pres = ctx != 0xFFFFFFFF
    return {"centres": cen, "contexts": ctx, "negs": neg,
            "keys": torch.cat([cen, V + ctx[pres], V + neg[pres].reshape(-1)])}


def _inputs(c, seed):
    g = torch.Generator(device=DEV).manual_seed(1_000_003 * (seed + 1))
    init = _store(c, g)
    ring = c.get("lookahead", 1) + 2
    batches = [[_batch(c, w, g) for w in range(c["workers"])] for _ in range(ring)]
    deltas = None
    if c["kind"] in ("clock", "access"):
        deltas = [torch.empty((c["batch"], c["dim"]), device=DEV).normal_(0.0, DELTA_STD, generator=g)
                  for _ in range(c["workers"])]
    return init, batches, deltas


def _read_back(c, batch):
    """The distinct keys of one clock's batches, ascending, and the list that a pass reads back: a fixed number of
    them (some twice, since the number of distinct keys varies a little with the data)."""
    t = torch.unique(torch.cat([b["keys"] for b in batch]))
    n = int(1.03 * _touched(c)) + 128
    return t, t[torch.arange(n, device=DEV) % t.numel()]


def _int32(x):
    """Keys as the manager takes them: 32 bits (0xFFFFFFFF, "no context", wraps to -1)."""
    return x.reshape(-1).to(torch.int32)


def prepare(case, seed):
    c = dict(case)
    init, batches, deltas = _inputs(c, seed)
    touched = [_read_back(c, bs)[1] for bs in batches]
    K, D, W, B = c["keys"], c["dim"], c["workers"], c["batch"]
    most = max(b["keys"].numel() for bs in batches for b in bs)
    if c["kind"] == "access":
        pm = adapm.ParameterManager(K, D, W, replica_capacity=1024, init_values=init)
    else:
        hold = c["span"] + 1 + (0 if c["timing"] == "start" else c["lookahead"])
        pm = adapm.ParameterManager(K, D, W, replica_capacity=min(W * K, W * hold * most), init_values=init,
                                    relocate=c["relocate"], delta_refresh=c["refresh"], action_timing=c["timing"])
    del init
    data = [[{k: (v if v.dtype == torch.float32 else _int32(v)) for k, v in b.items()} for b in bs]
            for bs in batches]
    if c.get("host"):
        data = [[{k: v.cpu().pin_memory() for k, v in b.items()} for b in bs] for bs in data]
    st = {"c": c, "pm": pm, "data": data, "deltas": deltas, "touched": [_int32(t) for t in touched], "clock": 0,
          "merged": torch.empty((touched[0].numel(), D), device=DEV)}
    if c["kind"] in ("clock", "access"):
        st["out"] = [torch.empty((B, D), device=DEV) for _ in range(W)]
    else:
        st["loss"] = torch.zeros(W, dtype=torch.float64, device=DEV)
    if c["kind"] != "access":
        for j in range(c["lookahead"]):
            for w in range(W):
                pm.intent(w, data[j][w]["keys"], j, j + c["span"])
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    st, c, pm = state, state["c"], state["pm"]
    cl = st["clock"]
    st["clock"] = cl + 1
    now = st["data"][cl % len(st["data"])]
    touched, merged = st["touched"][cl % len(st["data"])], st["merged"]
    if c["kind"] == "access":
        keys = now[0]["keys"]
        pm.pull(0, keys, out=st["out"][0])
        (pm.push_noalloc if c["noalloc"] else pm.push)(0, keys, st["deltas"][0])
        pm.pull(0, touched, out=merged)
        return {"rows": st["out"], "merged": merged}
    nxt = cl + c["lookahead"]
    ahead = st["data"][nxt % len(st["data"])]
    for w in range(c["workers"]):
        pm.intent(w, ahead[w]["keys"], nxt, nxt + c["span"])
        b = now[w]
        if c["kind"] == "clock":
            pm.pull(w, b["keys"], out=st["out"][w])
            pm.push(w, b["keys"], st["deltas"][w])
        elif c["kind"] == "mf":
            pm.mf_step(w, b["rows"], b["cols"], b["vals"], c["rank"], c["adagrad"], LR, EPS,
                       loss_out=st["loss"][w:w + 1])
        elif c["kind"] == "complex":
            pm.complex_step(w, b["heads"], b["rels"], b["tails"], b["negs"], c["negs"], 2 * c["half"], LR, EPS,
                            loss_out=st["loss"][w:w + 1])
        else:
            pm.sgns_step(w, b["centres"], b["contexts"], b["negs"], 2 * c["window"], c["negs"], c["vocab"],
                         c["dim"], LR, loss_out=st["loss"][w:w + 1])
        pm.advance_clock(w)
    pm.sync()
    pm.pull(0, touched, out=merged)
    return {"rows": st["out"], "merged": merged} if c["kind"] == "clock" else {"loss": st["loss"], "merged": merged}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _distinct(draws, size, s):
    """Expected number of distinct ranks among `draws` draws of _ranks(., size, s)."""
    if s == 0.0:
        return size * -math.expm1(-draws / size)
    x = np.exp(np.linspace(0.0, math.log(size + 1.0), 1 << 16))
    f = np.log(x) / math.log(size + 1.0) if s == 1.0 else (x ** (1 - s) - 1) / ((size + 1.0) ** (1 - s) - 1)
    count, mass = np.diff(x), np.diff(f)
    edge = np.arange(1.0, min(size, 4096) + 1)        # the first ranks one by one
    fe = np.log(edge) / math.log(size + 1.0) if s == 1.0 else (edge ** (1 - s) - 1) / ((size + 1.0) ** (1 - s) - 1)
    head = float(-np.expm1(-draws * np.diff(fe)).sum())
    tail = x[:-1] >= edge[-1]
    return head + float((count * -np.expm1(-draws * mass / count))[tail].sum())


def _touched(c):
    """Expected number of distinct keys in one clock's batches of all workers."""
    W, B = c["workers"], c["batch"]
    if c["kind"] in ("clock", "access"):
        u = _distinct(W * B, c["keys"], c["s"])
    elif c["kind"] == "mf":
        u = W * _distinct(B, c["rows"] // W, c["s"]) + _distinct(W * B, c["cols"], c["s"])
    elif c["kind"] == "complex":
        E = c["entities"]
        u = min(E, E * -math.expm1(-W * B * c["negs"] / E) + _distinct(2 * W * B, E, 1.0))
        u += _distinct(W * B, c["relations"], 1.2)
    else:
        V, pairs = c["vocab"], W * B * 2 * c["window"]
        u = _distinct(W * B, V, 1.0) + min(V, _distinct(pairs * c["negs"], V, 0.75))
    return min(c["keys"], u)


def work(case):
    c = case
    W, B, D = c["workers"], c["batch"], c["dim"]
    row, u = 4 * D, _touched(c)
    if c["kind"] in ("clock", "access"):
        keys = W * B * (2 if c["kind"] == "access" else 3) + u        # pull, push (and intent) keys, touched keys
        # delta rows in, pulled rows out; each distinct row read, updated and read back once
        return {"bytes": int(4 * keys + 2 * W * B * row + 3 * u * row), "flops": int(W * B * D)}
    if c["kind"] == "mf":
        n, extra, flops = 2 * W * B, 4 * W * B, W * B * (12 if c["adagrad"] else 6) * c["rank"]
    elif c["kind"] == "complex":
        n, extra = W * B * (3 + c["negs"]), 0
        flops = n * 2 * c["half"] * 12
    else:
        n, extra = W * B * (1 + 2 * c["window"] * (1 + c["negs"])), 0
        flops = n * D * 6
    # step and intent keys, cell values, touched keys; each distinct row read, updated and read back once
    return {"bytes": int(8 * n + extra + 4 * u + 3 * u * row), "flops": int(flops)}


def tolerance(case):
    """Pulled rows are copies; merged rows and losses are fp32 sums, in another order about as far apart as from
    the sums in 64 bits; stated: four times that."""
    if case["kind"] in ("clock", "access"):     # 2.5e-8 to 4e-8 off 64 bits
        return {"rel": 2e-7, "max": 2e-5}
    return {"rel": 5e-7, "max": 1e-4}           # 3e-8 to 1e-7 off 64 bits


# ---------------------------------------------------------------------------
# the first pass in 64 bits
# ---------------------------------------------------------------------------
def _softplus(x):
    return torch.log1p(torch.exp(-x.abs())) + x.clamp_min(0.0)


def _ada(gr, acc):
    return torch.cat([-LR * gr / torch.sqrt(acc + gr * gr + EPS), gr * gr], dim=1)


def exact(case, seed):
    c = dict(case)
    # With relocation a key moves to the worker that alone uses it, which then reads the main copy with the updates
    # of workers that went before it: rows read within the clock have no closed form, only what is merged has.
    if c.get("relocate") and c["kind"] == "mf":
        return None
    init, batches, deltas = _inputs(c, seed)
    t, back = _read_back(c, batches[0])
    base = init[t].double()          # every worker reads the initial rows: all updates follow its pull
    merged = base.clone()

    def at(keys):
        return torch.searchsorted(t, keys)

    def add(keys, d):
        merged.index_add_(0, at(keys), d)

    if c["kind"] in ("clock", "access"):
        rows = []
        for w in range(c["workers"]):
            k = batches[0][w]["keys"]
            rows.append(init[k])     # copies: the 32-bit rows themselves
            for i in range(0, k.numel(), 1 << 18):
                add(k[i:i + (1 << 18)], deltas[w][i:i + (1 << 18)].double())
        return {"rows": [None if c.get("relocate") else r.double() for r in rows], "merged": merged[at(back)]}
    del init
    losses = []
    for w in range(c["workers"]):
        b, loss = batches[0][w], 0.0
        step = {"mf": 1 << 16, "complex": 512, "sgns": 256}[c["kind"]]
        for i in range(0, c["batch"], step):
            j = slice(i, min(i + step, c["batch"]))
            if c["kind"] == "mf":
                r = c["rank"]
                U, Wc = base[at(b["rows"][j])], base[at(b["cols"][j])]
                e = b["vals"][j].double() - (U[:, :r] * Wc[:, :r]).sum(1)
                loss = loss + 0.5 * (e * e).sum()
                for k, own, other in (("rows", U, Wc), ("cols", Wc, U)):
                    gr = -e[:, None] * other[:, :r]
                    add(b[k][j], _ada(gr, own[:, r:]) if c["adagrad"] else -LR * gr)
            elif c["kind"] == "complex":
                m, N = c["half"], c["negs"]
                neg = b["negs"].view(-1, N)[j]
                tk = torch.cat([b["tails"][j][:, None], neg], dim=1)                   # true tail, negatives
                H, R, T = base[at(b["heads"][j])], base[at(b["rels"][j])], base[at(tk.reshape(-1))]
                th = [torch.complex(x[:, :m], x[:, m:2 * m]) for x in (H, R, T)]
                h, r, tl = th[0], th[1], th[2].view(-1, 1 + N, m)
                x = h * r
                phi = (x[:, None, :] * tl.conj()).real.sum(2)
                sign = torch.ones(1 + N, device=DEV, dtype=torch.float64)
                sign[0] = -1.0
                loss = loss + _softplus(sign * phi).sum()
                coef = sign * torch.sigmoid(sign * phi)
                S = (coef[:, :, None] * tl).sum(1)
                gh, gr = r.conj() * S, h.conj() * S
                gt = (coef[:, :, None] * x[:, None, :]).reshape(-1, m)
                for keys, gz, own in ((b["heads"][j], gh, H), (b["rels"][j], gr, R), (tk.reshape(-1), gt, T)):
                    add(keys, _ada(torch.cat([gz.real, gz.imag], dim=1), own[:, 2 * m:]))
            else:
                V, N = c["vocab"], c["negs"]
                cen, ctx, neg = b["centres"][j], b["contexts"][j], b["negs"][j]
                toks = torch.cat([ctx[:, :, None], neg], dim=2)
                pres = (ctx != 0xFFFFFFFF)[:, :, None].expand_as(toks)
                # (rows of absent contexts get weight 0: any touched key stands in for theirs)
                ok = torch.where(pres, V + toks, (V + b["contexts"][-1, 0]).expand_as(toks))
                n = cen.numel()
                v, u = base[at(cen)], base[at(ok.reshape(-1))].view(n, -1, c["dim"])
                sc = (u * v[:, None, :]).sum(2)
                sign = torch.ones(1 + N, device=DEV, dtype=torch.float64)
                sign[0] = -1.0
                sign = sign.expand(2 * c["window"], 1 + N).reshape(1, -1)
                p = pres.reshape(n, -1).double()
                loss = loss + (p * _softplus(sign * sc)).sum()
                coef = p * sign * torch.sigmoid(sign * sc)
                add(cen, -LR * (coef[:, :, None] * u).sum(1))
                add(ok.reshape(-1), (-LR * coef[:, :, None] * v[:, None, :]).reshape(-1, c["dim"]))
        losses.append(loss)
    return {"loss": torch.stack(losses), "merged": merged[at(back)]}
