"""Performance cases of the GF(2) encoder-learning path, through the binding's public calls.

A case is a dict of plain values; ``kind`` says what a pass does:

* ``learn``   a store forgets its state and learns a batch (or a sequence of incremental batches)
              resident on the device, solves every affine map and hands out the learned state:
              what a training run does with its corpus.
* ``encode``  queries resident on the device go through the span check and the learned maps, with or
              without the epilogue that merges scheduler control and opaque bits: assembling code.
* ``pool``    the bases of groups of contexts are merged into one map per group: what follows
              training, before the maps are stored.
* ``host``    a corpus and queries in page-locked host memory are learned and encoded from there:
              the first pass over data that was just parsed.

The corpora follow the package's seeded synthetic workloads (``workloads``): field-structured operand
features with duplicates and a few contradictions, parsed 64-bit values of low rank, and dense
uniform bits (the last two made on the device, which is quicker).  Every output is a set of bits that
has one right value, so the tolerance is "exact".
"""
import ctypes
import math

import numpy as np
import torch

from paper_2608_20532_gb300 import binding, workloads

SHAPE_SEED = 20260000  # widths and row counts of a case


def listed():
    return [
        # one kernel's worth of new encodings: every launch of the call is in its latency
        dict(name="learn-256", kind="learn", corpus="regs", contexts=256, n_min=48, n_max=48, rows=200, sigma=0.0,
             rows_max=200, dup=0.3, contra=3, batches=1, raw=False),
        # one library's corpus: contexts of uneven size, half of the rows repeated
        dict(name="learn-4096", kind="learn", corpus="fields", contexts=4096, n_min=32, n_max=128, rows=300, sigma=1.2,
             rows_max=20000, dup=0.5, contra=20, batches=1, raw=False),
        # the joint corpus of one architecture: heavy-tailed contexts, most rows repeated
        dict(name="learn-77926", kind="learn", corpus="fields", contexts=77926, n_min=16, n_max=256, rows=500,
             sigma=1.2, rows_max=200000, dup=0.85, contra=0, batches=1, raw=False),
        # operands as parsed 64-bit values: wide rows of low rank
        dict(name="learn-parsed", kind="learn", corpus="parsed", contexts=10000, group=8, raw=False),
        # dense wide features streamed in batches: contexts that reach full rank and are then checked
        dict(name="stream-dense", kind="learn", corpus="dense", contexts=64, n_min=1024, n_max=1024, rows=131072,
             sigma=0.0, rows_max=131072, dup=0.0, contra=8, batches=2, raw=False),
        # a learned store kept up to date: small batches for every context, call after call
        dict(name="stream-small", kind="learn", corpus="fields", contexts=4096, n_min=80, n_max=80, rows=256, sigma=0.0,
             rows_max=256, dup=0.0, contra=4, batches=8, raw=False),
        # the held-out queries of a small store (100 a context, half outside the span)
        dict(name="encode-25600", kind="encode", corpus="regs", contexts=256, n_min=48, n_max=48, rows=200, dup=0.3,
             queries=25600, zipf=0.0, out=0.5, epilogue=False, raw=False),
        # one library assembled: evenly used contexts, full words with control and opaque bits
        dict(name="encode-1M", kind="encode", corpus="fields", contexts=4096, n_min=32, n_max=128, rows=200, dup=0.3,
             queries=1_000_000, zipf=0.0, out=0.05, epilogue=True, raw=False),
        # all code of one architecture assembled: a few contexts take most of the queries
        dict(name="encode-10M", kind="encode", corpus="fields", contexts=77926, n_min=16, n_max=256, rows=150, dup=0.3,
             queries=10_000_000, zipf=1.1, out=0.05, epilogue=False, raw=False),
        # exact contexts merged into one map per group
        dict(name="pool-10000", kind="pool", corpus="parsed", contexts=10000, group=8, raw=False),
        # a corpus that arrives from the host, learned and encoded in one go
        dict(name="host-10000", kind="host", corpus="fields", contexts=10000, n_min=16, n_max=256, rows=500, sigma=1.2,
             rows_max=200000, dup=0.85, contra=0, batches=1, queries=1_000_000, zipf=1.1, out=0.05, raw=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["learn", "learn", "learn", "stream", "encode", "encode", "parsed", "pool", "host"])
    if kind in ("parsed", "pool"):
        return dict(kind="learn" if kind == "parsed" else "pool", corpus="parsed", contexts=_log_int(rng, 100, 10000),
                    group=rng.randint(2, 16), raw=False)
    if kind == "stream":  # equal contexts, a multiple of the batch each
        batches = rng.randint(2, 8)
        if rng.random() < 0.5:
            n, dense = rng.randint(200, 1024), True
            contexts = _log_int(rng, 8, 128)
            per = _log_int(rng, 64, max(65, 4_000_000 // (contexts * batches)))
        else:
            n, dense = rng.randint(24, 256), False
            contexts = _log_int(rng, 64, 10000)
            per = _log_int(rng, 8, max(9, 4_000_000 // (contexts * batches)))
        return dict(kind="learn", corpus="dense" if dense else "fields", contexts=contexts, n_min=n, n_max=n,
                    rows=per * batches, sigma=0.0, rows_max=per * batches, dup=0.0,
                    contra=rng.randint(0, max(1, contexts // 200)), batches=batches, raw=rng.random() < 0.3)
    n_lo = rng.randint(16, 128)
    n_hi = rng.randint(n_lo, 256)
    base = dict(kind=kind, corpus="fields", n_min=n_lo, n_max=n_hi, raw=rng.random() < 0.25)
    if kind in ("learn", "host"):
        most = 20_000_000 if kind == "learn" else 8_000_000
        sigma = round(rng.uniform(0.2, 1.3), 3)
        contexts = _log_int(rng, 16, 60000 if kind == "learn" else 20000)
        rows = _log_int(rng, 30, min(5000, max(31, int(most / contexts / math.exp(0.5 * sigma * sigma)))))
        base.update(contexts=contexts, rows=rows, sigma=sigma, rows_max=min(200000, 200 * rows),
                    dup=round(rng.uniform(0.0, 0.95), 3), batches=1)
        # a contradiction takes the place of a repeated row
        base["contra"] = rng.randint(0, contexts // 100) if base["dup"] > 0.1 else 0
    else:
        base.update(contexts=_log_int(rng, 16, 60000), rows=150, dup=0.3, epilogue=rng.random() < 0.3)
    if kind != "learn":
        base.update(queries=_log_int(rng, 100, 6_000_000 if kind == "encode" else 1_000_000),
                    zipf=rng.choice([0.0, round(rng.uniform(0.6, 1.3), 3)]), out=round(rng.uniform(0.0, 0.5), 3))
    return base


def _generate(case, seed):
    """The field-structured corpus of a case and, for the kinds that encode, its queries."""
    layout = workloads.LAYOUT_REGS_IMM16_ONEHOT if case["corpus"] == "regs" else workloads.LAYOUT_CYCLIC_FIELDS
    cfg = dict(num_ctx=case["contexts"], layout=layout, dup_frac=case["dup"], density=0.05,
               n_contra=case.get("contra", 0))
    if case["n_min"] == case["n_max"]:
        cfg["n_fixed"] = case["n_min"]
    elif case["n_min"] == 16 and case["n_max"] == 256:  # the joint corpus: widths cluster at 64 bits
        cfg.update(n_min=16, n_max=256, n_median=64, n_sigma=0.6)
    else:
        cfg.update(n_min=case["n_min"], n_max=case["n_max"])
    if case.get("sigma", 0.0) > 0:
        cfg.update(rows_median=case["rows"], rows_sigma=case["sigma"], rows_max=case["rows_max"])
    else:
        cfg["rows_fixed"] = case["rows"]
    if case.get("batches", 1) > 1:
        cfg["batch_rows"] = case["rows"] // case["batches"]
    if "queries" in case:
        cfg["queries"] = dict(ctx_mode=1, count=case["queries"], zipf_s=case["zipf"], out_frac=case["out"])
    return _fill(cfg, seed)


def _fill(cfg, seed):
    """``workloads.generate`` with the widths and row counts of the case (a fixed seed) and the rows
    of ``seed``: a case has one shape whatever its inputs."""
    lib, p, C, ptr = workloads._load(), workloads._params(cfg), cfg["num_ctx"], workloads._ptr
    by = ctypes.byref(p)
    n_bits, fresh, dups = np.zeros(C, np.int32), np.zeros(C, np.int64), np.zeros(C, np.int64)
    contra, two = np.zeros(C, np.uint8), np.zeros(C, np.uint8)
    if lib.f2gen_plan(by, SHAPE_SEED, ptr(n_bits), ptr(fresh), ptr(dups), ptr(contra), ptr(two)) != 0:
        raise ValueError("invalid workload parameters")
    rows, W = fresh + dups, (n_bits.astype(np.int64) + 31) // 32
    per = cfg.get("batch_rows", 0)
    if per:  # batch-major, equal contexts
        row = np.arange(C + 1, dtype=np.int64) * per
        batches = [(i * C * per + row, (i * C * per + row[:-1]) * W[0]) for i in range(int(rows[0]) // per)]
    else:
        batches = [(np.concatenate([[0], np.cumsum(rows)]), np.concatenate([[0], np.cumsum((rows * W)[:-1])]))]
    x, y = np.zeros(int((rows * W).sum()), np.uint32), np.zeros((int(rows.sum()), 4), np.uint32)
    A, b = np.zeros((int(n_bits.sum()), 4), np.uint32), np.zeros((C, 4), np.uint32)
    a_off = np.concatenate([[0], np.cumsum(n_bits[:-1].astype(np.int64))])
    pos, bit = np.full(C, -1, np.int64), np.full(C, -1, np.int32)
    (row_off, x_off) = batches[0]
    if lib.f2gen_fill(by, seed, ptr(n_bits), ptr(fresh), ptr(dups), ptr(contra), ptr(two), ptr(row_off), ptr(x_off),
                      ptr(x), ptr(y), ptr(A), ptr(a_off), ptr(b), ptr(pos), ptr(bit), workloads._threads()) != 0:
        raise MemoryError("workload fill failed")
    wl = workloads.Workload(name="case", params=dict(cfg), seed=seed, n_bits=n_bits, rows=rows, fresh=fresh, dups=dups,
                            contra=contra, two_stream=two, row_off=row_off, x_off=x_off, x=x, y=y, a_off=a_off, A=A,
                            b=b, contra_pos=pos, contra_bit=bit, batches=batches)
    if "queries" in cfg:
        wl.queries = workloads.make_queries(wl, cfg["queries"], seed)
    return wl


def _dense(case, seed, dev):
    """Uniform features, a planted dense map and, in some contexts, one repeated row with a flipped
    bit: n_bits and the batches (row_off, x, x_off, y), batch-major, equal contexts."""
    C, n, T, nb = case["contexts"], case["n_min"], case["rows"], case["batches"]
    W, per = (n + 31) // 32, T // nb
    g = torch.Generator(device=dev).manual_seed(seed)

    def words(*shape):
        return torch.randint(-2 ** 31, 2 ** 31, shape, dtype=torch.int64, device=dev, generator=g).to(torch.int32)

    x = words(nb, C, per, W)
    if n % 32:
        x[..., W - 1] &= (1 << (n % 32)) - 1
    y = torch.empty((nb, C, per, 4), dtype=torch.int32, device=dev)
    bit = torch.arange(32, device=dev, dtype=torch.int32)
    weight = torch.ones(32, dtype=torch.int64, device=dev) << torch.arange(32, device=dev)
    for c in range(C):
        A = torch.randint(0, 2, (32 * W, 128), device=dev, generator=g).half()
        b = torch.randint(0, 2, (128,), device=dev, generator=g)
        for i in range(nb):
            xb = ((x[i, c].unsqueeze(-1) >> bit) & 1).reshape(per, 32 * W).half()
            yb = ((xb @ A).to(torch.int64) + b) & 1  # sums of at most 1024 ones: exact
            y[i, c] = (yb.reshape(per, 4, 32) * weight).sum(-1).to(torch.int32)
    rng = np.random.default_rng(seed)
    for c in rng.choice(C, min(C, case["contra"]), replace=False):
        i, r = int(rng.integers(nb)), int(rng.integers(1, per))
        x[i, c, r], y[i, c, r] = x[i, c, r - 1].clone(), y[i, c, r - 1].clone()
        y[i, c, r, 0] ^= 1
    x, y = x.reshape(-1), y.reshape(-1, 4)
    row = torch.arange(C + 1, dtype=torch.int64, device=dev) * per
    batches = [(i * C * per + row, x, (i * C * per + row[:-1]) * W, y) for i in range(nb)]
    return np.full(C, n, np.int32), batches


def _parsed(case, seed, dev):
    """Contexts of k int64 operand values (64k feature bits) whose rows span few dimensions: an offset
    and a subset of one-bit generators a row; groups of contexts share k and the planted map.  Sizes
    and ranks as in ``workloads.PARSED_LOWRANK``: n_bits and the one batch."""
    p = workloads.PARSED_LOWRANK
    C, gs = case["contexts"], case["group"]
    rng = np.random.default_rng(SHAPE_SEED)
    k = np.repeat(rng.integers(p["k_min"], p["k_max"] + 1, (C + gs - 1) // gs), gs)[:C]
    sigma = math.log(p["rank_p95"] / p["rank_median"]) / 1.6449
    gens = np.clip(np.rint(np.exp(rng.normal(math.log(p["rank_median"]), sigma, C))), 1, 64).astype(np.int64) - 1
    T = np.rint((gens + 1) * p["rows_per_rank"] * np.exp(rng.normal(0.0, 0.5, C))).astype(np.int64)
    T = np.clip(T, np.maximum(gens + 1, 2), p["rows_max"])
    K, G, R = int(k.max()), int(gens.max()), int(T.sum())
    row_off = np.concatenate([[0], np.cumsum(T)])
    x_off = np.concatenate([[0], np.cumsum(2 * T * k)[:-1]])
    rng = np.random.default_rng(seed)
    # generator j of a context flips one bit of one value: low-order, mid-order or the sign
    value = rng.integers(0, k[:, None], (C, max(G, 1)))
    u = rng.random((C, max(G, 1)))
    bit = np.where(u < 0.6, rng.integers(0, 8, u.shape), np.where(u < 0.95, rng.integers(8, 32, u.shape), 63))
    off = rng.integers(0, 256, (C, K)) * np.where(rng.random((C, K)) < 0.1, -1, 1)
    g = torch.Generator(device=dev).manual_seed(seed)

    def up(a):
        return torch.from_numpy(np.ascontiguousarray(a)).to(dev)

    ng = (C + gs - 1) // gs
    A = (torch.rand((ng, K * 64, 4, 32), device=dev, generator=g) < p["density"]).to(torch.int64)
    A = (A << torch.arange(32, device=dev)).sum(-1)  # 32-bit words in int64, added as planted columns
    group = up(np.arange(C) // gs)
    value, bit = up(value), up(bit)
    word_of = A[group[:, None], 64 * value + bit]    # [C, G, 4]
    ctx = torch.repeat_interleave(torch.arange(C, device=dev), up(T))
    xv = up(off)[ctx]
    bits = (up(off).unsqueeze(-1) >> torch.arange(64, device=dev)) & 1
    y_off = torch.randint(0, 2 ** 32, (ng, 4), dtype=torch.int64, device=dev, generator=g)[group]
    for v in range(K):  # the offset's own word: its set bits' columns, one value at a time
        for b in range(64):
            y_off = y_off ^ (A[group, 64 * v + b] * (bits[:, v, b] * up((v < k).astype(np.int64)))[:, None])
    y = y_off[ctx]
    left = up(gens)
    rows = torch.arange(R, device=dev)
    for j in range(G):
        rows = rows[left[ctx[rows]] > j]
        on = rows[torch.rand(len(rows), device=dev, generator=g) < 0.5]
        c = ctx[on]
        xv[on, value[c, j]] ^= torch.ones_like(c) << bit[c, j]
        y[on] ^= word_of[c, j]
    rng_c = rng.choice(C, max(1, C // 500), replace=False)
    at = up(row_off[rng_c] + 1)
    xv[at], y[at] = xv[at - 1], y[at - 1]            # a repeat of the row before with one flipped bit
    y[at, 0] ^= 1
    keep = torch.arange(K, device=dev)[None, :] < up(k)[ctx][:, None]
    x = xv[keep].view(torch.int32)
    return (64 * k).astype(np.int32), [(up(row_off), x, up(x_off), y.to(torch.int32))]


def _device():
    return torch.device("cuda", torch.cuda.current_device())


def _pinned(a):
    return torch.from_numpy(a.view(np.int32) if a.dtype == np.uint32 else a).pin_memory()


def prepare(case, seed):
    dev = _device()

    def up(a):
        return binding.to_device(a, dev)

    wl = None
    if case["corpus"] == "dense":
        n_bits, batches = _dense(case, seed, dev)
    elif case["corpus"] == "parsed":
        n_bits, batches = _parsed(case, seed, dev)
    else:
        wl = _generate(case, seed)
        n_bits = wl.n_bits
    store = binding.Store(n_bits, raw=case["raw"], device=dev)
    s = dict(kind=case["kind"], store=store)
    if case["kind"] == "host":
        q = wl.queries
        s["rows"] = tuple(_pinned(a) for a in (wl.row_off, wl.x, wl.x_off, wl.y))
        s["ctx_id"], s["x"] = _pinned(q.ctx_id), _pinned(q.x)
        s["y"] = torch.empty((len(q.ctx_id), 4), dtype=torch.int32).pin_memory()
        s["in_span"] = torch.empty(len(q.ctx_id), dtype=torch.uint8).pin_memory()
        return s
    if wl is not None:
        x, y = up(wl.x), up(wl.y)
        batches = [(up(ro), x, up(xo), y) for ro, xo in wl.batches]
    if case["kind"] == "learn":
        s["batches"] = batches
        return s
    for b in batches:  # a learned store
        store.learn(*b)
    torch.cuda.synchronize()
    if case["kind"] == "pool":
        gs = case["group"]
        s["group_of"] = (np.arange(case["contexts"]) // gs).astype(np.int32)
        s["groups"] = int(s["group_of"][-1]) + 1
        # learned output bits of each context; one group in eight mixes two masks
        rng = np.random.default_rng(seed)
        mask = np.repeat(rng.integers(0, 2 ** 32, (s["groups"], 4), dtype=np.uint64).astype(np.uint32), gs,
                         axis=0)[:case["contexts"]].copy()
        mask[::8 * gs] ^= 1
        s["out_mask"] = mask
        return s
    s["ctx_id"], s["x"] = up(wl.queries.ctx_id), up(wl.queries.x)
    if case["epilogue"]:
        rng = np.random.default_rng(seed)
        Q, C = case["queries"], case["contexts"]
        s["sched"] = up(rng.integers(0, 1 << 17, Q, dtype=np.int64).astype(np.int32))
        s["state"] = up(rng.integers(-2 ** 31, 2 ** 31, (Q, 4), dtype=np.int64).astype(np.int32))
        opaque = np.zeros((C, 4), np.int32)  # bits 122 and 124 of one context in sixteen
        opaque[::16, 3] = (1 << 26) | (1 << 28)
        s["opaque"] = up(opaque)
    return s


def run(s):
    store = s["store"]
    if s["kind"] == "learn":
        store.reset()
        for b in s["batches"]:
            store.learn(*b)
        return dict(store.basis(), W=store.solve())
    if s["kind"] == "encode":
        y, ok = store.encode(s["ctx_id"], s["x"])
        if "sched" in s:
            store.encode_epilogue(s["ctx_id"], ok, y, sched=s["sched"], state=s["state"], opaque_mask=s["opaque"])
        return dict(y=y, in_span=ok)
    if s["kind"] == "pool":
        merged, mask_ok = store.merge(s["group_of"], s["groups"], out_mask=s["out_mask"])
        return dict(merged.basis(), mask_ok=mask_ok)
    store.reset()
    store.learn_host(*s["rows"])
    W = store.solve()
    y, ok = store.encode_host(s["ctx_id"], s["x"], s["y"], s["in_span"])
    return dict(W=W, y=y, in_span=ok)


def _mean_rows(case):
    if case.get("sigma", 0.0) > 0:
        return case["rows"] * math.exp(0.5 * case["sigma"] ** 2)
    return round(case["rows"] * (1.0 + case["dup"]))


def work(case):
    """Bytes of the rows read (packed features and word), of the learned state and maps written and,
    where queries are encoded, of the queries and their words; the arithmetic is XOR on bits."""
    C = case["contexts"]
    if case["corpus"] == "parsed":  # k in [2, 8] values of 64 bits; about 200 rows a rank, mean rank 6.1
        n, rows, rank = 320.0, 1360.0, 6.1
    else:
        n = 76.0 if (case["n_min"], case["n_max"]) == (16, 256) else 0.5 * (case["n_min"] + case["n_max"])
        rows, rank = _mean_rows(case), None
    d = n + (0 if case["raw"] else 1)
    basis = C * d * (16 + d / 8)  # words and feature rows of every slot
    total = 0.0
    if case["kind"] == "pool":
        total += C * rank * (16 + d / 8) + basis / case["group"]
    if case["kind"] in ("learn", "host"):
        total += C * rows * (n / 8 + 16) + C * d * 16
    if case["kind"] == "learn":
        total += basis
    if "queries" in case:
        total += case["queries"] * (4 + n / 8 + 16 + 1) + min(C, case["queries"]) * d * (16 + d / 8)
        if case.get("epilogue"):
            total += case["queries"] * (4 + 16)
    return {"bytes": total, "flops": 0}


def tolerance(case):
    return "exact"


def exact(case, seed):
    """Whole bits on every path: there is no rounding to measure against a wider type."""
    return None
