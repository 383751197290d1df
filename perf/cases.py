"""Performance cases of the hash tables: what a program built on this package does with them.

A case is a dict of plain values. ``prepare`` makes its inputs from a seed and the handles a
program keeps (an empty or a built table, a batch with its layout, a pool with its tables);
``run`` is one pass through the package's entry points and returns the find answers, which
depend on the keys, values and queries alone (a table's slot layout does not: keys are
inserted concurrently). Keys are unique, random and never the sentinel 0xFFFFFFFF; arrays are
int32 tensors carrying uint32 bits.

Kinds of cases:
  lookup  a built table answers one batch of queries
  table   a table is built from keys and values, then answers a batch of queries (or, with
          ``separate``, one batch of present keys and one of absent ones)
  host    the same from page-locked host arrays through the host-buffer entry points
  batch   many independent tables of uneven sizes, built and queried by one call
  pool    a served pool of built tables answers a burst of find requests of mixed sizes
"""

import math

import numpy as np
import torch

import paper_2108_07232_gb300 as ght

DEVICE = "cuda"
M32 = 0xFFFFFFFF
SENTINEL = 0xFFFFFFFF


def listed():
    return [
        # a service asks a resident table for a handful of keys: launch and latency only
        dict(name="lookup bcht 2^16 few", kind="lookup", scheme="bcht", keys=1 << 16, load_factor=0.95, queries=300,
             positive=0.7),
        # a small dictionary rebuilt and read at once
        dict(name="table bcht 20k", kind="table", scheme="bcht", keys=20000, load_factor=0.95, queries=40000,
             positive=0.5),
        # the paper's method at its plainest: a million keys, the table fits in the L2
        dict(name="table bcht 2^20", kind="table", scheme="bcht", keys=1 << 20, load_factor=0.9, queries=1 << 20,
             positive=0.5),
        # the scheme sweep's size, one case per scheme at a load factor the scheme is used at
        dict(name="table bcht 2^24", kind="table", scheme="bcht", keys=1 << 24, load_factor=0.95, queries=1 << 24,
             positive=0.5),
        dict(name="table p2bht 2^24", kind="table", scheme="p2bht", keys=1 << 24, load_factor=0.8, queries=1 << 24,
             positive=0.5),
        dict(name="table iht 2^24", kind="table", scheme="iht", keys=1 << 24, load_factor=0.8, queries=1 << 24,
             positive=0.5),
        dict(name="table cuckoo1 2^24", kind="table", scheme="cuckoo1", keys=1 << 24, load_factor=0.8,
             queries=1 << 24, positive=0.5),
        # a membership set of the paper's 50 million keys, mostly asked for absent ones (a filter)
        dict(name="table set 50M", kind="table", scheme="bcht_set", keys=50_000_000, load_factor=0.95,
             queries=50_000_000, positive=0.25),
        # far beyond the L2 and nearly full: build, then present and absent queries (the headline workload)
        dict(name="table bcht 2^28", kind="table", scheme="bcht", keys=1 << 28, load_factor=0.99, queries=1 << 28,
             positive=0.5, separate=True),
        # keys and queries that live in host memory
        dict(name="host bcht 2^24", kind="host", scheme="bcht", keys=1 << 24, load_factor=0.9, queries=1 << 24,
             positive=0.5),
        # many uneven tables at once (one per shard, tenant or column)
        dict(name="batch 512 tables", kind="batch", tables=512, log2_min=10.0, log2_max=20.0, lf_min=0.8, lf_max=0.99,
             queries_per_key=2.0, positive=0.5),
        # a burst of requests against resident tables
        dict(name="pool 32 tables", kind="pool", tables=32, log2_min=16.0, log2_max=22.0, load_factor=0.95,
             requests=128, log2_queries=20.0, positive=0.7),
    ]


LOAD_FACTORS = {"bcht": (0.6, 0.99), "p2bht": (0.6, 0.82), "iht": (0.6, 0.84), "cuckoo1": (0.5, 0.82),
                "bcht_set": (0.6, 0.99), "bcht_lb": (0.6, 0.95)}


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lookup"] * 3 + ["table"] * 9 + ["host"] * 2 + ["batch", "pool"])
    if kind == "batch":
        lo = rng.uniform(9.0, 12.0)
        return dict(kind="batch", tables=_log(rng, 16, 512), log2_min=lo, log2_max=lo + rng.uniform(4.0, 9.0),
                    lf_min=rng.uniform(0.7, 0.85), lf_max=rng.uniform(0.86, 0.99),
                    queries_per_key=rng.uniform(0.5, 2.0), positive=rng.choice([0.1, 0.5, 1.0]))
    if kind == "pool":
        lo = rng.uniform(12.0, 16.0)
        return dict(kind="pool", tables=rng.randint(4, 48), log2_min=lo, log2_max=lo + rng.uniform(2.0, 6.0),
                    load_factor=rng.uniform(0.8, 0.95), requests=_log(rng, 16, 128),
                    log2_queries=rng.uniform(12.0, 20.0), positive=0.7)
    if kind == "lookup":
        scheme = rng.choice(["bcht"] * 3 + ["p2bht", "iht", "cuckoo1", "bcht_set"])
        keys, queries = _log(rng, 1 << 12, 1 << 24), _log(rng, 32, 1 << 20)
    elif kind == "host":
        scheme = rng.choice(["bcht"] * 3 + ["p2bht", "iht", "cuckoo1", "bcht_set"])
        keys = _log(rng, 1 << 14, 1 << 25)
        queries = max(1, int(keys * rng.uniform(0.25, 2.0)))
    else:
        scheme = rng.choice(["bcht"] * 5 + ["p2bht", "iht", "cuckoo1", "bcht_lb"] + ["bcht_set"] * 2)
        keys = _log(rng, 1 << 10, 1 << (27 if scheme in ("bcht", "bcht_set") else 25))
        queries = max(1, int(keys * rng.uniform(0.25, 2.0)))
    lo, hi = LOAD_FACTORS[scheme]
    return dict(kind=kind, scheme=scheme, keys=keys, load_factor=round(rng.uniform(lo, hi), 3), queries=queries,
                positive=rng.choice([0.1, 0.3, 0.5, 0.7, 0.9 if scheme == "bcht_set" else 1.0]))


# --- inputs ---------------------------------------------------------------------


def _generator(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed & 0x7FFFFFFFFFFFFFFF)
    return g


def _words(count, seed):
    """``count`` distinct random 32-bit words without the sentinel, as int32: a bijection of 32-bit
    words (odd multiplications and xor-shifts) of consecutive indices from a seeded start."""
    r = np.random.default_rng(seed)
    start, a, b, c = (int(x) for x in r.integers(0, 1 << 32, 4))
    w = torch.arange(start, start + count + 1, dtype=torch.int64, device=DEVICE)
    w.mul_(a | 1).bitwise_and_(M32)
    for odd, shift in ((b | 1, 16), (c | 1, 15), (0x9E3779B1, 13)):
        w ^= w >> shift
        w.mul_(odd).bitwise_and_(M32)
    w ^= w >> 16
    w = w[w != SENTINEL][:count]
    return w.to(torch.int32)  # keeps the low 32 bits


def _values(count, g):
    """Random 32-bit values without the sentinel."""
    v = torch.randint(-(1 << 31), 1 << 31, (count,), generator=g, device=DEVICE, dtype=torch.int64)
    return v.to(torch.int32).bitwise_and_(-2)  # even, so never all ones


def _table_inputs(case, seed):
    """keys, values, and per query batch (queries, index of its key or -1)."""
    n, q = case["keys"], case["queries"]
    g = _generator(seed)
    separate = case.get("separate", False)
    words = _words(n + q, seed)
    keys, absent = words[:n].contiguous(), words[n:]
    values = _values(n, g)
    at = torch.randint(0, n, (q,), generator=g, device=DEVICE)
    if separate:
        return keys, values, [(keys[at], at), (absent.contiguous(), torch.full_like(at, -1))]
    at[torch.rand(q, generator=g, device=DEVICE) >= case["positive"]] = -1
    return keys, values, [(torch.where(at >= 0, keys[at.clamp(min=0)], absent), at)]


def _sizes(case):
    """Keys and load factor per table of a batch or pool: drawn once per case, not per seed."""
    r = np.random.default_rng(case["tables"])
    sizes = np.exp2(r.uniform(case["log2_min"], case["log2_max"], case["tables"])).astype(np.int64)
    if case["kind"] == "pool":
        return sizes, np.full(case["tables"], case["load_factor"])
    return sizes, r.uniform(case["lf_min"], case["lf_max"], case["tables"])


def _offsets(sizes):
    return np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)


def _segments(case):
    """(table, queries) of each query segment: one per table of a batch, one per request of a pool."""
    sizes, _ = _sizes(case)
    if case["kind"] == "batch":
        return np.arange(case["tables"]), np.maximum(1, np.round(sizes * case["queries_per_key"])).astype(np.int64)
    r = np.random.default_rng(case["requests"] + 1)
    lengths = np.exp2(r.uniform(0.0, case["log2_queries"], case["requests"])).astype(np.int64)
    return r.integers(0, case["tables"], case["requests"]), lengths


def _many_inputs(case, seed):
    """All tables' keys and values, all segments' queries, and the index of each query's key or -1."""
    sizes, _ = _sizes(case)
    table, lengths = _segments(case)
    offs = torch.from_numpy(_offsets(sizes).astype(np.int64)).to(DEVICE)
    n, q = int(sizes.sum()), int(lengths.sum())
    g = _generator(seed)
    words = _words(n + q, seed)
    keys, absent = words[:n].contiguous(), words[n:]
    values = _values(n, g)
    of = torch.repeat_interleave(torch.from_numpy(table).to(DEVICE), torch.from_numpy(lengths).to(DEVICE))
    size = offs[of + 1] - offs[of]
    u = torch.rand(q, generator=g, device=DEVICE, dtype=torch.float64)
    at = torch.minimum((u * size).to(torch.int64), size - 1) + offs[of]
    at[torch.rand(q, generator=g, device=DEVICE) >= case["positive"]] = -1
    return keys, values, torch.where(at >= 0, keys[at.clamp(min=0)], absent), at


# --- the interface ----------------------------------------------------------------


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("lookup", "table", "host"):
        keys, values, batches = _table_inputs(case, seed)
        if case["scheme"] == "bcht_set":
            values = None
        table = ght.HashTable(case["scheme"], case["keys"], case["load_factor"], seed=seed)
        queries = [q for q, _ in batches]
        if kind == "lookup":
            table.build(keys, values)
            return dict(kind=kind, table=table, queries=queries)
        if kind == "host":
            keys, values, *queries = (_pinned(x) for x in (keys, values, *queries))
            outs = [torch.empty_like(q).pin_memory() for q in queries]
            return dict(kind=kind, table=table, keys=keys, values=values, queries=queries, outs=outs)
        return dict(kind=kind, table=table, keys=keys, values=values, queries=queries)
    keys, values, queries, _ = _many_inputs(case, seed)
    sizes, lfs = _sizes(case)
    table, lengths = _segments(case)
    out = torch.empty_like(queries)
    if kind == "batch":
        batch = ght.Batch(sizes, lfs, seed=seed)
        batch.set_layout(_offsets(sizes), _offsets(lengths))
        return dict(kind=kind, batch=batch, keys=keys, values=values, queries=queries, out=out)
    pool = ght.Pool(8 << 30)
    offs = _offsets(sizes).astype(np.int64)
    tickets = [pool.submit_build(int(sizes[t]), float(lfs[t]), seed + t, keys[offs[t]:offs[t + 1]],
                                 values[offs[t]:offs[t + 1]]) for t in range(case["tables"])]
    ids = []
    torch.cuda.synchronize()
    for ticket, table_id in tickets:
        assert pool.wait(ticket)["status"] == 0
        ids.append(table_id)
    cuts = _offsets(lengths).astype(np.int64)
    requests = [(ids[t], queries[cuts[i]:cuts[i + 1]], out[cuts[i]:cuts[i + 1]]) for i, t in enumerate(table)]
    return dict(kind=kind, pool=pool, requests=requests, out=out)


def _pinned(x):
    return None if x is None else torch.empty(x.shape, dtype=x.dtype, pin_memory=True).copy_(x)


def run(state):
    kind = state["kind"]
    if kind == "lookup":
        return [state["table"].find(q) for q in state["queries"]]
    if kind == "table":
        state["table"].build(state["keys"], state["values"])
        return [state["table"].find(q) for q in state["queries"]]
    if kind == "host":
        state["table"].build(state["keys"], state["values"])
        return [state["table"].find(q, out) for q, out in zip(state["queries"], state["outs"])]
    if kind == "batch":
        return state["batch"].run(state["keys"], state["values"], state["queries"], state["out"])
    pool = state["pool"]
    for ticket in [pool.submit_find(t, q, o) for t, q, o in state["requests"]]:
        pool.wait(ticket)
    return state["out"]


def _bytes(keys, load_factor, queries, slot, built):
    """A build reads every key (and value) and writes every slot once; a find reads every query,
    writes every answer, and reads a 128-byte line of the table per query, or the table once where
    that is less."""
    table = keys / load_factor * slot
    build = keys * slot + table if built else 0.0
    return build + 8.0 * queries + min(table, 128.0 * queries)


def work(case):
    if case["kind"] in ("lookup", "table", "host"):
        slot = 4.0 if case["scheme"] == "bcht_set" else 8.0
        total = _bytes(case["keys"], case["load_factor"], case["queries"], slot, case["kind"] != "lookup")
        if case.get("separate", False):
            total += _bytes(case["keys"], case["load_factor"], case["queries"], slot, False)
        return {"bytes": total, "flops": 0.0}
    sizes, lfs = _sizes(case)
    table, lengths = _segments(case)
    asked = np.bincount(table, weights=lengths, minlength=case["tables"])
    built = case["kind"] == "batch"
    return {"bytes": float(sum(_bytes(n, f, q, 8.0, built) for n, f, q in zip(sizes, lfs, asked))), "flops": 0.0}


def exact(case, seed):
    """The definitional answers: the value of a present key (1 in a set), the sentinel (0) otherwise."""
    if case["kind"] in ("lookup", "table", "host"):
        keys, values, batches = _table_inputs(case, seed)
        answers = []
        for _, at in batches:
            if case["scheme"] == "bcht_set":
                answers.append((at >= 0).to(torch.int32))
            else:
                answers.append(torch.where(at >= 0, values[at.clamp(min=0)], torch.full_like(values[:1], -1)))
        return answers
    _, values, _, at = _many_inputs(case, seed)
    return torch.where(at >= 0, values[at.clamp(min=0)], torch.full_like(values[:1], -1))
