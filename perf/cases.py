"""The work that a program has the flow tables do, as cases that can be timed.

A case is a dict of plain values; ``kind`` says which calls one pass makes:

  lookup   one ``FlowTable.lookup`` (``refresh`` > 0: a timers table, one batch per time unit,
           and each hit restarts its flow's timer)
  host     one lookup whose keys and results stay in pinned host memory
  batched  one ``BatchedLookup.launch`` over a burst of keys for each of many tables
  cycle    new flows arrive, are looked up and leave: insert, lookup, delete on one table
  flush    the same insert and delete over many tables at once (the served form's write turns)
  timers   a time step of a table with timers: lookups that refresh, inserts of short-lived
           flows, deletes, and the expire scan that removes the flows whose time has run out

Every pass leaves the table with the flows that it had before, so that passes repeat. Keys are
5-tuples (addresses, ports, TCP or UDP, padding) and values are flow numbers.
"""

from __future__ import annotations

import math

import torch

from paper_1712_09624_gb300 import FlowTable
from paper_1712_09624_gb300 import _ckpp as K
from paper_1712_09624_gb300.batched import BatchedLookup

DEV = "cuda"
SLOTS = 8
CHUNK = 1 << 24  # keys per call when a table is filled
TTL = 1000  # of the flows that stay; each pass of a timers case refreshes them


def listed() -> list[dict]:
    return [
        # one port's small packet burst against a table of a million slots: latency
        {"name": "lookup_burst", "kind": "lookup", "n": 64, "nb": 1 << 17, "lf": 0.9, "neg": 0.2, "refresh": 0},
        # a core's share of traffic on 32M slots at load 0.8 with 20 % unknown flows; ragged sizes
        {"name": "lookup_core", "kind": "lookup", "n": 50_021, "nb": 4_000_037, "lf": 0.8, "neg": 0.2, "refresh": 0},
        # the small configuration: a table that fits in L2
        {"name": "lookup_small", "kind": "lookup", "n": 1 << 20, "nb": 1 << 17, "lf": 0.9, "neg": 0.5, "refresh": 0},
        # the large configuration: 128M slots, batches of 16M keys
        {"name": "lookup_scale", "kind": "lookup", "n": 1 << 24, "nb": 1 << 24, "lf": 0.9, "neg": 0.5, "refresh": 0},
        # a table with timers, nearly all packets of known flows, each restarting its flow's timer
        {"name": "lookup_refresh", "kind": "lookup", "n": 1 << 22, "nb": 6_250_000, "lf": 0.6, "neg": 0.01,
         "refresh": TTL},
        # packets that the host's own memory holds, looked up in place
        {"name": "lookup_host", "kind": "host", "n": 1 << 22, "nb": 1 << 22, "lf": 0.9, "neg": 0.5},
        # many tenants' tables, 1K to 4M slots each, a batch for every one of them in one launch
        {"name": "batched_tables", "kind": "batched", "tables": 512, "jobs": 512, "lo": 32, "hi": 65536,
         "nb_lo": 128, "nb_hi": 1 << 19, "lf": 0.85, "neg": 0.3},
        # one turn of the served form: the bursts of some ports, each for the table of its tenant
        {"name": "batched_turn", "kind": "batched", "tables": 256, "jobs": 48, "lo": 32, "hi": 4096,
         "nb_lo": 1 << 12, "nb_hi": 1 << 17, "lf": 0.8, "neg": 0.3},
        # a few new flows (some packets of one flow) come and go: latency of the write calls
        {"name": "cycle_burst", "kind": "cycle", "n": 64, "nb": 1 << 17, "base": 0.8, "dup": 0.1, "timers": False},
        # the served form's write turn: 32K keys for 256 tables
        {"name": "flush", "kind": "flush", "n": 32768, "tables": 256, "nb_lo": 1 << 12, "nb_hi": 1 << 17, "base": 0.8,
         "dup": 0.05},
        # a million flows come and go on the large table while it is nearly full
        {"name": "cycle_scale", "kind": "cycle", "n": 1 << 20, "nb": 1 << 24, "base": 0.89, "dup": 0.02,
         "timers": False},
        # a time step: flows refreshed, new ones inserted, some deleted, the rest expired by the scan
        {"name": "timers_step", "kind": "timers", "stay": 6_000_000, "new": 1_700_000, "gone": 400_000,
         "nb": 1_500_000, "neg": 0.01},
    ]


def draw(rng) -> dict:
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["lookup", "lookup", "lookup", "host", "batched", "cycle", "cycle", "flush", "timers"])
    if kind == "lookup":
        return {"kind": kind, "n": log(32, 1 << 24), "nb": log(1 << 10, 1 << 24), "lf": round(rng.uniform(0.5, 0.95), 3),
                "neg": round(rng.uniform(0, 1), 3), "refresh": rng.choice([0, 0, TTL])}
    if kind == "host":
        return {"kind": kind, "n": log(32, 1 << 22), "nb": log(1 << 10, 1 << 22), "lf": round(rng.uniform(0.5, 0.95), 3),
                "neg": round(rng.uniform(0, 1), 3)}
    if kind == "batched":
        jobs = log(4, 512)
        return {"kind": kind, "tables": jobs + log(1, 256), "jobs": jobs, "lo": 32, "hi": log(1024, 65536),
                "nb_lo": 128, "nb_hi": log(1 << 10, 1 << 18), "lf": round(rng.uniform(0.5, 0.9), 3),
                "neg": round(rng.uniform(0, 1), 3)}
    if kind == "cycle":
        nb = log(1 << 11, 1 << 23)
        base = round(rng.uniform(0, 0.85), 3)
        n = log(32, min(1 << 21, int((0.92 - base) * SLOTS * nb)))
        return {"kind": kind, "n": n, "nb": nb, "base": base, "dup": round(rng.uniform(0, 0.3), 3),
                "timers": rng.choice([False, True])}
    if kind == "flush":
        tables = log(8, 512)
        return {"kind": kind, "n": log(32, 128 * tables), "tables": tables, "nb_lo": 1 << 11, "nb_hi": log(1 << 12, 1 << 17),
                "base": round(rng.uniform(0.4, 0.8), 3), "dup": round(rng.uniform(0, 0.2), 3)}
    nb = log(1 << 12, 1_500_000)
    stay, new = int(nb * SLOTS * rng.uniform(0.3, 0.5)), int(nb * SLOTS * rng.uniform(0.01, 0.15))
    return {"kind": kind, "stay": stay, "new": new, "gone": int(new * rng.uniform(0.05, 0.5)), "nb": nb,
            "neg": round(rng.uniform(0, 0.2), 3)}


# ------------------------------------------------------------------ inputs
def _gen(seed: int, stream: int) -> torch.Generator:
    g = torch.Generator(device=DEV)
    g.manual_seed((seed * 1_000_003 + stream) & (2**62 - 1))
    return g


def _keys(seed: int, stream: int, n: int) -> torch.Tensor:
    """n 5-tuples: 64 bits of addresses, 32 of ports, a protocol byte, three zero bytes."""
    g = _gen(seed, stream)
    w = torch.empty((n, 2), dtype=torch.int64, device=DEV)
    w[:, 0] = torch.randint(-(2**63), 2**63 - 1, (n,), generator=g, device=DEV)
    r = torch.randint(0, 2**33, (n,), generator=g, device=DEV)
    w[:, 1] = (r & 0xFFFFFFFF) | ((6 + 11 * (r >> 32)) << 32)
    return w.view(torch.uint8).view(n, 16)


def _pick(seed: int, stream: int, n: int, m: int) -> torch.Tensor:
    return torch.randint(0, max(m, 1), (n,), generator=_gen(seed, stream), device=DEV)


def _values(lo: int, hi: int) -> torch.Tensor:
    return torch.arange(lo, hi, dtype=torch.int64, device=DEV)


def _fill(table: FlowTable, keys: torch.Tensor, now: int = 0, ttl: int = 0):
    for lo in range(0, keys.shape[0], CHUNK):
        hi = min(lo + CHUNK, keys.shape[0])
        table.insert(keys[lo:hi], _values(lo, hi), now, ttl)
    table._ws = None  # the next calls' workspace is sized by them


def _spread(stream: int, count: int, lo: int, hi: int) -> list[int]:
    """count whole numbers between lo and hi, spread over their logarithm; the case's own, whatever the seed."""
    u = torch.rand(count, generator=_gen(0, stream), device=DEV, dtype=torch.float64)
    return torch.exp(math.log(lo) + u * math.log(hi / lo)).round().to(torch.int64).clamp(lo, hi).tolist()


def _lookups(case: dict, seed: int, m: int):
    """(flow looked up or -1 for an unknown one), for a batch of lookups over m flows."""
    neg = torch.rand(case["n"], generator=_gen(seed, 3), device=DEV) < case["neg"]
    return torch.where(neg, torch.full((), -1, dtype=torch.int64, device=DEV), _pick(seed, 4, case["n"], m))


def _lookup_keys(seed: int, flow: torch.Tensor, fill: torch.Tensor) -> torch.Tensor:
    fresh = _keys(seed, 2, flow.shape[0])
    return torch.where((flow >= 0)[:, None], fill[flow.clamp(min=0)], fresh).contiguous()


def _answers(flow: torch.Tensor):
    return flow.clamp(min=0), flow >= 0


def _arrivals(case: dict, seed: int, n: int):
    """Which of n new flows each of n packets belongs to: a share ``dup`` of them repeats another's flow."""
    own = _values(0, n)
    again = torch.rand(n, generator=_gen(seed, 6), device=DEV) < case["dup"]
    return torch.where(again, _pick(seed, 7, n, n), own)


def _first_last(flow: torch.Tensor):
    """For each packet, whether it is its flow's first in the batch, and the flow's last packet."""
    n = flow.shape[0]
    i = _values(0, n)
    first = torch.full((n,), n, dtype=torch.int64, device=DEV).scatter_reduce_(0, flow, i, "amin")
    last = torch.full((n,), -1, dtype=torch.int64, device=DEV).scatter_reduce_(0, flow, i, "amax")
    return first[flow] == i, last[flow]


def _status(first: torch.Tensor, yes: int, no: int) -> torch.Tensor:
    return torch.where(first, torch.full((), yes, device=DEV), torch.full((), no, device=DEV)).to(torch.uint8)


# ---------------------------------------------------------------- prepare
def prepare(case: dict, seed: int):
    return globals()["_prepare_" + case["kind"]](case, seed)


def _filled(case: dict, seed: int, flows: int, timers: bool):
    table = FlowTable(case["nb"], timers=timers, seed=seed)
    keys = _keys(seed, 1, flows)
    _fill(table, keys, 0, TTL if timers else 0)
    return table, keys


def _prepare_lookup(case, seed):
    m = int(case["lf"] * SLOTS * case["nb"])
    table, fill = _filled(case, seed, m, case["refresh"] > 0)
    return {"case": case, "table": table, "keys": _lookup_keys(seed, _lookups(case, seed, m), fill), "now": 0}


def _prepare_host(case, seed):
    m = int(case["lf"] * SLOTS * case["nb"])
    table, fill = _filled(case, seed, m, False)
    n = case["n"]
    keys = torch.empty((n, 16), dtype=torch.uint8, pin_memory=True)
    keys.copy_(_lookup_keys(seed, _lookups(case, seed, m), fill))
    return {"case": case, "table": table, "keys": keys, "vals": torch.empty(n, dtype=torch.int64, pin_memory=True),
            "found": torch.empty(n, dtype=torch.bool, pin_memory=True)}


def _many_tables(case, seed, load):
    nbs = _spread(10, case["tables"], case["nb_lo"], case["nb_hi"])
    counts = [int(load * SLOTS * nb) for nb in nbs]
    tables = [FlowTable(nb, seed=seed + t) for t, nb in enumerate(nbs)]
    total = sum(counts)
    fill = _keys(seed, 1, total)
    owner = torch.repeat_interleave(torch.arange(len(nbs), dtype=torch.int32, device=DEV),
                                    torch.tensor(counts, device=DEV), output_size=total)
    return tables, counts, fill, owner


def _fill_many(batch, fill, owner):
    n = min(CHUNK, fill.shape[0])
    ws = torch.empty(K.ckpp_workspace_bytes(n), dtype=torch.uint8, device=DEV)
    status = torch.empty(n, dtype=torch.uint8, device=DEV)
    for lo in range(0, fill.shape[0], CHUNK):
        hi = min(lo + CHUNK, fill.shape[0])
        K.ckpp_batch_insert(batch.handle, fill[lo:hi], owner[lo:hi], _values(lo, hi), status[:hi - lo], ws)


def _jobs(case, seed, counts):
    """Each job's table and size, and each lookup's flow within its table (-1: unknown)."""
    ids = torch.randperm(case["tables"], generator=_gen(seed, 11), device=DEV)[:case["jobs"]].tolist()
    sizes = _spread(12, case["jobs"], case["lo"], case["hi"])
    bound = torch.repeat_interleave(torch.tensor([counts[t] for t in ids], device=DEV), torch.tensor(sizes, device=DEV))
    total = sum(sizes)
    u = torch.rand(total, generator=_gen(seed, 4), device=DEV, dtype=torch.float64)
    flow = torch.minimum((u * bound).to(torch.int64), bound - 1)
    neg = torch.rand(total, generator=_gen(seed, 3), device=DEV) < case["neg"]
    start = [0]
    for c in counts:
        start.append(start[-1] + c)
    first = torch.repeat_interleave(torch.tensor([start[t] for t in ids], device=DEV), torch.tensor(sizes, device=DEV))
    return ids, sizes, torch.where(neg, torch.full((), -1, dtype=torch.int64, device=DEV), first + flow)


def _prepare_batched(case, seed):
    tables, counts, fill, owner = _many_tables(case, seed, case["lf"])
    batch = BatchedLookup(tables, max_jobs=case["jobs"])
    _fill_many(batch, fill, owner)
    ids, sizes, flow = _jobs(case, seed, counts)
    keys = _lookup_keys(seed, flow, fill)
    vals = torch.empty(keys.shape[0], dtype=torch.int64, device=DEV)
    found = torch.empty(keys.shape[0], dtype=torch.bool, device=DEV)
    jobs, at = [], 0
    for t, n in zip(ids, sizes):
        jobs.append((t, keys[at:at + n], vals[at:at + n], found[at:at + n]))
        at += n
    batch.set_jobs(jobs)
    return {"case": case, "batch": batch, "vals": vals, "found": found}


def _prepare_cycle(case, seed):
    m = int(case["base"] * SLOTS * case["nb"])
    table, _ = _filled(case, seed, m, case["timers"])
    n = case["n"]
    keys = _keys(seed, 5, n)[_arrivals(case, seed, n)].contiguous()
    return {"case": case, "table": table, "keys": keys, "values": _values(m, m + n)}


def _prepare_flush(case, seed):
    tables, counts, fill, owner = _many_tables(case, seed, case["base"])
    batch = BatchedLookup(tables, max_jobs=1)
    _fill_many(batch, fill, owner)
    n = case["n"]
    flow = _arrivals(case, seed, n)
    room = torch.tensor([t.capacity for t in tables], dtype=torch.float64, device=DEV)  # busier tables are larger
    ids = torch.multinomial(room, n, replacement=True, generator=_gen(seed, 8)).to(torch.int32)
    return {"case": case, "batch": batch, "keys": _keys(seed, 5, n)[flow].contiguous(), "ids": ids[flow].contiguous(),
            "values": _values(0, n), "inserted": torch.empty(n, dtype=torch.uint8, device=DEV),
            "deleted": torch.empty(n, dtype=torch.uint8, device=DEV),
            "ws": torch.empty(K.ckpp_workspace_bytes(n), dtype=torch.uint8, device=DEV)}


def _prepare_timers(case, seed):
    table, fill = _filled(case, seed, case["stay"], True)
    order = torch.randperm(case["stay"], generator=_gen(seed, 4), device=DEV)
    extra = _keys(seed, 2, int(case["neg"] * case["stay"]))  # unknown flows among the packets
    mix = torch.randperm(case["stay"] + extra.shape[0], generator=_gen(seed, 9), device=DEV)
    packets = torch.cat([fill[order], extra])[mix].contiguous()
    new = _keys(seed, 5, case["new"])
    return {"case": case, "table": table, "packets": packets, "new": new, "gone": new[:case["gone"]].contiguous(),
            "values": _values(case["stay"], case["stay"] + case["new"]), "now": 1}


# -------------------------------------------------------------------- run
def run(state):
    return globals()["_run_" + state["case"]["kind"]](state)


def _run_lookup(s):
    refresh = s["case"]["refresh"]
    if refresh:
        s["now"] += 1
    return s["table"].lookup(s["keys"], s["now"], refresh)


def _run_host(s):
    K.ckpp_bulk_lookup(s["table"].handle, s["keys"], s["vals"], s["found"])
    return s["vals"], s["found"]


def _run_batched(s):
    s["batch"].launch()
    return s["vals"], s["found"]


def _run_cycle(s):
    t, keys = s["table"], s["keys"]
    ttl = TTL if s["case"]["timers"] else 0
    inserted = t.insert(keys, s["values"], 0, ttl)
    vals, found = t.lookup(keys, 0)
    return inserted, vals, found, t.delete(keys, 0)


def _run_flush(s):
    h = s["batch"].handle
    K.ckpp_batch_insert(h, s["keys"], s["ids"], s["values"], s["inserted"], s["ws"])
    K.ckpp_batch_delete(h, s["keys"], s["ids"], s["deleted"], s["ws"])
    return s["inserted"], s["deleted"]


def _run_timers(s):
    t, now = s["table"], s["now"]
    vals, found = t.lookup(s["packets"], now, TTL)
    inserted = t.insert(s["new"], s["values"], now, 3)
    deleted = t.delete(s["gone"], now + 1)
    s["now"] = now + 6
    return vals, found, inserted, deleted, t.expire(now + 5)


# ------------------------------------------------------------------ exact
def exact(case: dict, seed: int):
    """What run returns, from the draws alone: flow numbers, and what a map would answer."""
    kind = case["kind"]
    if kind in ("lookup", "host"):
        return _answers(_lookups(case, seed, int(case["lf"] * SLOTS * case["nb"])))
    if kind == "batched":
        nbs = _spread(10, case["tables"], case["nb_lo"], case["nb_hi"])
        _, _, flow = _jobs(case, seed, [int(case["lf"] * SLOTS * nb) for nb in nbs])
        return _answers(flow)
    if kind in ("cycle", "flush"):
        first, last = _first_last(_arrivals(case, seed, case["n"]))
        inserted = _status(first, K.ST_INSERTED, K.ST_UPDATED)
        deleted = _status(first, K.ST_DELETED, K.ST_NOT_FOUND)
        if kind == "flush":
            return inserted, deleted
        m = int(case["base"] * SLOTS * case["nb"])
        return inserted, last + m, torch.ones_like(first), deleted
    order = torch.randperm(case["stay"], generator=_gen(seed, 4), device=DEV)
    unknown = torch.full((int(case["neg"] * case["stay"]),), -1, dtype=torch.int64, device=DEV)
    mix = torch.randperm(case["stay"] + unknown.shape[0], generator=_gen(seed, 9), device=DEV)
    vals, found = _answers(torch.cat([order, unknown])[mix])
    return (vals, found, torch.full((case["new"],), K.ST_INSERTED, dtype=torch.uint8, device=DEV),
            torch.full((case["gone"],), K.ST_DELETED, dtype=torch.uint8, device=DEV),
            torch.tensor([case["new"] - case["gone"]], device=DEV))


# ------------------------------------------------------------------- work
# What the method reads and writes, whatever the layout: a bucket's lookup fields and an entry
# (key and value) are 32 bytes each; a key is 16 bytes, a value 8, a flag or status 1.
def _lookup_bytes(n, neg):
    return n * (16 + 9 + 32 + 32 * (1 - neg))


def _insert_bytes(n):
    return n * (16 + 8 + 1 + 32 + 32 + 32)  # the bucket's fields read and written, the entry written


def _delete_bytes(n):
    return n * (16 + 1 + 32 + 32 + 32)  # the bucket's fields read and written, the entry read


def work(case: dict) -> dict:
    kind = case["kind"]
    if kind in ("lookup", "host"):
        b = _lookup_bytes(case["n"], case["neg"])
    elif kind == "batched":
        lo, hi = case["lo"], case["hi"]
        b = _lookup_bytes(case["jobs"] * ((hi - lo) / math.log(hi / lo) if hi > lo else lo), case["neg"])
    elif kind == "cycle":
        b = _insert_bytes(case["n"]) + _lookup_bytes(case["n"], 0) + _delete_bytes(case["n"])
    elif kind == "flush":
        b = _insert_bytes(case["n"]) + _delete_bytes(case["n"])
    else:
        b = (_lookup_bytes(case["stay"] * (1 + case["neg"]), case["neg"]) + _insert_bytes(case["new"]) +
             _delete_bytes(case["gone"]) + 64 * case["nb"])
    return {"bytes": float(b), "flops": 0.0}
