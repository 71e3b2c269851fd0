"""The work that users of the Hive tables have them do, as cases to measure.

Every case goes through the package's public Python entry points on tables
filled with seeded unique 32-bit keys.  A case is a dict of plain values:

* ``find``    lookups on a fixed table (device tensors, or pinned host
              buffers with ``host``), uniform or Zipf(0.99) over the live keys;
* ``mixed``   two mixed batches on a fixed table, the second undoing the first,
              so that a pass leaves the table's contents as they were
              (``fused``: the single-kernel form);
* ``plain``   empty a table, insert, find, erase half, find again;
* ``build``   empty a table and bulk-load it in two batches, the second one
              mixing new keys with keys to overwrite;
* ``stream``  a resizable table taken up by mixed batches and down again;
* ``multi``   two multi-table steps (the second undoes the first) over many
              tables, fixed or resizable, waiting or asynchronous;
* ``set32``   a set of 32-bit keys in 4-byte entries: empty, insert, find,
              erase half, find again.

Key, value and batch generation is in this file; the results of every op
follow from how the batches are made, which is what ``exact`` returns.
"""
import math

import torch

from paper_2510_15095_gb300 import hive

INSERT, FIND, ERASE = 0, 1, 2
ST_INSERTED, ST_REPLACED, ST_ERASED, ST_NOT_FOUND, ST_FOUND = 0, 1, 2, 3, 4
M32 = 0xFFFFFFFF
DEV = "cuda"


def listed():
    return [
        # a service looks up one request's worth of ids in a small table
        {"name": "find_point", "kind": "find", "slots": 1 << 16, "bucket_slots": 32, "load": 80,
         "n": 256, "hit": 90, "zipf": False, "host": False},
        # a small update-and-lookup batch on a mid-size table
        {"name": "mixed_small", "kind": "mixed", "slots": 1 << 20, "bucket_slots": 32, "load": 80,
         "n": 4096, "ins": 50, "erase": 25, "fused": False},
        # the same kind of batch in the single-kernel mode, at an ordinary size
        {"name": "fused_mid", "kind": "mixed", "slots": 1 << 24, "bucket_slots": 32, "load": 90,
         "n": 1000003, "ins": 25, "erase": 25, "fused": True},
        # one table of 2^20 slots through its whole life (L2-resident)
        {"name": "plain_2e20", "kind": "plain", "slots": 1 << 20, "bucket_slots": 32, "load": 80},
        # lookups, half of them present, on a full table of 2^26 slots
        {"name": "find_2e26", "kind": "find", "slots": 1 << 26, "bucket_slots": 32, "load": 95,
         "n": 1 << 26, "hit": 50, "zipf": False, "host": False},
        # skewed lookups whose queries and answers sit in pinned host memory
        {"name": "find_host_zipf", "kind": "find", "slots": 1 << 24, "bucket_slots": 16,
         "load": 85, "n": (1 << 22) + 77, "hit": 90, "zipf": True, "host": True},
        # bulk load of 2^26 slots to 95%
        {"name": "build_2e26", "kind": "build", "slots": 1 << 26, "bucket_slots": 32, "load": 95},
        # a large mixed batch on a full table of 2^26 slots
        {"name": "mixed_2e24", "kind": "mixed", "slots": 1 << 26, "bucket_slots": 16, "load": 95,
         "n": 1 << 24, "ins": 25, "erase": 25, "fused": False},
        # a resizable table through a stream of 40/20/40 batches, up and down
        {"name": "stream_2e22", "kind": "stream", "slots": 1 << 20, "bucket_slots": 32,
         "n": 1 << 22, "batches": 3},
        # many independent fixed tables serviced by one captured batch
        {"name": "multi_256", "kind": "multi", "tables": 256, "cap_lo": 10, "cap_hi": 22,
         "ops_lo": 6, "ops_hi": 18, "ins": 50, "erase": 25, "bucket_slots": 16,
         "resizable": False, "asynchronous": False},
        # a serving step: requests of uneven size against growing tables
        {"name": "serve_64", "kind": "multi", "tables": 64, "cap_lo": 16, "cap_hi": 20,
         "ops_lo": 0, "ops_hi": 14, "ins": 40, "erase": 20, "bucket_slots": 16,
         "resizable": True, "asynchronous": True},
        # a set of 32-bit keys: membership tests and churn
        {"name": "set_2e25", "kind": "set32", "slots": 1 << 25, "load": 90},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["find", "find", "mixed", "mixed", "plain", "build", "stream", "multi",
                       "multi", "set32"])
    bs = rng.choice([16, 32])
    if kind == "find":
        slots = _log_uniform(rng, 1 << 12, 1 << 26)
        host = rng.random() < 0.25
        return {"kind": kind, "slots": slots, "bucket_slots": bs, "load": rng.randint(50, 95),
                "n": _log_uniform(rng, 64, 1 << (23 if host else 26)), "hit": rng.randint(10, 100),
                "zipf": rng.random() < 0.4, "host": host}
    if kind == "mixed":
        slots = _log_uniform(rng, 1 << 14, 1 << 26)
        ins = rng.randint(10, 50)
        n = _log_uniform(rng, 64, max(65, min(slots // 4, 1 << 24)))
        # a batch's new keys (at most 2/5 of it) keep the load at 95% or below
        load = min(rng.randint(50, 95), 94 - 40 * n // slots)
        return {"kind": kind, "slots": slots, "bucket_slots": bs, "load": load, "n": n, "ins": ins,
                "erase": min(ins, rng.randint(5, 25)), "fused": rng.random() < 0.3}
    if kind == "plain":
        return {"kind": kind, "slots": _log_uniform(rng, 1 << 12, 1 << 23), "bucket_slots": bs,
                "load": rng.randint(50, 95)}
    if kind == "build":
        return {"kind": kind, "slots": _log_uniform(rng, 1 << 14, 1 << 26), "bucket_slots": bs,
                "load": rng.randint(50, 95)}
    if kind == "stream":
        return {"kind": kind, "slots": _log_uniform(rng, 1 << 16, 1 << 20), "bucket_slots": bs,
                "n": _log_uniform(rng, 1 << 10, 1 << 22), "batches": rng.randint(1, 3)}
    if kind == "multi":
        lo = rng.randint(0, 8)
        cap = rng.randint(10, 16)
        res = rng.random() < 0.5
        return {"kind": kind, "tables": rng.randint(8, 256), "cap_lo": cap,
                "cap_hi": cap + rng.randint(2, 6), "ops_lo": lo, "ops_hi": lo + rng.randint(4, 10),
                "ins": rng.randint(25, 50), "erase": rng.randint(10, 25), "bucket_slots": bs,
                "resizable": res, "asynchronous": res and rng.random() < 0.5}
    return {"kind": kind, "slots": _log_uniform(rng, 1 << 14, 1 << 25),
            "load": rng.randint(50, 95)}


# ---- keys, values, batches ---------------------------------------------------

def _mix(x, seed):
    """A bijection of 32-bit words held in int64."""
    s = (seed * 2654435761 + 0x9E3779B9) & M32
    x = ((x ^ s) * 0x2C1B3C6D) & M32
    x = x ^ (x >> 15)
    x = (x * 0x297A2D39) & M32
    x = x ^ (x >> 16)
    x = ((x + s) * 0x85EBCA6B) & M32
    return x ^ (x >> 13)


def _key_of(ids, seed):
    """The keys of stream positions `ids` (int64).  The two reserved words are
    swapped for the keys of two positions that no case uses."""
    k = _mix(ids, seed)
    for i, word in enumerate((M32, M32 - 1)):
        spare = _mix(torch.full((1,), M32 - 5 - i, dtype=torch.int64, device=ids.device), seed)
        k = torch.where(k == word, spare, k)
    return k


def _val_of(keys, seed):
    x = (keys + seed * 40503 + 0x9E3779B9) & M32
    x = ((x ^ (x >> 16)) * 0x85EBCA6B) & M32
    x = ((x ^ (x >> 13)) * 0xC2B2AE35) & M32
    return x ^ (x >> 16)


def _i32(x):
    """Unsigned 32-bit words held in int64, as int32 storage."""
    return (x - ((x >> 31) << 32)).to(torch.int32)


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 13)
    return g


def _iota(lo, hi):
    return torch.arange(lo, hi, dtype=torch.int64, device=DEV)


def _pick(n, items, zipf, g):
    """`n` positions in [0, items): uniform, or Zipf(0.99) by rank."""
    u = torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    if not zipf:
        return (u * items).to(torch.int64).clamp_(0, items - 1)
    e = 1.0 - 0.99
    r = ((float(items + 1) ** e - 1.0) * u + 1.0) ** (1.0 / e)
    return (r.to(torch.int64) - 1).clamp_(0, items - 1)


ABSENT = 3 << 30  # stream positions from here on are never inserted


def _batch(seed, g, new, gone, swap, keep, n_find, zipf, back):
    """One mixed batch over stream positions: inserts `new`, erases `gone`,
    overwrites the values of `swap` (`back`: with their first values again),
    and finds among `keep` (one in eight absent).  Returns inputs and results."""
    n_abs = n_find // 8
    hits = keep[_pick(n_find - n_abs, keep.numel(), zipf, g)] if keep.numel() else keep
    miss = ABSENT + _pick(n_find - hits.numel(), 1 << 28, False, g)
    parts = [(new, INSERT, ST_INSERTED), (swap, INSERT, ST_REPLACED), (gone, ERASE, ST_ERASED),
             (hits, FIND, ST_FOUND), (miss, FIND, ST_NOT_FOUND)]
    ids = torch.cat([p[0] for p in parts])
    ops = torch.cat([torch.full((p[0].numel(),), p[1], dtype=torch.uint8, device=DEV)
                     for p in parts])
    st = torch.cat([torch.full((p[0].numel(),), p[2], dtype=torch.uint8, device=DEV)
                    for p in parts])
    order = torch.randperm(ids.numel(), generator=g, device=DEV)
    ids, ops, st = ids[order], ops[order], st[order]
    keys = _key_of(ids, seed)
    first = _val_of(keys, seed)
    zero = torch.zeros_like(first)
    other = first if back else first ^ 0x5A5A5A5A
    vals = torch.where(st == ST_REPLACED, other, torch.where(ops == INSERT, first, zero))
    want = torch.where(st == ST_FOUND, first, zero)
    return {"ops": ops, "keys": _i32(keys), "vals": _i32(vals), "want": _i32(want), "st": st}


def _pair(seed, g, live, new0, n, ins, erase, zipf=False):
    """A batch and the batch that undoes it, for a table holding the stream
    positions `live`; inserts take positions from `new0` on.  A quarter of the
    inserts' share overwrites present keys.  Also returns how many inserts."""
    n_ins = n * ins // 100
    n_er = n * erase // 100
    n_find = n - n_ins - n_er
    n_sw = min(n_ins // 4, live.numel() // 4)
    n_new = n_ins - n_sw
    n_er = min(n_er, live.numel() // 2)
    perm = live[torch.randperm(live.numel(), generator=g, device=DEV)]
    gone, swap, keep = perm[:n_er], perm[n_er:n_er + n_sw], perm[n_er + n_sw:]
    new = _iota(new0, new0 + n_new)
    a = _batch(seed, g, new, gone, swap, keep, n_find, zipf, False)
    b = _batch(seed, g, gone, new, swap, keep, n_find, zipf, True)
    return a, b


def _filled(case, seed, load):
    """Positions, keys and values that fill `load` percent of the slots."""
    n = case["slots"] * load // 100
    keys = _key_of(_iota(0, n), seed)
    return n, _i32(keys), _i32(_val_of(keys, seed))


def _table(case, **kw):
    return hive.HiveTable(case["slots"], bucket_slots=case["bucket_slots"], **kw)


def _find_inputs(case, seed):
    g = _gen(seed)
    live = case["slots"] * case["load"] // 100
    n = case["n"]
    is_hit = torch.rand(n, generator=g, device=DEV) < case["hit"] / 100
    ids = _pick(n, live, case["zipf"], g)
    if case["zipf"]:  # ranks in an order that is not the order of insertion
        ids = torch.randperm(live, generator=g, device=DEV)[ids]
    ids = torch.where(is_hit, ids, ABSENT + _pick(n, 1 << 28, False, g))
    keys = _key_of(ids, seed)
    want = torch.where(is_hit, _val_of(keys, seed), torch.zeros_like(keys))
    return _i32(keys), _i32(want), is_hit.to(torch.uint8)


def _mixed_inputs(case, seed):
    live = case["slots"] * case["load"] // 100
    return _pair(seed, _gen(seed), _iota(0, live), live, case["n"], case["ins"], case["erase"])


def _life_inputs(case, seed):
    """Inputs of ``plain`` and ``set32``: keys and values, queries over present
    and absent keys, and the half to erase, with the results of each phase."""
    g = _gen(seed)
    n, keys, vals = _filled(case, seed, case["load"])
    perm = torch.randperm(n, generator=g, device=DEV)
    gone = perm[: n // 2]
    here = torch.ones(n, dtype=torch.uint8, device=DEV)
    absent = _i32(_key_of(ABSENT + _iota(0, n), seed))
    order = torch.randperm(2 * n, generator=g, device=DEV)
    q = torch.cat([keys, absent])[order]
    zero8, zero32 = torch.zeros_like(here), torch.zeros_like(vals)
    left = here.clone()
    left[gone] = 0
    f1 = torch.cat([here, zero8])[order]
    f2 = torch.cat([left, zero8])[order]
    v = torch.cat([vals, zero32])[order]
    return {"keys": keys, "vals": vals, "q": q, "gone": keys[gone], "v": v, "f1": f1, "f2": f2}


def _build_inputs(case, seed):
    """Keys and values of the two batches of a bulk load, and the results of the
    second one: the last eighth of the keys among as many loaded already."""
    n, keys, vals = _filled(case, seed, case["load"])
    a = n - n // 8
    rest = torch.cat([_iota(a, n), _iota(0, n - a)])
    rest = rest[torch.randperm(rest.numel(), generator=_gen(seed), device=DEV)]
    st = torch.where(rest >= a, ST_INSERTED, ST_REPLACED).to(torch.uint8)
    return [(keys[:a], vals[:a]), (keys[rest], vals[rest] ^ 0x0F0F0F0F)], st


def _stream_inputs(case, seed):
    g = _gen(seed)
    n = case["n"]
    base = case["slots"] * 3 // 10  # below the load at which a table contracts to its first size
    live, nxt = _iota(0, base), base
    up, down = [], []
    for _ in range(case["batches"]):
        n_new, n_er = n * 2 // 5, min(n // 5, live.numel() // 2)
        perm = live[torch.randperm(live.numel(), generator=g, device=DEV)]
        gone, keep = perm[:n_er], perm[n_er:]
        new = _iota(nxt, nxt + n_new)
        nxt += n_new
        none = new[:0]
        up.append(_batch(seed, g, new, gone, none, keep, n - n_new - n_er, True, False))
        down.insert(0, _batch(seed, g, gone, new, none, keep, n - n_new - n_er, True, True))
        live = torch.cat([keep, new])
    return base, nxt, up + down


def _multi_shape(case):
    """Capacities and ops of the tables: log-uniform, the same for every seed."""
    import random
    r = random.Random(case["tables"] * 131 + case["cap_lo"])
    caps, ops = [], []
    for _ in range(case["tables"]):
        c = int(2 ** r.uniform(case["cap_lo"], case["cap_hi"]))
        caps.append(c)
        ops.append(max(1, min(int(2 ** r.uniform(case["ops_lo"], case["ops_hi"])), c // 4)))
    return caps, ops


def _multi_inputs(case, seed):
    g = _gen(seed)
    caps, n_ops = _multi_shape(case)
    base, fills, pairs = 0, [], []
    for c, n in zip(caps, n_ops):
        live = c * 7 // 10
        fills.append((base, base + live))
        pairs.append(_pair(seed, g, _iota(base, base + live), base + live, n, case["ins"],
                           case["erase"]))
        base += live + n
    steps = []
    for side in (0, 1):
        steps.append({k: torch.cat([p[side][k] for p in pairs])
                      for k in ("ops", "keys", "vals", "want", "st")})
    return caps, fills, [(p[0]["keys"].numel(), p[1]["keys"].numel()) for p in pairs], steps


def _inputs_of(b):
    return {k: b[k] for k in ("ops", "keys", "vals")}


# ---- the cases ---------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind}
    if kind == "set32":
        life = _life_inputs(case, seed)
        s["t"] = hive.Hive32Table(case["slots"], layout=hive.KEY_ONLY)
        s.update({k: life[k] for k in ("keys", "q", "gone")})
    elif kind == "plain":
        life = _life_inputs(case, seed)
        s["t"] = _table(case)
        s.update({k: life[k] for k in ("keys", "vals", "q", "gone")})
    elif kind == "build":
        s["t"] = _table(case)
        s["parts"] = _build_inputs(case, seed)[0]
    elif kind == "find":
        s["t"] = _table(case)
        _, keys, vals = _filled(case, seed, case["load"])
        s["t"].insert(keys, vals, status=None)
        s["q"] = _find_inputs(case, seed)[0]
        s["host"] = case["host"]
        if case["host"]:
            s["q"] = s["q"].cpu().pin_memory()
            s["v"] = torch.empty(case["n"], dtype=torch.int32).pin_memory()
            s["f"] = torch.empty(case["n"], dtype=torch.uint8).pin_memory()
    elif kind == "mixed":
        s["t"] = _table(case)
        _, keys, vals = _filled(case, seed, case["load"])
        s["t"].insert(keys, vals, status=None)
        s["batches"] = [_inputs_of(b) for b in _mixed_inputs(case, seed)]
        s["fused"] = case["fused"]
    elif kind == "stream":
        base, top, batches = _stream_inputs(case, seed)
        s["t"] = _table(case, resizable=True, max_slots=max(4 * top, 4 * case["slots"]))
        keys = _key_of(_iota(0, base), seed)
        s["t"].insert(_i32(keys), _i32(_val_of(keys, seed)), status=None)
        s["batches"] = [_inputs_of(b) for b in batches]
        s["top"] = len(batches) // 2
    else:
        caps, fills, counts, steps = _multi_inputs(case, seed)
        res = case["resizable"]
        s["tables"], s["steps"], s["out"] = [], [], []
        for c, (lo, hi) in zip(caps, fills):
            kw = {"resizable": True, "max_slots": 4 * c} if res else {}
            t = hive.HiveTable(c, bucket_slots=case["bucket_slots"], **kw)
            if hi > lo:
                keys = _key_of(_iota(lo, hi), seed)
                t.insert(_i32(keys), _i32(_val_of(keys, seed)), status=None)
            s["tables"].append(t)
        most = max(int(x["keys"].numel()) for x in steps)
        s["group"] = hive.HiveMulti(s["tables"], max_segments=len(caps), max_ops=most,
                                    use_graph=True, asynchronous=case["asynchronous"])
        for side, x in enumerate(steps):
            vo = torch.empty_like(x["keys"])
            st = torch.empty_like(x["ops"])
            segs, at = [], 0
            for ti, c in enumerate(counts):
                sl = slice(at, at + c[side])
                at += c[side]
                segs.append({"table": ti, "ops": x["ops"][sl], "keys": x["keys"][sl],
                             "vals": x["vals"][sl], "vals_out": vo[sl], "status": st[sl],
                             "n_insert": int((x["ops"][sl] == INSERT).sum())})
            s["steps"].append(segs)
            s["out"].append([vo, st])
    return s


def run(state):
    kind = state["kind"]
    if kind == "multi":
        for segs in state["steps"]:
            state["group"].execute(segs)
        return state["out"]
    t = state["t"]
    if kind == "find":
        if state["host"]:
            return list(t.find_host(state["q"], state["v"], state["f"]))
        return list(t.find(state["q"]))
    if kind == "mixed":
        return [list(t.execute(b["ops"], b["keys"], b["vals"], fused=state["fused"]))
                for b in state["batches"]]
    if kind == "build":
        t.clear()
        return [t.insert(keys, vals) for keys, vals in state["parts"]]
    if kind == "stream":
        out, caps = [], []
        for i, b in enumerate(state["batches"]):
            if i == state["top"]:
                caps.append(t.capacity())
            out.append(list(t.execute(b["ops"], b["keys"], b["vals"])))
        return [out, caps, t.size()]
    t.clear()
    st = t.insert(state["keys"], state["vals"]) if kind == "plain" else t.insert(state["keys"])
    first = list(t.find(state["q"]))
    gone = t.erase(state["gone"])
    return [st, first, gone, list(t.find(state["q"]))]


def _counts(case, n):
    n_ins = n * case["ins"] // 100
    n_er = n * case["erase"] // 100
    return n_ins, n_er, n - n_ins - n_er


SECTOR = 32  # the least that memory moves for one table entry


def work(case):
    """Bytes of one pass: the op arrays, and one sector of table memory read for
    each key that is found and one read and one written for each update."""
    kind = case["kind"]
    if kind == "find":
        n = case["n"]
        return {"bytes": 9 * n + SECTOR * (n * case["hit"] // 100), "flops": 0}

    def mixed(n, n_ins, n_er, n_find):
        return 10 * n + 4 * n_ins + 2 * SECTOR * (n_ins + n_er) + SECTOR * (n_find * 7 // 8)

    if kind == "mixed":
        return {"bytes": 2 * mixed(case["n"], *_counts(case, case["n"])), "flops": 0}
    if kind == "stream":
        n = case["n"]
        return {"bytes": 2 * case["batches"] * mixed(n, n * 2 // 5, n // 5, n - n * 2 // 5 - n // 5),
                "flops": 0}
    if kind == "multi":
        return {"bytes": 2 * sum(mixed(n, *_counts(case, n)) for n in _multi_shape(case)[1]),
                "flops": 0}
    n = case["slots"] * case["load"] // 100
    entry = 4 if kind == "set32" else 8
    load = entry * case["slots"] + (5 if kind == "set32" else 9) * n
    if kind == "build":
        return {"bytes": load + (n // 8) * (9 + 2 * SECTOR), "flops": 0}
    finds = 2 * 9 * 2 * n + SECTOR * (n + n // 2)
    return {"bytes": load + finds + (n // 2) * (5 + 2 * SECTOR), "flops": 0}


def exact(case, seed):
    kind = case["kind"]
    if kind == "find":
        _, want, found = _find_inputs(case, seed)
        return [want, found]
    if kind == "mixed":
        return [[b["want"], b["st"]] for b in _mixed_inputs(case, seed)]
    if kind == "build":
        parts, st = _build_inputs(case, seed)
        return [torch.zeros_like(parts[0][0], dtype=torch.uint8), st]
    if kind == "stream":
        base, _, batches = _stream_inputs(case, seed)
        return [[[b["want"], b["st"]] for b in batches], [None], base]
    if kind == "multi":
        return [[x["want"], x["st"]] for x in _multi_inputs(case, seed)[3]]
    life = _life_inputs(case, seed)
    st = torch.zeros_like(life["keys"], dtype=torch.uint8)
    gone = torch.full_like(life["gone"], ST_ERASED, dtype=torch.uint8)
    if kind == "set32":
        v1 = v2 = torch.zeros_like(life["v"])
    else:
        v1 = life["v"]
        v2 = torch.where(life["f2"] == 1, life["v"], torch.zeros_like(life["v"]))
    return [st, [v1, life["f1"]], gone, [v2, life["f2"]]]
