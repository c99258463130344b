"""Work that programs have these filters do, as measurable cases.

A case is a dict of plain values. `prepare` makes its keys and filters on the
GPU, `run` is one pass over them through the public binding, and `work` says
how many bytes such a pass cannot do without. Two kinds of pass:

  "fill"    a filter's whole life: clear, insert up to the load in batches,
            query stored and fresh keys, remove part of the keys, query again;
  "update"  a filter already at its load (filled in prepare) takes one batch:
            insert, query, remove, as a service does with its live filters.

A pass returns what the calls answered (statuses, found flags, counts,
values) and the filter's table itself, through the device view.
"""
import math

import torch

import paper_2212_09005_gb300 as gf

# the fill and query shapes of each kind of filter, without their sizes
TCF = {"filter": "tcf", "tag_bits": 16, "mode": "bulk", "value_bits": 0, "block_slots": 0, "load": 0.9, "remove": 0.5}
GQF = {"filter": "gqf", "tag_bits": 8, "keys": "uniform", "remove": 0.125}


def listed():
    return [
        # a live two-choice filter of 2^20 slots that takes 1000 keys at a
        # time and asks for statuses: the smallest batches of the serving
        # workload; launches and latency count
        dict(TCF, name="tcf update 1000", work="update", log2_slots=20, batch=1000, queries=2001, status=True),
        # the same service at an ordinary batch: 2^24 slots, 100,003 keys
        dict(TCF, name="tcf update 100003", work="update", log2_slots=24, batch=100_003, queries=200_007, status=True),
        # the benchmark's TCF: 2^26 slots filled in 2^22-key batches
        dict(TCF, name="tcf fill 2^26", work="fill", log2_slots=26, batch=1 << 22, queries=1 << 25, status=False),
        # the target size: 2^28 slots in 2^24-key batches, past the L2
        dict(TCF, name="tcf fill 2^28", work="fill", log2_slots=28, batch=1 << 24, queries=1 << 25, status=False),
        # a small value stored with every key (4 bits in 16-bit slots)
        dict(TCF, name="tcf values 2^24", work="fill", log2_slots=24, batch=1 << 20, queries=1 << 22, status=True,
             value_bits=4),
        # Alg. 1 of the paper: one compare-and-swap per key, no sorted blocks
        dict(TCF, name="tcf point 2^24", work="fill", log2_slots=24, batch=1 << 20, queries=1 << 23, status=False,
             mode="point"),
        # the paper's bulk TCF block of 128 slots (Sec. 4.2)
        dict(TCF, name="tcf blocks of 128", work="fill", log2_slots=22, batch=(1 << 19) - 3, queries=1 << 21,
             status=False, block_slots=128),
        # a live counting filter of 2^20 slots that takes 1000 keys at a time
        dict(GQF, name="gqf update 1000", work="update", log2_slots=20, load=0.85, batch=1000, queries=2001,
             status=True, remove=1.0),
        # the paper's smallest bulk build: 2^20 slots in one batch
        dict(GQF, name="gqf fill 2^20", work="fill", log2_slots=20, load=0.9, batch=943_718, queries=1 << 21,
             status=False),
        # the counting benchmark: 2.4e8 Zipf(1.0) keys over 2^32
        dict(GQF, name="gqf zipf 2^28", work="fill", log2_slots=28, load=240_000_000 / (1 << 28), batch=240_000_000,
             queries=1 << 24, status=False, keys="zipf", remove=(1 << 24) / 240_000_000),
        # keys that bring their counts (values through the counters), 16-bit
        # remainders
        dict(GQF, name="gqf counts 2^24", work="fill", log2_slots=24, tag_bits=16, load=0.19, batch=3_187_671,
             queries=1 << 21, status=True, keys="counts"),
        # many small filters driven by one call each operation: half TCF,
        # half GQF, 2^10 .. 2^18 slots, as one filter per user or shard
        {"name": "groups of 512", "filter": "groups", "members": 512, "emin": 10, "emax": 18, "rounds": 4},
    ]


def draw(rng):
    """One more case of the listed ones' ranges; sizes log-uniform, mostly odd."""
    def size(lo, hi):
        return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))

    kind = rng.choice(["tcf update", "tcf fill", "tcf option", "gqf update", "gqf fill", "groups"])
    if kind == "groups":
        lo = rng.randint(10, 12)
        return {"filter": "groups", "members": 2 * size(8, 512), "emin": lo, "emax": rng.randint(lo + 1, 18),
                "rounds": rng.randint(1, 6)}
    if kind == "tcf update":
        lg = rng.randint(18, 26)
        return dict(TCF, work="update", log2_slots=lg, batch=size(256, (1 << lg) // 32), queries=size(256, 1 << 22),
                    status=rng.random() < 0.7, tag_bits=rng.choice([16, 16, 16, 8]))
    if kind == "tcf fill":
        lg = rng.randint(18, 28)
        return dict(TCF, work="fill", log2_slots=lg, batch=size((1 << lg) // 32, (1 << lg) // 12),
                    queries=size(1 << 16, 1 << 24), status=rng.random() < 0.3, load=rng.uniform(0.8, 0.9),
                    tag_bits=rng.choice([16, 16, 16, 8]))
    if kind == "tcf option":
        lg = rng.randint(18, 24)
        c = dict(TCF, work="fill", log2_slots=lg, batch=size((1 << lg) // 20, (1 << lg) // 10),
                 queries=size(1 << 14, 1 << 22), status=rng.random() < 0.5)
        c.update(rng.choice([{"value_bits": 4}, {"value_bits": 2, "tag_bits": 8}, {"mode": "point", "load": 0.85},
                             {"block_slots": 128}, {"block_slots": 64}, {"block_slots": 32},
                             {"block_slots": 21, "tag_bits": 12}]))
        return c
    if kind == "gqf update":
        lg = rng.randint(16, 26)
        return dict(GQF, work="update", log2_slots=lg, load=rng.uniform(0.5, 0.9), batch=size(256, (1 << lg) // 16),
                    queries=size(256, 1 << 22), status=rng.random() < 0.7, remove=1.0, tag_bits=rng.choice([8, 8, 16]))
    lg = rng.randint(16, 27)
    keys = rng.choice(["uniform", "uniform", "zipf", "counts"])
    load = rng.uniform(0.1, 0.19) if keys == "counts" else rng.uniform(0.6, 0.9)
    return dict(GQF, work="fill", log2_slots=lg, load=load, batch=size((1 << lg) // 8, 1 << lg),
                queries=size(1 << 12, 1 << 24), status=rng.random() < 0.3, keys=keys,
                remove=rng.choice([0.02, 0.125, 0.5]), tag_bits=rng.choice([8, 8, 16]))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def uniform_keys(g, n):
    return torch.randint(-(1 << 63), (1 << 63) - 1, (n,), dtype=torch.int64, device="cuda", generator=g)


def zipf_keys(g, n, universe=1 << 32):
    """n keys rank - 1 with P(rank) proportional to 1 / rank: rejection-inversion
    (Hoermann and Derflinger 1996) with H(x) = ln x."""
    h1, hn = math.log(1.5) - 1.0, math.log(universe + 0.5)
    squeeze = 2.0 - math.exp(math.log(2.5) - 0.5)
    out, have = torch.empty(n, dtype=torch.int64, device="cuda"), 0
    while have < n:
        u = hn + torch.rand(min(n - have, 1 << 26), dtype=torch.float64, device="cuda", generator=g) * (h1 - hn)
        x = u.exp()
        k = (x + 0.5).floor().clamp(1.0, float(universe))
        k = k[(k - x <= squeeze) | (u >= (k + 0.5).log() - 1.0 / k)]
        out[have:have + k.numel()] = k.to(torch.int64) - 1
        have += k.numel()
    return out


def half_and_half(g, keys, n):
    """n query keys: stored ones drawn with replacement, then fresh ones."""
    pos = keys[torch.randint(0, keys.numel(), (n - n // 2,), device="cuda", generator=g)]
    return torch.cat([pos, uniform_keys(g, n // 2)])


def bytes_out(n):
    return torch.zeros(n, dtype=torch.uint8, device="cuda")


def longs_out(n):
    return torch.zeros(n, dtype=torch.int64, device="cuda")


class DeviceArray:
    """n bytes of a filter's memory; a tensor made of it keeps the filter alive."""

    def __init__(self, owner, pointer, n):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": "|u1", "data": (pointer, False), "version": 3}


def n_keys(case):
    return int(case["load"] * (1 << case["log2_slots"]))


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    if case["filter"] == "groups":
        return prepare_groups(case, seed, g)
    n, batch, tcf = n_keys(case), case["batch"], case["filter"] == "tcf"
    update = case["work"] == "update"
    fill = max(batch, n // 12) if update else batch  # the batches that bring an updated filter to its load
    if tcf:
        f = gf.TCF(case["log2_slots"], case["tag_bits"], gf.MODE_POINT if case["mode"] == "point" else gf.MODE_BULK,
                   seed=seed, max_batch=fill, value_bits=case["value_bits"], block_slots=case["block_slots"])
    else:
        f = gf.GQF(case["log2_slots"], case["tag_bits"], seed=seed, max_batch=fill)
    zipf = not tcf and case["keys"] == "zipf"
    keys = zipf_keys(g, n) if zipf else uniform_keys(g, n)
    s = {"case": case, "filter": f, "tables": {}}
    if update:
        for k in keys.split(fill):
            f.insert(k)
        keys = uniform_keys(g, batch)
        s["removed"] = keys
    else:
        step = max(1, round(1.0 / case["remove"]))
        s["removed"] = keys[step - 1::step].contiguous()
    s["batches"] = list(keys.split(batch))
    s["removed_batches"] = list(s["removed"].split(batch))
    s["status"] = [bytes_out(k.numel()) if case["status"] else None for k in s["batches"]]
    s["removed_status"] = [bytes_out(k.numel()) if case["status"] else None for k in s["removed_batches"]]
    s["queries"] = half_and_half(g, keys, case["queries"])
    out = longs_out if not tcf else bytes_out
    s["answers"], s["after"] = out(case["queries"]), out(case["queries"])
    if tcf and case["value_bits"]:
        s["values"] = [torch.randint(0, 1 << case["value_bits"], (k.numel(),), dtype=torch.uint8, device="cuda",
                                     generator=g) for k in s["batches"]]
    if not tcf and case["keys"] == "counts":
        s["counts"] = [torch.randint(1, 9, (k.numel(),), dtype=torch.int32, device="cuda", generator=g)
                       for k in s["batches"]]
    return s


def prepare_groups(case, seed, g):
    """Half TCF, half GQF members of 2^emin .. 2^emax slots, 85 to 95 % load
    (the sizes belong to the case, the keys to the seed); the TCF half takes
    its keys in rounds of near-equal chunks per member."""
    m = case["members"] // 2
    sizes = torch.Generator(device="cuda")
    sizes.manual_seed(m)
    halves = []
    for kind in (gf.FILTER_TCF, gf.FILTER_GQF):
        e = torch.randint(case["emin"], case["emax"] + 1, (m,), device="cuda", generator=sizes)
        load = 0.85 + 0.1 * torch.rand(m, device="cuda", generator=sizes, dtype=torch.float64)
        length = (load * 2.0 ** e).long()
        rounds = case["rounds"] if kind == gf.FILTER_TCF else 1
        cuts = [length * j // rounds for j in range(rounds + 1)]
        offsets = [torch.cat([length.new_zeros(1), (b - a).cumsum(0)]) for a, b in zip(cuts, cuts[1:])]
        keys = [uniform_keys(g, int(o[-1])) for o in offsets]
        group = gf.FilterGroup(kind, e.tolist(), 16 if kind == gf.FILTER_TCF else 8,
                               torch.randint(0, 1 << 62, (m,), device="cuda", generator=g).tolist(),
                               max(k.numel() for k in keys))
        # queries: the last round's keys of every member, mixed with fresh ones
        q = torch.where(torch.rand(keys[-1].numel(), device="cuda", generator=g) < 0.5, keys[-1],
                        uniform_keys(g, keys[-1].numel()))
        halves.append({"kind": kind, "group": group, "offsets": offsets, "keys": keys, "queries": q,
                       "answers": (bytes_out if kind == gf.FILTER_TCF else longs_out)(q.numel()),
                       "status": bytes_out(keys[-1].numel())})
    return {"case": case, "halves": halves}


# ---------------------------------------------------------------------------
# A pass
# ---------------------------------------------------------------------------
def table(s):
    """The filter's table (blocks and buckets, or metadata and remainders)."""
    v, case = s["filter"].device_view(), s["case"]
    if v.table not in s["tables"]:
        if case["filter"] == "tcf":
            sizes = v.n_blocks * 32, v.n_aux * 64
        else:
            sizes = v.n_blocks * 32, v.n_aux * (case["tag_bits"] // 8)
        s["tables"][v.table] = [torch.as_tensor(DeviceArray(s["filter"], p, n), device="cuda")
                                for p, n in zip((v.table, v.aux), sizes)]
    return s["tables"][v.table]


def ask(s, out):
    f, case = s["filter"], s["case"]
    if case["filter"] == "gqf":
        f.count(s["queries"], out)
    elif case["value_bits"]:
        f.query_values(s["queries"], out)
    else:
        f.query(s["queries"], out)


def run(s):
    case = s["case"]
    if case["filter"] == "groups":
        return run_groups(s)
    f, values, counts = s["filter"], s.get("values"), s.get("counts")
    if case["work"] == "fill":
        f.clear()
    for i, (keys, status) in enumerate(zip(s["batches"], s["status"])):
        if counts:
            f.insert_counts(keys, counts[i], status)
        elif values:
            f.insert(keys, status, values=values[i])
        else:
            f.insert(keys, status)
    ask(s, s["answers"])
    for keys, status in zip(s["removed_batches"], s["removed_status"]):
        f.remove(keys, status)
    ask(s, s["after"])
    out = {"answers": s["answers"], "after": s["after"]}
    if case["status"]:
        out["status"], out["removed_status"] = s["status"][-1], s["removed_status"][-1]
    # which slot of a block a point-mode key takes depends on the threads'
    # order, and other block sizes have no device view: the answers tell
    if case["filter"] == "gqf" or (case["mode"] == "bulk" and not case["block_slots"]):
        out["table"] = table(s)
    return out


def run_groups(s):
    out = {}
    for h in s["halves"]:
        group, name = h["group"], "tcf" if h["kind"] == gf.FILTER_TCF else "gqf"
        group.clear()
        for offsets, keys in zip(h["offsets"], h["keys"]):
            group.insert(offsets, keys)
        if h["kind"] == gf.FILTER_TCF:
            group.query(offsets, h["queries"], h["answers"])
        else:
            group.count(offsets, h["queries"], h["answers"])
        group.remove(offsets, keys, h["status"])
        out[name] = {"answers": h["answers"], "status": h["status"]}
    return out


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def calls_bytes(table_bytes, record, calls):
    """calls: (keys, bytes in and out per key, records touched per key, written?).
    A call reads each record it touches once, at most the table, and writes it
    once when it changes it."""
    total = 0
    for n, io, touched, written in calls:
        total += n * io + min(table_bytes, n * touched * record) * (2 if written else 1)
    return total


def work(case):
    if case["filter"] == "groups":
        # expected sizes: e uniform over the range, mean load 0.9
        span = case["emax"] - case["emin"] + 1
        slots = case["members"] / 2 * sum(2.0 ** e for e in range(case["emin"], case["emax"] + 1)) / span
        n, r = 0.9 * slots, case["rounds"]
        tcf = calls_bytes(2 * slots, 32, [(n / r, 8, 1, True)] * r + [(n / r, 9, 2, False), (n / r, 9, 1, True)])
        gqf = calls_bytes(1.5 * slots, 64, [(n, 8, 1, True), (n, 16, 1, False), (n, 9, 1, True)])
        return {"bytes": tcf + gqf + 3.5 * slots, "flops": 0}
    n, st = n_keys(case), 1 if case["status"] else 0
    slots, size = 1 << case["log2_slots"], case["batch"]
    if case["work"] == "update":
        n, cleared, removed = case["batch"], 0, case["batch"]
    else:
        cleared, removed = 1, n // max(1, round(1.0 / case["remove"]))
    inserts, removes = (([size] * (k // size) + ([k % size] if k % size else [])) for k in (n, removed))
    if case["filter"] == "tcf":
        b = case["block_slots"] or 256 // case["tag_bits"]
        record = (b * case["tag_bits"] + 255) // 256 * 32
        size, extra = slots // b * record, 1 if case["value_bits"] else 0
        calls = [(k, 8 + st + extra, 1, True) for k in inserts] + [(k, 8 + st, 1, True) for k in removes]
        calls += [(case["queries"], 9, 2, False)] * 2
    else:
        record = 32 + 32 * case["tag_bits"] // 8  # a metadata record and a 32-slot stretch of remainders
        size, extra = slots * (case["tag_bits"] / 8 + 0.5), 4 if case["keys"] == "counts" else 0
        calls = [(k, 8 + st + extra, 1, True) for k in inserts] + [(k, 8 + st, 1, True) for k in removes]
        calls += [(case["queries"], 16, 1, False)] * 2
    return {"bytes": calls_bytes(size, record, calls) + cleared * size, "flops": 0}
