"""Performance cases of the hash containers: the calls a program makes, through
the package's public entry points, from a few thousand keys on a small table to
the 2^28-slot map.

Keys are a bijective mix of consecutive counters, so the keys of a stream are
distinct and the streams of one case never overlap; absent keys come from a
counter range that is never inserted.  Batches that modify a table undo
themselves (or clear it first), so a pass can be repeated.  Every output is a
whole number (statuses, flags, keys, values) that does not depend on the order
in which the GPU's threads run, so outputs compare exactly and there is nothing
to state in floating point.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1908_05936_gb300 import _lib as L
from paper_1908_05936_gb300.batch import Batch, Item
from paper_1908_05936_gb300.table import KEY_BYTES, KEY_NUMPY, KEY_TORCH, KIND_NAMES, VAL_BYTES, VAL_NUMPY, Table

#: Slots of the multi-table case's tables are log-uniform between these powers of two.
TABLE_LO, TABLE_HI = 10.0, 20.0
#: Layers of voxel blocks a reconstructed surface fills (noise spreads it over a few).
LAYERS = 5


def listed():
    return [
        # One small query: a few thousand block lookups against a small scene's map with the paper's short3 keys.
        # The call's latency is what its user waits for.
        dict(name="lookup_4k", do="find", kind="map_i64_i32", slots=1 << 16, bucket=64, hash="short3", load=0.6,
             n=4097, hit=0.5),
        # The set<u32> workload of the benchmark: 2^21 slots, 10^6 inserts, 10^6 queries, 5 * 10^5 erases, L2-resident.
        dict(name="set_u32_step", do="step", kind="set_u32", slots=1 << 21, bucket=32, load=1000000 / (1 << 21),
             batch=1 << 26, n=1000000, erase=500000),
        # One RGB-D frame of the reconstruction workload: 400,000 candidate blocks with repeats, 12.5 M slots,
        # spatial hash: look up, insert what is missing, look up the block indices, drop the frame's new blocks.
        dict(name="frame_400k", do="frame", slots=12500000, bucket=128, hash="teschner", n=400000),
        # Bulk lookups at the headline size: 2^26 queries, half of them present, on 2^28 slots at load factor 0.8.
        dict(name="map_find_64m", do="find", kind="map_u64_u64", slots=1 << 28, bucket=64, hash="mix", load=0.8,
             n=1 << 26, hit=0.5),
        # The headline step: clear, fill to 0.8 in batches of 2^26, 2^26 present and 2^26 absent lookups, 2^26 erases.
        dict(name="map_step_256m", do="step", kind="map_u64_u64", slots=1 << 28, bucket=64, load=0.8, batch=1 << 26,
             n=1 << 26, erase=1 << 26),
        # Steady traffic on a resident map in batches of about a million (an odd size): new keys come, all are
        # looked up, the same keys leave.
        dict(name="map_churn_1m", do="churn", kind="map_u64_u64", slots=50000000, bucket=64, load=0.7, n=1000003),
        # Deduplication against a large set: 30 M membership queries, most of them new, 32-byte buckets (the default).
        dict(name="set_contains_30m", do="find", kind="set_u64", slots=100000000, bucket=32, hash="mix", load=0.7,
             n=30000001, hit=0.25),
        # Many tables at once: one graph launch of inserts, lookups and erases on 192 sets of 2^10 .. 2^20 slots.
        dict(name="batch_192_tables", do="batch", kind="set_u64", tables=192, bucket=32),
        # Reproducible ingestion: batches in which every key repeats and the lowest index has to win.
        dict(name="ordered_4m", do="ordered", kind="map_u64_u64", slots=1 << 25, bucket=64, load=0.5, n=1 << 22,
             repeat=2),
        # A free-running mixed batch (50 / 30 / 20 inserts, lookups, erases) on a table rebuilt before it.
        dict(name="mixed_4m", do="mixed", kind="map_u64_u64", slots=1 << 24, bucket=64, load=0.4, n=1 << 22),
        # Maintenance of a resident map: rehash, flag the entries of a key class, dump every entry.
        dict(name="maintain_64m", do="maintain", kind="map_u64_u64", slots=1 << 26, bucket=64, load=0.6),
        # The same operations on page-locked host arrays, as a program without device arrays calls them.
        dict(name="host_4m", do="host", kind="map_u64_u64", slots=1 << 26, bucket=64, load=0.5, n=1 << 22,
             pinned=True),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    do = rng.choice(["find", "find", "step", "frame", "churn", "churn", "batch", "ordered", "mixed", "maintain",
                     "host"])
    kind = rng.choice(["set_u32", "set_u64", "map_i64_i32", "map_u64_u64", "map_u64_u64"])
    if do == "batch":
        return dict(do=do, kind=rng.choice(["set_u64", "map_u64_u64"]), tables=log(8, 256),
                    bucket=rng.choice([32, 64, 128]))
    if do == "frame":
        return dict(do=do, slots=log(2000000, 30000000), bucket=rng.choice([32, 64, 128]),
                    hash=rng.choice(["teschner", "mix"]), n=log(20000, 1000000))
    if do == "maintain" and kind in ("set_u32", "set_u64"):
        kind = "map_i64_i32"
    top = {"find": 1 << 28, "step": 1 << 27, "mixed": 1 << 25, "ordered": 1 << 26}.get(do, 1 << 26)
    slots = log(1 << 12, top if kind != "set_u32" else min(top, 1 << 26))
    case = dict(do=do, kind=kind, slots=slots, bucket=rng.choice([32, 64, 128]), load=round(rng.uniform(0.3, 0.8), 3))
    if do == "maintain":
        return case
    room = int(slots * min(0.9 - case["load"], 0.5))
    if do == "find":
        case.update(hash="mix", n=log(1000, 1 << 26), hit=round(rng.uniform(0.0, 1.0), 2))
    elif do == "step":
        stored = int(slots * case["load"])
        case.update(batch=log(max(1000, stored // 64), 1 << 26), n=log(1000, min(1 << 26, 2 * slots)),
                    erase=rng.randint(1, stored))
    else:
        case.update(n=rng.randint(1, room) if room < 2000 else log(1000, min(room, 1 << 23)))
        if do == "ordered":
            case.update(repeat=rng.choice([1, 2, 3, 8]))
        if do == "host":
            case.update(pinned=rng.random() < 0.7)
    return case


# ------------------------------------------------------------------ keys ---

def _mix(x, salt):
    """A bijection of 64-bit words (xor-shifts and odd multipliers), in place."""
    for mul in (-0x61C8864680B583EB, -0x40A7B892E31B1A47, -0x6B2FB644ECCEEE15):
        x ^= salt
        x ^= (x >> 32) & 0xFFFFFFFF
        x *= mul
    x ^= (x >> 32) & 0xFFFFFFFF
    return x


def _mix32(x, salt):
    """The same for 32-bit words held in int64; returns int32 bit patterns."""
    for mul in (0x85EBCA6B, 0xC2B2AE35, 0x9E3779B1):
        x = x ^ (salt & 0xFFFF)
        x = x ^ (x >> 16)
        x = (x * mul) & 0xFFFFFFFF
    x = x ^ (x >> 16)
    return x.to(torch.int32)


def _keys_at(kind, idx, seed):
    """Keys number idx (int64 tensor, taken over) of a case's stream."""
    if kind == L.SET_U32:
        return _mix32(idx, seed * 2654435761 + 12345)
    return _mix(idx, (seed * 2654435761 + 12345) & 0xFFFFFFFFFFFF)


def _keys(kind, start, n, seed):
    return _keys_at(kind, torch.arange(start, start + n, dtype=torch.int64, device="cuda"), seed)


def _spread(n, of):
    """n distinct positions below `of`, scattered (n <= of)."""
    i = torch.arange(n, dtype=torch.int64, device="cuda")
    return (i * 2654435761 + 40503) % of if of % 2654435761 else i


def _vals(kind, keys):
    if kind == L.MAP_U64_U64:
        return keys * 0x2545F4914F6CDD1D + 1
    if kind == L.MAP_I64_I32:
        return (keys * 0x2545F4914F6CDD1D >> 33).to(torch.int32)
    return None


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _short3(idx):
    """Distinct block coordinates of a 64 x 64 x 16 scene patch and its surroundings, as (n, 3) int16."""
    return torch.stack([idx % 64 - 32, (idx // 64) % 64 - 32, idx // 4096 - 8], 1).to(torch.int16).contiguous()


def _pack21(x, y, z):
    m = (1 << 21) - 1
    return (x & m) | ((y & m) << 21) | ((z & m) << 42)


def _table(case, kind, hash_mode=L.HASH_MIX64):
    return Table(kind, case["slots"], bucket_bytes=case["bucket"], hash_mode=hash_mode)


def _fill(t, kind, n, seed, step=1 << 26):
    """Stores keys 0 .. n of the stream."""
    for a in range(0, n, step):
        k = _keys(kind, a, min(step, n - a), seed)
        t.insert(k, _vals(kind, k), status=False)


# --------------------------------------------------------------- prepare ---

def prepare(case, seed):
    s = {"case": case, "kind": KIND_NAMES[case.get("kind", "map_i64_i32")]}
    globals()["_prepare_" + case["do"]](s, case, s["kind"], seed)
    return s


def _prepare_find(s, case, kind, seed):
    stored, n = int(case["slots"] * case["load"]), case["n"]
    g = _gen(seed)
    pick = torch.randint(0, stored, (n,), generator=g, device="cuda")
    hit = torch.rand(n, generator=g, device="cuda") < case["hit"]
    idx = torch.where(hit, pick, pick + stored)
    del pick, hit
    if case["hash"] == "short3":
        from paper_1908_05936_gb300.table import pack_short3
        place = torch.randperm(1 << 17, generator=g, device="cuda")
        s["t"] = _table(case, kind, L.HASH_TESCHNER_SHORT3)
        keys = pack_short3(_short3(place[:stored]))
        s["t"].insert(keys, _vals(kind, keys), status=False)
        s["q"] = pack_short3(_short3(place[idx]))
    else:
        s["t"] = _table(case, kind)
        _fill(s["t"], kind, stored, seed)
        s["q"] = _keys_at(kind, idx, seed)


def _prepare_step(s, case, kind, seed):
    stored, n = int(case["slots"] * case["load"]), case["n"]
    s["t"] = _table(case, kind)
    s["keys"] = _keys(kind, 0, stored, seed)
    s["vals"] = _vals(kind, s["keys"])
    g = _gen(seed)
    idx = torch.randint(0, stored, (n,), generator=g, device="cuda")
    if kind in VAL_BYTES:                                               # maps: all present, then all absent
        s["queries"] = [_keys_at(kind, idx, seed), _keys(kind, stored, n, seed)]
    else:                                                               # sets: half of each, shuffled together
        idx += (torch.rand(n, generator=g, device="cuda") < 0.5) * stored
        s["queries"] = [_keys_at(kind, idx, seed)]
    s["leave"] = s["keys"][_spread(case["erase"], stored)]


def _prepare_frame(s, case, kind, seed):
    # stored: LAYERS block layers of a floor wide * length (load factor about 0.75), as a camera leaves it behind
    wide = 531
    length = int(case["slots"] * 0.75) // (wide * LAYERS)
    i = torch.arange(wide * length * LAYERS, dtype=torch.int64, device="cuda")
    keys = _pack21(i % wide - wide // 2, i // wide % length, i // (wide * length))
    s["t"] = _table(case, kind, L.HASH_TESCHNER if case["hash"] == "teschner" else L.HASH_MIX64)
    s["t"].insert(keys, i.to(torch.int32), status=False)
    # the frame: samples over a 12 m band of the floor, noise across the layers; what falls outside them is new
    g, n = _gen(seed), case["n"]
    band = min(188, length)
    x = torch.randint(0, wide, (n,), generator=g, device="cuda") - wide // 2
    y = torch.randint(0, band, (n,), generator=g, device="cuda") + seed % max(1, length - band)
    z = torch.round(torch.randn(n, generator=g, device="cuda") * 1.6 + (LAYERS - 1) / 2).to(torch.int64)
    s["cand"] = _pack21(x, y, z)
    s["index"] = (s["cand"] * 0x2545F4914F6CDD1D >> 33).to(torch.int32)
    # what leaves again: the frame's new blocks, among blocks that are not there (n / 6 in all)
    new = torch.unique(s["cand"][(z < 0) | (z >= LAYERS)])[:n // 6]
    m = n // 6 - new.numel()
    new = torch.cat([new, _pack21(torch.arange(m, device="cuda") % wide, torch.arange(m, device="cuda") // wide,
                                  torch.full((m,), 1000, device="cuda"))])
    s["leave"] = new[torch.randperm(n // 6, generator=g, device="cuda")]


def _prepare_churn(s, case, kind, seed):
    stored = int(case["slots"] * case["load"])
    s["t"] = _table(case, kind)
    _fill(s["t"], kind, stored, seed)
    s["keys"] = _keys(kind, stored, case["n"], seed)
    s["vals"] = _vals(kind, s["keys"])
    s["queries"] = _some_absent(kind, stored, case["n"], seed)


def _some_absent(kind, start, n, seed):
    """Queries for the n keys from number `start` on, in another order, every fourth or so for an absent key."""
    g = _gen(seed)
    idx = start + torch.randperm(n, generator=g, device="cuda")
    idx += (torch.rand(n, generator=g, device="cuda") < 0.25) * n
    return _keys_at(kind, idx, seed)


def _prepare_batch(s, case, kind, seed):
    rng = np.random.RandomState(case["tables"])                         # the sizes belong to the case
    slots = [int(-(-round(2.0 ** u) // 16) * 16) for u in rng.uniform(TABLE_LO, TABLE_HI, case["tables"])]
    parts = [(round(0.3 * c), round(0.15 * c)) for c in slots]          # inserts (all erased again), lookups
    pad = [[-(-n // 16) * 16 for n in p] for p in parts]
    ins = _keys(kind, 0, sum(p[0] for p in pad), seed)
    vals = _vals(kind, ins)
    n_find = sum(p[1] for p in pad)
    s["status"] = torch.zeros(ins.numel(), dtype=torch.uint8, device="cuda")
    s["gone"] = torch.zeros(ins.numel(), dtype=torch.uint8, device="cuda")
    s["found"] = torch.zeros(n_find, dtype=torch.uint8, device="cuda")
    s["got"] = torch.zeros(n_find, dtype=torch.int64, device="cuda") if kind == L.MAP_U64_U64 else None
    fresh, g = _keys(kind, ins.numel(), n_find, seed), _gen(seed)
    items, a, f = [], 0, 0
    s["tables"] = []
    for c, (n, q), (pn, pq) in zip(slots, parts, pad):
        t = Table(kind, c, bucket_bytes=case["bucket"])
        s["tables"].append(t)
        k, look = ins[a:a + n], fresh[f:f + q]
        look.copy_(torch.where(torch.rand(q, generator=g, device="cuda") < 0.5, k[:q], look))   # half: keys of this batch
        items.append(Item(t, L.OP_INSERT, k, vals[a:a + n] if vals is not None else None, s["status"][a:a + n]))
        items.append(Item(t, L.OP_FIND, look, None, s["found"][f:f + q],
                          s["got"][f:f + q] if s["got"] is not None else None))
        items.append(Item(t, L.OP_ERASE, k, None, s["gone"][a:a + n]))
        a, f = a + pn, f + pq
    s["batch"] = Batch(items)


def _prepare_ordered(s, case, kind, seed):
    stored, n = int(case["slots"] * case["load"]), case["n"]
    s["t"] = _table(case, kind)
    _fill(s["t"], kind, stored, seed)
    pick = torch.randint(0, max(1, n // case["repeat"]), (n,), generator=_gen(seed), device="cuda") + stored
    s["keys"] = _keys_at(kind, pick, seed)
    i = torch.arange(n, dtype=torch.int64, device="cuda")               # values tell the occurrences apart
    s["vals"] = None if kind not in VAL_BYTES else i.to(KEY_TORCH[VAL_BYTES[kind]])


def _prepare_mixed(s, case, kind, seed):
    stored, n = int(case["slots"] * case["load"]), case["n"]
    s["t"] = _table(case, kind)
    s["base"] = _keys(kind, 0, stored, seed)
    s["base_vals"] = _vals(kind, s["base"])
    g = _gen(seed)
    draw_ = torch.rand(n, generator=g, device="cuda")
    op = torch.where(draw_ < 0.5, L.OP_INSERT, torch.where(draw_ < 0.8, L.OP_FIND, L.OP_ERASE))
    # erases take distinct stored keys of the first half, lookups any of the second, inserts new ones
    half = max(1, stored // 2)
    leave = torch.cumsum((op == L.OP_ERASE).to(torch.int64), 0) - 1
    op[(op == L.OP_ERASE) & (leave >= half)] = L.OP_FIND
    idx = torch.where(op == L.OP_INSERT, torch.arange(n, dtype=torch.int64, device="cuda") + stored,
                      torch.where(op == L.OP_FIND, torch.randint(half, max(half + 1, stored), (n,), generator=g,
                                                                 device="cuda"), leave))
    s["keys"] = _keys_at(kind, idx, seed)
    s["vals"] = _vals(kind, s["keys"])
    s["ops"] = op.to(torch.uint8)


def _prepare_maintain(s, case, kind, seed):
    stored = int(case["slots"] * case["load"])
    s["t"] = _table(case, kind)
    s["n"] = stored
    for a in range(0, stored, 1 << 26):                                 # values are dense entry numbers
        n = min(1 << 26, stored - a)
        s["t"].insert(_keys(kind, a, n, seed),
                      torch.arange(a, a + n, dtype=KEY_TORCH[VAL_BYTES[kind]], device="cuda"), status=False)


def _prepare_host(s, case, kind, seed):
    stored, n = int(case["slots"] * case["load"]), case["n"]
    s["t"] = _table(case, kind)
    _fill(s["t"], kind, stored, seed)

    def host(t, dtype):
        t = t.cpu()
        return (t.pin_memory() if case["pinned"] else t).numpy().view(dtype)

    def room(dtype):
        t = torch.empty(n * np.dtype(dtype).itemsize, dtype=torch.uint8)
        return (t.pin_memory() if case["pinned"] else t).numpy().view(dtype)

    keys = _keys(kind, stored, n, seed)
    s["keys"] = host(keys, KEY_NUMPY[kind])
    s["queries"] = host(_some_absent(kind, stored, n, seed), KEY_NUMPY[kind])
    s["vals"] = host(_vals(kind, keys), VAL_NUMPY[kind]) if kind in VAL_BYTES else None
    s["status"], s["found"], s["gone"] = room(np.uint8), room(np.uint8), room(np.uint8)
    s["got"] = room(VAL_NUMPY[kind]) if kind in VAL_BYTES else None


# ------------------------------------------------------------------- run ---

def run(s):
    return globals()["_run_" + s["case"]["do"]](s)


def _run_find(s):
    return s["t"].find(s["q"])


def _run_step(s):
    t, b = s["t"], s["case"]["batch"]
    t.clear()
    out = torch.empty(s["keys"].numel(), dtype=torch.uint8, device="cuda")
    for a in range(0, s["keys"].numel(), b):
        t.insert(s["keys"][a:a + b], s["vals"][a:a + b] if s["vals"] is not None else None, out[a:a + b])
    return out, [t.find(q) for q in s["queries"]], t.erase(s["leave"])


def _run_frame(s):
    t = s["t"]
    found, _ = t.find(s["cand"], vals_out=False)
    t.insert_if_absent(s["cand"], s["index"], found, status=False)
    return found, t.find(s["cand"]), t.erase(s["leave"])


def _run_churn(s):
    t = s["t"]
    return t.insert(s["keys"], s["vals"]), t.find(s["queries"]), t.erase(s["keys"])


def _run_batch(s):
    s["batch"].launch()
    return s["status"], s["found"], s["got"], s["gone"]


def _run_ordered(s):
    t = s["t"]
    st = t.insert_ordered(s["keys"], s["vals"])
    return st, t.find(s["keys"]), t.erase_ordered(s["keys"])


def _run_mixed(s):
    t = s["t"]
    t.clear()
    t.insert(s["base"], s["base_vals"], status=False)
    return t.apply_mixed(s["ops"], s["keys"], s["vals"], vals_out=True)


def _run_maintain(s):
    t, n = s["t"], s["n"]
    t.rehash(s["case"]["slots"])
    _, vals, count = t.select(L.PRED_KEY_MASK, lo=15, hi=3, cap=max(1024, n // 4))
    flags = torch.zeros(n, dtype=torch.uint8, device="cuda")            # entry numbers of the selected class
    flags[vals[:int(count.item())].to(torch.int64)] = 1
    keys, vals = t.dump()
    table = torch.empty(n, dtype=torch.int64, device="cuda")            # the dump in the order of the entry numbers
    table[vals.to(torch.int64)] = keys
    return flags, table


def _run_host(s):
    t = s["t"]
    t.insert_host(s["keys"], s["vals"], s["status"])
    t.find_host(s["queries"], s["found"], s["got"])
    t.erase_host(s["keys"], s["gone"])
    got = None if s["got"] is None else s["got"].view(np.int64 if s["got"].itemsize == 8 else np.int32)
    return s["status"], s["found"], got, s["gone"]


# ------------------------------------------------------------------ work ---

def work(case):
    """Bytes that the operations cannot do without: each key and value read, each result written, and for every
    operation one 32-byte sector of the table read (and written, where a slot changes)."""
    kind = KIND_NAMES[case.get("kind", "map_i64_i32")]
    kb, vb = KEY_BYTES[kind], VAL_BYTES.get(kind, 0)
    ins, find, erase = kb + vb + 1 + 64, kb + vb + 1 + 32, kb + 1 + 64
    do, n = case["do"], case.get("n", 0)
    slots = case.get("slots", 0)
    stored = int(slots * case.get("load", 0))
    whole = slots * (kb + vb)
    if do == "find":
        b = n * find
    elif do == "step":
        b = whole + stored * ins + (2 * n if vb else n) * find + case["erase"] * erase
    elif do == "frame":
        new = 0.12 * n                                                  # about 1 in 8 samples falls outside the layers
        b = n * (kb + 1 + 32) + n + new * ins + n * find + n / 6 * erase
    elif do in ("churn", "host"):
        b = n * (ins + find + erase)
    elif do == "batch":
        mean = (2.0 ** TABLE_HI - 2.0 ** TABLE_LO) / ((TABLE_HI - TABLE_LO) * math.log(2.0))
        b = case["tables"] * mean * (0.3 * ins + 0.15 * find + 0.3 * erase)
    elif do == "ordered":
        b = n * (ins + find + erase)
    elif do == "mixed":
        b = whole + stored * (ins - 1) + n * (0.5 * (ins + 1 + vb) + 0.3 * (find + 1) + 0.2 * (erase + 1 + vb))
    else:                                                               # maintain: old and new arrays, select, dump
        b = 2 * whole + 2 * whole + stored * (1 + 8) + stored * 2 * (kb + vb) + stored / 16 * (kb + vb)
    return {"bytes": float(b), "flops": 0.0}
