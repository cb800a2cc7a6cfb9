"""Performance cases of the GPU LSM dictionary: what a program that uses the library has it do.

A case is one pass over the public Python layer (``gpulsm.LSM`` / ``gpulsm.MultiLSM``) with its inputs on the
device.  Kinds:

  update    an empty dictionary takes its batches one call each (``insert`` without deletes, ``update`` with
            them), then answers lookups
  load      one ``insert`` call of many batches' worth of pairs, then lookups
  bulk      ``bulk_build`` of all pairs, then lookups
  cleanup   update batches, then ``cleanup``, then lookups
  lookup    point queries on a dictionary built beforehand
  count     interval counts on a dictionary built beforehand
  range     interval contents on a dictionary built beforehand
  session   a small dictionary's life: mixed and ordered batches, then each kind of query once
  batched   rounds of one batch and one set of lookups for many dictionaries (``MultiLSM``)

Fields: ``b`` batch size, ``n`` operations in all (the last batch is short when b does not divide n), ``deletes``
their fraction of the operations after the first batch, ``dist`` of the keys (uniform, or Zipf(1.1) over the key
space), ``space`` the keys' bound, ``nq`` queries, ``expect`` results expected per interval.
"""

import math

import numpy as np
import torch

from paper_1707_05354_gb300 import gpulsm

TOP = (1 << 31) - 1   # keys are below it


def listed():
    return [
        # the paper's insertion experiment (its Table II row b = 2^20): 128 batches of uniform 31-bit keys, then
        # 2^24 lookups, half of them hits, on the one full level that is left
        dict(name="insert_2p20", kind="update", b=1 << 20, n=1 << 27, deletes=0.0, dist="uniform", space=TOP,
             nq=1 << 24, expect=0),
        # a stream of small mixed batches (the sweep's smallest b, a quarter deletes, 30-bit keys): many launches
        # for little work each; the last batch is short
        dict(name="update_2p16", kind="update", b=1 << 16, n=(1 << 24) - 12345, deletes=0.25, dist="uniform",
             space=1 << 30, nq=1 << 21, expect=0),
        # skewed keys (the sweep's Zipf points): hot keys repeat many times within a batch and across levels
        dict(name="update_zipf_2p18", kind="update", b=1 << 18, n=1 << 23, deletes=0.25, dist="zipf",
             space=1 << 30, nq=1 << 20, expect=0),
        # few large batches, no power of two (the sweep's upper end, above the batch size of the bucket sort)
        dict(name="update_3m", kind="update", b=3000000, n=48000000, deletes=0.1, dist="uniform", space=TOP,
             nq=1 << 22, expect=0),
        # loading a dictionary of records by their ids (whole numbers below 2^25, not spread over all 31 bits): one
        # call with all pairs, cut into 39 batches inside
        dict(name="load_ids_10m", kind="load", b=1 << 18, n=10000000, deletes=0.0, dist="uniform", space=1 << 25,
             nq=1 << 20, expect=0),
        # building a dictionary at once from unsorted pairs (the paper's bulk build)
        dict(name="bulk_50m", kind="bulk", b=1 << 20, n=50000001, deletes=0.0, dist="uniform", space=TOP,
             nq=1 << 22, expect=0),
        # the paper's cleanup experiment: half of the operations deletes, all 31 batches merged and compacted
        dict(name="cleanup_31x2p20", kind="cleanup", b=1 << 20, n=31 << 20, deletes=0.5, dist="uniform",
             space=1 << 30, nq=1 << 22, expect=0),
        # the lookups' worst case: seven full levels, so that a miss probes all seven
        dict(name="lookup_7_levels", kind="lookup", b=1 << 20, n=127 << 20, deletes=0.0, dist="uniform", space=TOP,
             nq=1 << 24, expect=0),
        # counts of short intervals over four levels (the paper's Table IV, L = 8)
        dict(name="count_4_levels", kind="count", b=1 << 18, n=85 << 18, deletes=0.25, dist="uniform",
             space=1 << 30, nq=1 << 22, expect=8),
        # contents of longer intervals over several levels with deleted keys in them
        dict(name="range_64", kind="range", b=1 << 16, n=363 << 16, deletes=0.25, dist="uniform", space=1 << 30,
             nq=200000, expect=64),
        # the smallest calls: a thousand operations or queries each, where launches and waits are the cost
        dict(name="session_1k", kind="session", b=1000, n=15900, deletes=0.1, dist="uniform", space=1 << 20,
             nq=4096, expect=8),
        # many dictionaries of uneven sizes (1024 to 2^18, no powers of two), eight rounds of a batch and its lookups
        dict(name="batched_128", kind="batched", b=1 << 18, n=8, deletes=0.2, dist="uniform", space=TOP, nq=128,
             expect=0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["update", "update", "update", "load", "bulk", "cleanup", "lookup", "lookup", "count", "range",
                       "session", "batched"])
    c = dict(kind=kind, deletes=rng.choice([0.0, 0.1, 0.25, 0.5]), dist="uniform",
             space=rng.choice([TOP, 1 << 30, _log(rng, 1 << 25, TOP)]), expect=0)
    if kind == "session":
        c.update(b=_log(rng, 16, 8192), nq=_log(rng, 64, 16384), expect=_log(rng, 1, 64))
        c["n"] = c["b"] * rng.randint(2, 24) - rng.randint(0, c["b"] - 1)
    elif kind == "batched":
        c.update(b=_log(rng, 1 << 12, 1 << 18), n=rng.randint(2, 8), nq=_log(rng, 8, 128))
    else:
        c["b"] = _log(rng, 1 << 10, 1 << 22)
        most = 127 if kind in ("update", "cleanup") else 255 if kind == "load" else 1023
        c["n"] = max(c["b"], min(_log(rng, 1 << 16, 1 << 25), c["b"] * most))
        if c["space"] < 1 << 28:   # ids: no more of them than in the listed case
            c["n"] = min(c["n"], 1 << 22)
            c["b"] = min(c["b"], c["n"])
        c["nq"] = _log(rng, 1 << 10, 1 << 22)
        if kind in ("load", "bulk"):
            c["deletes"] = 0.0
        elif kind == "update":
            c["dist"] = rng.choice(["uniform", "uniform", "zipf"])
            if c["dist"] == "zipf":
                c["n"] = min(c["n"], 1 << 23)
        elif kind in ("count", "range"):
            c["expect"] = _log(rng, 1, 512)
            c["nq"] = max(1024, min(c["nq"], (1 << 24) // c["expect"]))
    return c


# ------------------------------------------------------------------- inputs --
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _u32(g, n):
    return torch.randint(-(1 << 31), 1 << 31, (n,), generator=g, device="cuda", dtype=torch.int32)


def _keys(g, n, case):
    space = case["space"]
    if case["dist"] == "zipf":   # continuous power law over the ranks, ranks spread over the keys by an odd factor
        u = torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
        rank = torch.floor(((float(space) ** -0.1 - 1.0) * u + 1.0) ** -10.0).clamp_(1, space).to(torch.int64)
        return ((rank * 0x9E3779B1) % space).to(torch.int32)
    return torch.randint(0, space, (n,), generator=g, device="cuda", dtype=torch.int32)


def _ops(g, case):
    """(keys, values, delete flags): from the second batch on, deletes name keys drawn from the operations before
    their batch, so that most of them hit a stored key."""
    n, b = case["n"], case["b"]
    keys, vals = _keys(g, n, case), _u32(g, n)
    if case["deletes"] <= 0:
        return keys, vals, None
    at = torch.arange(n, device="cuda", dtype=torch.int64)
    first = at // b * b
    flag = (torch.rand(n, generator=g, device="cuda") < case["deletes"]) & (first > 0)
    back = (torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * first).to(torch.int64)
    return torch.where(flag, keys[back], keys), vals, flag.to(torch.uint8)


def _queries(g, keys, nq, case):
    """Half of the queries are keys of the operations, half uniform over the key space."""
    hits = keys[torch.randint(0, keys.numel(), (nq // 2,), generator=g, device="cuda")]
    rest = torch.randint(0, case["space"], (nq - nq // 2,), generator=g, device="cuda", dtype=torch.int32)
    q = torch.cat([hits, rest])
    return q[torch.randperm(nq, generator=g, device="cuda")]


def _intervals(g, nq, case, stored):
    """Intervals expecting `expect` results at the stored keys' density (widths from half to one and a half of it)."""
    width = max(1.0, case["expect"] * case["space"] / max(1, stored))
    k1 = torch.randint(0, case["space"], (nq,), generator=g, device="cuda", dtype=torch.int64)
    w = (torch.rand(nq, generator=g, device="cuda", dtype=torch.float64) + 0.5) * width
    k2 = torch.clamp(k1 + w.to(torch.int64), max=TOP - 1)
    return k1.to(torch.int32), k2.to(torch.int32)


def _batches(case):
    return [(s, min(s + case["b"], case["n"])) for s in range(0, case["n"], case["b"])]


def _make(seed, case):
    g = _gen(seed)
    s = dict(zip(("keys", "vals", "flag"), _ops(g, case)))
    first = min(case["b"], case["n"])   # holds no deletes; of the rest a share of (1 - d) / (1 + d) stays alive
    stored = first + (case["n"] - first) * (1.0 - case["deletes"]) / (1.0 + case["deletes"])
    s["k1"], s["k2"] = _intervals(g, case["nq"], case, stored) if case["expect"] else (None, None)
    s["q"] = _queries(g, s["keys"], case["nq"], case)
    return s


def _sizes(case):
    """Batch sizes of the dictionaries: log-uniform whole numbers from 1024 to b, the same for every seed."""
    u = np.random.default_rng(case["nq"]).uniform(10.0, math.log2(case["b"]), size=case["nq"])
    return np.rint(np.exp2(u)).astype(np.int64)


def _make_batched(seed, case):
    """One entry per round: keys, values, flags and queries of all dictionaries back to back."""
    g = _gen(seed)
    sizes = _sizes(case)
    tot = int(sizes.sum())
    off = torch.from_numpy(np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)).cuda()
    rounds = []
    for t in range(case["n"]):
        keys, vals = _keys(g, tot, case), _u32(g, tot)
        flag = torch.zeros(tot, dtype=torch.uint8, device="cuda")
        if t:   # deletes of keys that the same dictionary got in an earlier round
            flag = (torch.rand(tot, generator=g, device="cuda") < case["deletes"]).to(torch.uint8)
            old = rounds[int(torch.randint(0, t, (1,), generator=g, device="cuda"))][0]
            keys = torch.where(flag.bool(), old, keys)
        old = rounds[t // 2][0] if t else keys
        pick = torch.rand(tot, generator=g, device="cuda") < 0.5
        rounds.append((keys, vals, flag, torch.where(pick, old, _keys(g, tot, case))))
    return sizes, off, rounds


def _apply(d, s, case):
    for a, z in _batches(case):
        if s["flag"] is None:
            d.insert(s["keys"][a:z], s["vals"][a:z])
        else:
            d.update(s["keys"][a:z], s["vals"][a:z], s["flag"][a:z])


def _room(case):
    return 2 * case["expect"] * case["nq"] + 1024


def _range(s):
    rows, cap = s["rows"], s["rows"][1].numel()
    status, _ = gpulsm.lsm_range(s["d"].h, s["k1"].data_ptr(), s["k2"].data_ptr(), s["k1"].numel(),
                                 *(x.data_ptr() for x in rows), cap, torch.cuda.current_stream().cuda_stream)
    if status != gpulsm.LSM_OK:
        raise gpulsm.LSMError(status, "lsm_range")
    return rows


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batched":
        sizes, off, rounds = _make_batched(seed, case)
        return dict(case=case, off=off, rounds=rounds, d=gpulsm.MultiLSM(sizes.tolist(), case["n"]))
    s = _make(seed, case)
    s["case"] = case
    s["d"] = gpulsm.LSM(case["b"], -(-case["n"] // case["b"]) * case["b"])
    if kind in ("range", "session"):   # offsets, keys and values: buffers with room for twice the results expected
        s["rows"] = [torch.zeros(case["nq"] + 1, dtype=torch.int64, device="cuda")]
        s["rows"] += [torch.zeros(_room(case), dtype=torch.int32, device="cuda") for _ in range(2)]
    if kind in ("lookup", "count", "range"):
        _apply(s["d"], s, case)
        s["keys"] = s["vals"] = s["flag"] = None   # a program that queries keeps the dictionary, not its history
    return s


def run(s):
    case, d = s["case"], s["d"]
    kind = case["kind"]
    if kind == "lookup":
        return d.lookup(s["q"])
    if kind == "count":
        return d.count(s["k1"], s["k2"])
    if kind == "range":
        return _range(s)
    if kind == "batched":
        d.reset()
        out = []
        for keys, vals, flag, q in s["rounds"]:
            d.update(keys, vals, flag)
            out.append(d.lookup(q, s["off"]))
        return out
    gpulsm.lsm_reset(d.h)
    if kind == "session":
        for t, (a, z) in enumerate(_batches(case)):
            flag = s["flag"][a:z] if s["flag"] is not None else torch.zeros(z - a, dtype=torch.uint8, device="cuda")
            (d.update_ordered if t % 4 == 3 else d.update)(s["keys"][a:z], s["vals"][a:z], flag)
        return (d.lookup(s["q"]), d.count(s["k1"], s["k2"]), _range(s), d.neighbor(s["q"], True),
                d.neighbor(s["q"], False))
    if kind == "load":
        d.insert(s["keys"], s["vals"])
    elif kind == "bulk":
        d.bulk_build(s["keys"], s["vals"])
    else:
        _apply(d, s, case)
        if kind == "cleanup":
            d.cleanup()
    val, found = d.lookup(s["q"])
    return dict(val=val, found=found, r=d.r)


# --------------------------------------------------------------------- work --
def _fold_bytes(n, b):
    """Batch t ends in level k = ffz(t), 2^k b pairs, each read once and written once there (8 bytes a pair)."""
    return sum(16.0 * b * ((~t & (t + 1)) or 1) for t in range(-(-n // b)))


def work(case):
    """Bytes that the path cannot do without.  Updates: the batches through the binary counter's levels.  Queries:
    their inputs and outputs, a 32-byte sector of keys per query (the levels a query has to look into beyond one
    depend on the data) and one of values per hit."""
    n, b, nq, kind = case["n"], case["b"], case["nq"], case["kind"]
    lookups = nq * (4 + 5 + 32 + 16)
    if kind == "batched":
        mean = (case["b"] - 1024) / max(0.1, math.log(case["b"] / 1024))   # of log-uniform sizes
        return dict(bytes=nq * mean * (_fold_bytes(n, 1) + n * (1 + 57)), flops=0)
    if kind == "lookup":
        return dict(bytes=lookups, flops=0)
    if kind == "count":
        return dict(bytes=nq * (8 + 4 + 32), flops=0)
    if kind == "range":
        return dict(bytes=nq * (8 + 8 + 16.0 * case["expect"]), flops=0)
    if kind in ("load", "bulk"):
        return dict(bytes=16.0 * n + lookups, flops=0)
    each = 16.0 * n if kind == "cleanup" else 0.0
    if kind == "session":
        each = nq * (12 + 16 + 8.0 * case["expect"] + 2 * 13 + 4 * 32)
    return dict(bytes=_fold_bytes(n, b) + lookups + each, flops=0)


# -------------------------------------------------------------------- exact --
def _live(keys, vals, flag, b, ordered=()):
    """(sorted live keys, their values), as 64-bit whole numbers: the last batch that names a key decides; within it
    a delete beats the inserts and the last insert wins, or in an ordered batch the last operation."""
    n = keys.numel()
    at = torch.arange(n, device=keys.device)
    keys = keys.long()
    flag = torch.zeros_like(keys) if flag is None else flag.long()
    late = flag.clone()
    for t in ordered:
        late[t * b:(t + 1) * b] = 0
    order = torch.argsort((at // b) * 2 + late, stable=True)
    order = order[torch.argsort(keys[order], stable=True)]
    k = keys[order]
    last = torch.ones(n, dtype=torch.bool, device=k.device)
    last[:-1] = k[1:] != k[:-1]
    keep = order[last]
    keep = keep[flag[keep] == 0]
    return keys[keep], vals[keep].long()


def _exact_lookup(live, q):
    k, v = live
    if not k.numel():
        return torch.zeros_like(q), torch.zeros(q.numel(), dtype=torch.uint8, device=q.device)
    q = q.long()
    i = torch.searchsorted(k, q).clamp_(max=k.numel() - 1)
    hit = k[i] == q
    return torch.where(hit, v[i], torch.zeros_like(q)).to(torch.int32), hit.to(torch.uint8)


def _exact_bounds(live, k1, k2):
    lo = torch.searchsorted(live[0], k1.long())
    return lo, torch.searchsorted(live[0], k2.long(), right=True)


def _exact_range(live, k1, k2, room):
    lo, hi = _exact_bounds(live, k1, k2)
    off = torch.zeros(k1.numel() + 1, dtype=torch.int64, device=lo.device)
    off[1:] = torch.cumsum(hi - lo, 0)
    at = torch.repeat_interleave(lo - off[:-1], hi - lo) + torch.arange(int(off[-1]), device=lo.device)
    rows = torch.zeros((2, room), dtype=torch.int32, device=lo.device)
    rows[0, :at.numel()], rows[1, :at.numel()] = live[0][at].to(torch.int32), live[1][at].to(torch.int32)
    return [off, rows[0], rows[1]]


def _exact_neighbor(live, q, successor):
    k, v = live
    i = torch.searchsorted(k, q.long()) if successor else torch.searchsorted(k, q.long(), right=True) - 1
    hit = (i >= 0) & (i < k.numel())
    i = i.clamp(0, max(0, k.numel() - 1))
    if not k.numel():
        return torch.zeros_like(q), torch.zeros_like(q), hit.to(torch.uint8)
    zero = torch.zeros_like(i)
    return (torch.where(hit, k[i], zero).to(torch.int32), torch.where(hit, v[i], zero).to(torch.int32),
            hit.to(torch.uint8))


def exact(case, seed):
    kind, b = case["kind"], case["b"]
    if kind == "batched":
        sizes, off, rounds = _make_batched(seed, case)
        owner = torch.repeat_interleave(torch.arange(len(sizes), device="cuda"), torch.from_numpy(sizes).cuda()) << 32
        out, tot = [], int(off[-1])
        for t in range(case["n"]):
            seen = rounds[:t + 1]
            live = _live(torch.cat([owner | r[0].long() for r in seen]), torch.cat([r[1] for r in seen]),
                         torch.cat([r[2] for r in seen]), tot)
            out.append(_exact_lookup(live, owner | rounds[t][3].long()))
        return out
    s = _make(seed, case)
    nb = len(_batches(case))
    live = _live(s["keys"], s["vals"], s["flag"], b, [t for t in range(nb) if t % 4 == 3] if kind == "session" else ())
    if kind == "lookup":
        return _exact_lookup(live, s["q"])
    if kind == "count":
        lo, hi = _exact_bounds(live, s["k1"], s["k2"])
        return (hi - lo).to(torch.int32)
    if kind == "range":
        return _exact_range(live, s["k1"], s["k2"], _room(case))
    if kind == "session":
        lo, hi = _exact_bounds(live, s["k1"], s["k2"])
        rows = _exact_range(live, s["k1"], s["k2"], _room(case))
        return (_exact_lookup(live, s["q"]), (hi - lo).to(torch.int32), rows, _exact_neighbor(live, s["q"], True),
                _exact_neighbor(live, s["q"], False))
    val, found = _exact_lookup(live, s["q"])
    r = -(-live[0].numel() // b) if kind in ("bulk", "cleanup") else nb
    return dict(val=val, found=found, r=r)
