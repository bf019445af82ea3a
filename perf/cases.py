"""Measured cases of the batch index: what its users have it do, through the public calls.

Every case is a dict of plain values. `kind` names the call:

* point: a stream of query batches on one index (`Index.execute`, its allocation-free form or
  its host-buffer form, by `entry`). Searches hit or miss; overwrites and deletes fall on keys
  of the index; `window` is a sliding window: each batch inserts keys that the index does not
  hold and deletes as many that an earlier batch inserted, so the index keeps its size and
  every batch adds nodes.
* range: a batch of range queries (`Index.range_search`).
* batching: one batch for each of many indices in one call (`MultiSet.execute`).
* serving: a burst of variable-size requests through the server (`Server.replay`).
* bulk: build an index from unsorted pairs and read it back whole (`Index`, `Index.export`).

States that take updates hold a short cycle of batches; a pass takes the next one. All inputs
are drawn from the seed. Keys are 63-bit and uniform (a bijection of 0, 1, 2, ...), or dense
ascending identifiers.

Every output is whole numbers, so there is no `exact`: results are equal or wrong.
"""
import json
import math
import os

import numpy as np
import torch

import paper_1601_00159_gb300 as pi

M63 = (1 << 63) - 1
CYCLE = 4  # batches of a state's stream
POINT = {"n": 1 << 20, "q": 1 << 14, "p": 0.25, "keys": "uniform", "theta": 0.0, "miss": 0.0, "over": 0.0,
         "delete": 0.0, "window": 0.0, "entry": "device"}


def _point(name, **kw):
    return dict(POINT, kind="point", name=name, **kw)


def listed():
    return [
        # the smallest calls: one user's few hundred lookups against a table that sits in L2
        _point("lookup_1k", n=50_021, q=1_000, miss=0.1),
        # the repository's tiny workload: half the searches miss
        _point("tiny_search", n=1 << 16, q=1 << 14, p=0.5, miss=0.5),
        # a latency-bound loop that may not allocate: a session store, mostly reads, some
        # writes, deletes that come back
        _point("noalloc_session", n=1 << 20, q=6_000, over=0.1, delete=0.05, theta=0.9, entry="noalloc"),
        # a key-value cache, uniform reads and overwrites in halves (YCSB A's mix), ragged sizes
        _point("cache_100k", n=3_000_017, q=100_003, p=0.125, over=0.5, miss=0.05),
        # append at the end and expire at the front: dense ascending identifiers
        _point("append_window", n=4_000_000, q=1 << 18, p=0.0625, keys="dense", window=0.3, miss=0.02),
        # the repository's mid workload: half searches, half membership changes, every batch
        # adds nodes
        _point("mid_window", n=1 << 24, q=1 << 20, window=0.25, miss=0.25),
        # the repository's skewed workload, its headline: hot keys, few updates
        _point("skewed", n=1 << 27, q=1 << 22, theta=0.99, over=0.05, delete=0.05),
        # batches that live in host memory: the copies are part of the call
        _point("host_1m", n=1 << 24, q=1 << 20, theta=0.9, over=0.05, entry="host"),
        # the paper's range experiment at 100 keys a range
        {"kind": "range", "name": "range_100", "n": 1 << 24, "q": 1 << 16, "span": 100},
        # the repository's many-index workload: 256 indices of 2^10 to 2^20 keys
        {"kind": "batching", "name": "batching_256", "count": 256, "n_lo": 1 << 10, "n_hi": 1 << 20, "q_lo": 1 << 8,
         "q_hi": 1 << 16, "window": 0.1},
        # a burst on the server: requests of 1 to 4096 queries
        {"kind": "serving", "name": "serving_burst", "n": 1 << 26, "requests": 4_000, "q_max": 4_096, "over": 0.05,
         "theta": 0.9},
        # load a table and dump it
        {"kind": "bulk", "name": "bulk_load", "n": 10_000_019, "p": 0.25},
    ]


def _spread(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi]."""
    return max(lo, min(hi, int(round(2 ** rng.uniform(math.log2(lo), math.log2(hi))))))


def draw(rng):
    kind = rng.choice(["point"] * 6 + ["range", "batching", "serving", "bulk"])
    if kind == "point":
        mix = rng.choice(["read", "update", "churn", "window"])
        entry = rng.choice(["device"] * 3 + ["noalloc", "host"])
        n = _spread(rng, 1 << 14, 1 << 25 if mix == "window" else 1 << 27)
        q_hi = min(1 << 16 if entry == "noalloc" else 1 << 22 if entry == "device" else 1 << 20, n)
        c = dict(POINT, kind="point", n=n, q=_spread(rng, 256, q_hi), entry=entry,
                 p=rng.choice([0.5, 0.25, 0.25, 0.125, 0.0625]), theta=rng.choice([0.0, 0.0, 0.8, 0.9, 0.99]))
        if rng.random() < 0.25:
            c["keys"] = "dense"
        if mix != "churn":
            c["miss"] = rng.choice([0.0, 0.1, 0.5])
        if mix == "update":
            c["over"] = rng.choice([0.05, 0.5])
        elif mix == "churn":
            c["over"], c["delete"] = rng.choice([(0.05, 0.05), (0.2, 0.1)])
        elif mix == "window":
            c["window"] = rng.choice([0.05, 0.1, 0.25])
            c["q"] = min(c["q"], n // 4)
            c["miss"] = min(c["miss"], 0.1)
        return c
    if kind == "range":
        n, span = _spread(rng, 1 << 18, 1 << 26), _spread(rng, 1, 1000)
        return {"kind": "range", "n": n, "q": _spread(rng, 256, min(1 << 17, (1 << 23) // span)), "span": span}
    if kind == "batching":
        n_hi = _spread(rng, 1 << 13, 1 << 20)
        return {"kind": "batching", "count": _spread(rng, 8, 256), "n_lo": _spread(rng, 1 << 10, 1 << 12), "n_hi": n_hi,
                "q_lo": 1 << 8, "q_hi": _spread(rng, 1 << 10, min(1 << 16, n_hi // 8)), "window": rng.choice([0.0, 0.1])}
    if kind == "serving":
        return {"kind": "serving", "n": _spread(rng, 1 << 20, 1 << 26), "requests": _spread(rng, 64, 4_000),
                "q_max": _spread(rng, 64, 4_096), "over": rng.choice([0.0, 0.05]), "theta": rng.choice([0.0, 0.9])}
    return {"kind": "bulk", "n": _spread(rng, 1 << 14, 10_000_019), "p": rng.choice([0.5, 0.25, 0.0625])}


# --------------------------------------------------------------------------------------
# Inputs


class _Draws:
    """Seeded draws on the GPU."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(int(seed) * 2 + 1)
        self.salt = (int(seed) * 0x9E3779B97F4A7C15 + 0x1234567) & M63

    def unit(self, n):
        return torch.rand(n, dtype=torch.float64, device="cuda", generator=self.g)

    def below(self, n, hi):
        return torch.randint(0, hi, (n,), dtype=torch.int64, device="cuda", generator=self.g)

    def bits(self, n):
        return torch.randint(-(1 << 62), 1 << 62, (n,), dtype=torch.int64, device="cuda", generator=self.g)

    def order(self, n):
        return torch.randperm(n, device="cuda", generator=self.g)

    def keys(self, i):
        """A bijection of [0, 2^63) on key numbers: steps that are each invertible modulo 2^63."""
        x = (i + self.salt) & M63
        for mul, shift in ((0x3F58476D1CE4E5B9, 29), (0x14D049BB133111EB, 31)):
            x = (x * mul) & M63
            x = x ^ (x >> shift)
        return x

    def ranks(self, n, q, theta):
        """Zipf(theta) ranks in [0, n), by Gray et al. (1994); uniform for theta 0. Ranks are
        scattered over the key numbers, so that hot keys lie anywhere."""
        if not theta:
            return self.below(q, n)
        zetan = _zeta(n, theta)
        u = self.unit(q)
        eta = (1 - (2 / n) ** (1 - theta)) / (1 - (1 + 2 ** -theta) / zetan)
        r = (n * (eta * u - eta + 1) ** (1 / (1 - theta))).long().clamp_(0, n - 1)
        uz = u * zetan
        r = torch.where(uz < 1 + 0.5 ** theta, torch.ones_like(r), r)
        r = torch.where(uz < 1, torch.zeros_like(r), r)
        a = (self.salt % n) | 1
        while math.gcd(a, n) != 1:
            a += 2
        return (r * a + self.salt % 1000003) % n


def _zeta(n, theta):
    """Sum of i^-theta for i = 1..n: the first terms, then Euler and Maclaurin's formula."""
    m = min(n, 100_000)
    s = float((np.arange(1, m + 1, dtype=np.float64) ** -theta).sum())
    if n > m:
        s += (n ** (1 - theta) - m ** (1 - theta)) / (1 - theta) + (n ** -theta - m ** -theta) / 2
    return s


def _numbered(d, c, i):
    """Keys number i: spread over the key space, or dense and ascending."""
    return d.keys(i) if c["keys"] == "uniform" else i * 16


def _stream(d, c, cycle):
    """The index's first pairs and `cycle` batches. Window batch r inserts segment r of the
    window's keys and deletes segment r - 2; the first pairs hold the last two segments, so the
    cycle goes round."""
    n, q = c["n"], c["q"]
    w = int(q * c["window"])
    seg = [torch.arange(n + r * w, n + (r + 1) * w, device="cuda") for r in range(cycle)]
    first = torch.arange(n, device="cuda")
    if w:
        first = torch.cat([first] + seg[-2:])
    keys = _numbered(d, c, first)
    vals = keys ^ d.salt
    del first
    batches = []
    for r in range(cycle):
        rest = q - 2 * w
        u = d.unit(rest)
        i = d.ranks(n, rest, c["theta"])
        k = _numbered(d, c, i)
        ops = torch.zeros(rest, dtype=torch.uint8, device="cuda")
        ops[u < c["over"] + c["delete"]] = pi.PI_OP_DELETE
        ops[u < c["over"]] = pi.PI_OP_INSERT
        miss = u >= 1 - c["miss"]
        k = torch.where(miss, k + 7 if c["keys"] == "dense" else d.keys(i + (1 << 40)), k)
        if w:
            k = torch.cat([k, _numbered(d, c, seg[r]), _numbered(d, c, seg[r - 2])])
            ops = torch.cat([ops, torch.full((w,), pi.PI_OP_INSERT, dtype=torch.uint8, device="cuda"),
                             torch.full((w,), pi.PI_OP_DELETE, dtype=torch.uint8, device="cuda")])
            o = d.order(q)
            k, ops = k[o], ops[o]
        batches.append((ops, k, d.bits(q)))
    return keys, vals, batches


def _window_stream(d, n, q, window):
    """_stream for one index of a set: uniform keys, hits and misses in halves."""
    return _stream(d, dict(POINT, n=n, q=q, window=window, miss=0.4), CYCLE)


def _tuned_classes():
    """The size classes of the package's committed tuning table."""
    with open(os.path.join(os.path.dirname(pi.__file__), "multi_tuning.json")) as f:
        return [tuple(c) for c in json.load(f)["classes"]]


def _sizes(c):
    """Index and batch sizes of a batching case, log-uniform and fixed by the case."""
    r = np.random.RandomState(c["count"])
    n = np.exp2(r.uniform(math.log2(c["n_lo"]), math.log2(c["n_hi"]), c["count"])).astype(int)
    q = np.exp2(r.uniform(math.log2(c["q_lo"]), math.log2(c["q_hi"]), c["count"])).astype(int)
    return n, q


def _requests(c):
    """Request sizes of a serving case, log-uniform in [1, q_max]."""
    u = np.random.RandomState(c["requests"]).uniform(0, math.log2(c["q_max"]), c["requests"])
    return np.maximum(1, np.exp2(u).astype(np.uint32))


def _range_sizes(c):
    """Keys in each range of a range case: around its span, from one up."""
    r = np.random.RandomState(c["q"])
    return np.maximum(1, r.poisson(c["span"], c["q"])).astype(np.int64)


def _host(t):
    return t.cpu().pin_memory()


def prepare(case, seed):
    c, d = case, _Draws(seed)
    s = {"kind": c["kind"], "at": 0}
    if c["kind"] == "point":
        keys, vals, s["batches"] = _stream(d, c, CYCLE)
        s["index"] = pi.Index(keys, vals, c["p"], seed)
        s["entry"] = c["entry"]
        if c["entry"] == "host":
            s["batches"] = [tuple(_host(t) for t in b) for b in s["batches"]]
            s["out"] = torch.empty((c["q"], 2), dtype=torch.int64, pin_memory=True)
        elif c["entry"] == "noalloc":
            s["out"] = torch.empty((c["q"], 2), dtype=torch.int64, device="cuda")
    elif c["kind"] == "range":
        keys = d.keys(torch.arange(c["n"], device="cuda"))
        s["index"] = pi.Index(keys, keys ^ d.salt, 0.25, seed)
        # some keys have been deleted: their nodes are still in place
        gone = keys[: c["n"] // 32]
        s["index"].execute(torch.full((gone.numel(),), pi.PI_OP_DELETE, dtype=torch.uint8, device="cuda"), gone, gone)
        # ranges that hold as many keys as the case says, from anywhere, in any order
        live = keys[c["n"] // 32:].sort().values
        size = torch.from_numpy(_range_sizes(c)).cuda()[d.order(c["q"])]
        at = (d.unit(c["q"]) * (live.numel() - size)).long()
        s["lo"], s["hi"] = live[at], live[at + size - 1] + 1
        s["cap"] = int(_range_sizes(c).sum())
    elif c["kind"] == "batching":
        rounds = [[] for _ in range(CYCLE)]
        s["indices"] = []
        s["out"] = torch.empty((int(_sizes(c)[1].sum()), 2), dtype=torch.int64, device="cuda")
        at = 0
        for i, (n, q) in enumerate(zip(*_sizes(c))):
            keys, vals, bs = _window_stream(d, int(n), int(q), c["window"])
            s["indices"].append(pi.Index(keys, vals, 0.25, seed + i))
            for r, b in enumerate(bs):
                rounds[r].append((i, *b, s["out"][at:at + int(q)]))
            at += int(q)
        s["set"] = pi.MultiSet(s["indices"], _tuned_classes())
        s["rounds"] = [s["set"].prepare(r) for r in rounds]
    elif c["kind"] == "serving":
        keys = d.keys(torch.arange(c["n"], device="cuda"))
        s["index"] = pi.Index(keys, keys ^ d.salt, 0.25, seed)
        s["sizes"] = _requests(c)
        q = int(s["sizes"].sum())
        s["keys"] = d.keys(d.ranks(c["n"], q, c["theta"])).cpu().numpy().view(np.uint64)
        s["ops"] = (d.unit(q) < c["over"]).to(torch.uint8).cpu().numpy()
        s["vals"] = d.bits(q).cpu().numpy().view(np.uint64)
        s["arrivals"] = np.zeros(len(s["sizes"]))
        s["server"] = pi.Server(s["index"], max_batch=1 << 20, slots=3)
    else:
        i = torch.arange(c["n"], device="cuda")
        k = (c["n"] + 96) // 97  # one key in 97 comes twice, the second time somewhere else: the last value counts
        i[:: 97] = 97 * (d.order(k) % (k - 1)) + 1
        s["keys"], s["vals"] = d.keys(i), d.bits(c["n"])
        s["p"], s["seed"] = c["p"], seed
    return s


def run(s):
    kind = s["kind"]
    if kind == "point":
        b = s["batches"][s["at"] % CYCLE]
        s["at"] += 1
        if s["entry"] == "device":
            return s["index"].execute(*b)
        if s["entry"] == "noalloc":
            return s["index"].execute_noalloc(*b, s["out"])
        return s["index"].execute_host(*b, s["out"])
    if kind == "range":
        return s["index"].range_search(s["lo"], s["hi"], cap=s["cap"])
    if kind == "batching":
        s["set"].execute(s["rounds"][s["at"] % CYCLE])
        s["at"] += 1
        return s["out"]
    if kind == "serving":
        return s["server"].replay(s["ops"], s["keys"], s["vals"], s["sizes"], s["arrivals"])[0]
    index = pi.Index(s["keys"], s["vals"], s["p"], s["seed"])
    pairs = index.export()
    index.close()
    return pairs


def _distinct(n, q, theta):
    """Distinct keys expected among q draws of Zipf(theta) ranks in [0, n)."""
    if not theta:
        return n * -math.expm1(-q / n)
    e = np.unique(np.concatenate([np.arange(1, 65), np.geomspace(64, n + 1, 4096)]).astype(np.int64)).astype(np.float64)
    lo, hi = e[:-1], e[1:]
    pr = ((lo + hi - 1) / 2) ** -theta / _zeta(n, theta)
    return float(((hi - lo) * -np.expm1(-q * pr)).sum())


def _point_bytes(n, q, theta, inserts, deletes, window):
    """Each query's op, key and result; an inserted value; a key and a value (16 B) and a state
    byte of every distinct key looked up; a pair and a state byte of every key written."""
    d = min(q, _distinct(n, q * (1 - 2 * window), theta) + 2 * window * q)
    return q * 25 + 8 * inserts + 17 * d + 17 * min(d, inserts) + min(d, deletes)


def work(case):
    c = case
    if c["kind"] == "point":
        b = _point_bytes(c["n"], c["q"], c["theta"], c["q"] * (c["over"] + c["window"]),
                         c["q"] * (c["delete"] + c["window"]), c["window"])
    elif c["kind"] == "range":
        b = c["q"] * 24 + int(_range_sizes(c).sum()) * 33
    elif c["kind"] == "batching":
        b = sum(_point_bytes(n, q, 0.0, q * c["window"], q * c["window"], c["window"]) for n, q in zip(*_sizes(c)))
    elif c["kind"] == "serving":
        q = int(_requests(c).sum())
        b = _point_bytes(c["n"], q, c["theta"], q * c["over"], 0, 0.0)
    else:
        b = c["n"] * (16 + 17 + 16 + 16)
    return {"bytes": float(b), "flops": 0.0}
