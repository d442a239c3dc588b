"""The calls whose speed counts: what programs that use this library do, from the smallest call to the largest.

Every case goes through the public binding (``paper_1910_06416_gb300.recsplit``) with the launch shapes a
process starts with.  Keys are the seeded streams of ``paper_1910_06416_gb300.inputs`` made on the device:
64-bit outputs of splitmix64, and random byte strings of 8 to 32 bytes.  Kinds:

* ``build``: one structure from n keys in device or page-locked host memory, serialized (the words that a program
  stores or ships), then released.
* ``batch``: structures of many key sets of mixed sizes and parameters in one pass, each serialized, then released.
* ``lookup``: q queries (members, uniform with replacement) against one resident structure.
* ``lookup_batch``: q (structure id, key) queries against many resident structures.
* ``serve``: a round of the serving engine: builds and lookups submitted together, results collected as they complete.
"""
import math

import numpy as np
import torch

from paper_1910_06416_gb300 import inputs
from paper_1910_06416_gb300 import recsplit as rs

DEV = "cuda:0"
# 32-bit integer operations of one evaluation of the hash family: two xors, a 64-bit multiply (three), a 64-bit
# xorshift (four), the high word of a 64-bit multiply (three)
OPS = 12


def listed():
    return [
        # the smallest key sets of a batch, built alone: a request of a thousand keys, latency counts
        {"name": "build_1e3", "kind": "build", "key": "u64", "host": False, "n": 1000, "leaf": 8, "bucket": 100,
         "extra": 0},
        # the fast, compact-enough parameters (l = 5, b = 5) on 10^5 keys
        {"name": "build_1e5_l5_b5", "kind": "build", "key": "u64", "host": False, "n": 100000, "leaf": 5,
         "bucket": 5, "extra": 0},
        # the headline construction: 10^7 strings, l = 8, b = 100
        {"name": "build_strings_1e7", "kind": "build", "key": "bytes", "host": False, "n": 10000000, "leaf": 8,
         "bucket": 100, "extra": 0},
        # the space-optimal parameters: l = 16, b = 2000 on 10^6 keys (1.56 bits per key)
        {"name": "build_1e6_l16_b2000", "kind": "build", "key": "u64", "host": False, "n": 1000000, "leaf": 16,
         "bucket": 2000, "extra": 0},
        # the non-minimal variant, range 1.26 n, an odd number of keys
        {"name": "build_perfect_3e6_e2", "kind": "build", "key": "u64", "host": False, "n": 3000017, "leaf": 8,
         "bucket": 100, "extra": 2},
        # end to end from page-locked host memory, as a loader hands strings over
        {"name": "build_host_strings_1e6", "kind": "build", "key": "bytes", "host": True, "n": 1000000, "leaf": 8,
         "bucket": 100, "extra": 0},
        # many structures at once: sizes 10^3 .. 10^6, l in {5, 8, 12}, b in {5, 100, 2000}
        {"name": "batch_48", "kind": "batch", "count": 48, "lo": 1000, "hi": 1000000},
        # a handful of queries against a resident structure: latency counts
        {"name": "lookup_1e3", "kind": "lookup", "key": "u64", "n": 1000000, "leaf": 8, "bucket": 100, "extra": 0,
         "q": 1000},
        # an ordinary batch of 64-bit queries, ragged
        {"name": "lookup_1e6", "kind": "lookup", "key": "u64", "n": 10000000, "leaf": 8, "bucket": 100, "extra": 0,
         "q": 1000003},
        # the headline lookup: 10^8 string queries against 10^7 strings
        {"name": "lookup_strings_1e8", "kind": "lookup", "key": "bytes", "n": 10000000, "leaf": 8, "bucket": 100,
         "extra": 0, "q": 100000000},
        # queries over many resident structures in one launch
        {"name": "lookup_batch_1e7", "kind": "lookup_batch", "count": 256, "lo": 1000, "hi": 100000,
         "q": 10000000},
        # a round of the serving engine: three builds and three lookups of strings, from page-locked memory
        {"name": "serve_round", "kind": "serve", "n": 200000, "builds": 3, "build_lo": 10000, "build_hi": 500000,
         "lookups": 3, "q_lo": 1000, "q_hi": 100000},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["build", "build", "build", "batch", "lookup", "lookup", "lookup", "lookup_batch"])
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(2, 60), "lo": 1000, "hi": _log_int(rng, 3000, 1000000)}
    if kind == "lookup_batch":
        return {"kind": kind, "count": rng.randint(2, 300), "lo": 1000, "hi": _log_int(rng, 3000, 100000),
                "q": _log_int(rng, 1000, 10000000)}
    leaf = rng.choice([2, 3, 4, 5, 6, 7, 8, 8, 8, 9, 10, 11, 12, 14, 16])
    bucket = _log_int(rng, 5, 2000)
    extra = rng.choice([0, 0, 0, 0, 1, 2, 4, 8]) if leaf <= 12 else 0
    n = _log_int(rng, 1000, 10000000)
    most = 2e11 if kind == "build" else 4e10  # evaluations: a fifth of the largest listed build; less to prepare a lookup
    n = max(1000, min(n, int(n * most / max(1.0, _evaluations(n, leaf, bucket, extra)))))
    key = rng.choice(["u64", "u64", "bytes"])
    if kind == "build":
        return {"kind": kind, "key": key, "host": rng.random() < 0.25, "n": n, "leaf": leaf, "bucket": bucket,
                "extra": extra}
    return {"kind": kind, "key": key, "n": n, "leaf": leaf, "bucket": bucket, "extra": extra,
            "q": _log_int(rng, 100, 100000000 if key == "u64" else 30000000)}


# ---------------------------------------------------------------- inputs
def _mix_seed(seed, what):
    return (seed * 1000003 + what * 7919 + 12345) & 0x7FFFFFFFFFFF


def _u64(n, seed):
    return inputs.device_splitmix64(seed, n, device=DEV)


def _below(seed, count, m, start=0):
    """`count` integers uniform in [0, m), m < 2^31."""
    z = inputs.device_splitmix64(seed, count, start, device=DEV)
    return (((z >> 32) & 0xFFFFFFFF) * m) >> 32


def _strings(n, seed):
    """n random strings of 8 to 32 bytes: their 32-byte padded rows and lengths."""
    rows = inputs.device_splitmix64(seed ^ 0x5A5A5A5A, 4 * n, device=DEV).view(torch.uint8).view(n, 32)
    return rows, 8 + _below(seed, n, 25)


def _pack(rows, lengths, idx=None):
    """Packed bytes and offsets (n + 1) of rows[idx] (of all rows without idx)."""
    n = (lengths if idx is None else idx).shape[0]
    ln = lengths if idx is None else lengths[idx]
    offsets = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(ln, 0, out=offsets[1:])
    data = torch.empty(int(offsets[-1]), dtype=torch.uint8, device=DEV)
    col = torch.arange(32, device=DEV, dtype=torch.int64)
    step = 1 << 23
    for a in range(0, n, step):
        b = min(n, a + step)
        r = rows[a:b] if idx is None else rows[idx[a:b]]
        data[int(offsets[a]):int(offsets[b])] = r[col[None, :] < ln[a:b, None]]
    return data, offsets


def _sets(case, seed):
    """Key sets of a batch: (keys, leaf, bucket), sizes log-uniform; the sizes are the workload's, the keys the seed's."""
    return [(_u64(n, (key_seed ^ seed) & 0x7FFFFFFFFFFFFFFF), leaf, bucket)
            for n, leaf, bucket, key_seed in inputs.batch_sets(case["count"], case["lo"], case["hi"], 3)]


def _sizes(count, lo, hi):
    """`count` sizes spread over [lo, hi] by their logarithm."""
    return [int(round(lo * (hi / lo) ** (i / max(1, count - 1)))) + i for i in range(count)]


class _Handles:
    """Structures of a batch, released with the state that holds them."""

    def __init__(self, handles):
        self.handles = handles

    def __del__(self):
        for h in self.handles:
            rs.recsplit_free(h)


class _Server:
    def __init__(self):
        self.srv = rs.recsplit_server_create()

    def __del__(self):
        rs.recsplit_server_destroy(self.srv)


def _slab(n):
    """Host memory that a structure of n keys is stored into (at most about 4 bits per key, and the header)."""
    return np.zeros(n // 10 + 64, dtype=np.int64)


def _store(words, slab):
    slab[:words.shape[0]] = words.view(np.int64)
    return slab


def prepare(case, seed):
    torch.cuda.set_device(0)
    kind = case["kind"]
    s1, s2 = _mix_seed(seed, 1), _mix_seed(seed, 2)
    if kind == "build":
        keys = (_u64(case["n"], s1),) if case["key"] == "u64" else _pack(*_strings(case["n"], s1))
        if case["host"]:
            keys = tuple(k.cpu().pin_memory() for k in keys)
        return {"case": case, "keys": keys, "slab": _slab(case["n"])}
    if kind == "batch":
        sets = _sets(case, s1)
        return {"case": case, "sets": sets, "slabs": [_slab(k.shape[0]) for k, _, _ in sets]}
    if kind == "lookup":
        q = case["q"]
        idx = _below(s2, q, case["n"])
        if case["key"] == "u64":
            keys = _u64(case["n"], s1)
            s = rs.Structure.build_perfect_u64(keys, case["leaf"], case["bucket"], case["extra"])
            queries = (keys[idx],)
        else:
            rows, lengths = _strings(case["n"], s1)
            s = rs.Structure.build_perfect_bytes(*_pack(rows, lengths), case["leaf"], case["bucket"], case["extra"])
            queries = _pack(rows, lengths, idx)
        return {"case": case, "s": s, "queries": queries, "out": torch.empty(q, dtype=torch.int64, device=DEV)}
    if kind == "lookup_batch":
        q = case["q"]
        sets = _sets(case, s1)
        owner = _Handles(rs.recsplit_build_batch(sets))
        base = torch.tensor(np.cumsum([0] + [k.shape[0] for k, _, _ in sets]), device=DEV)
        g = _below(s2, q, int(base[-1]))  # any key of any set: larger sets are asked more often
        ids = torch.searchsorted(base, g, right=True) - 1
        return {"case": case, "owner": owner, "ids": ids.to(torch.int32),
                "keys": torch.cat([k for k, _, _ in sets])[g], "out": torch.empty(q, dtype=torch.int64, device=DEV)}
    # serve: a resident structure of n strings, host buffers of the round's requests
    rows, lengths = _strings(case["n"], s1)
    server = _Server()
    host = tuple(t.cpu().pin_memory() for t in _pack(rows, lengths))
    rs.recsplit_server_submit_build_bytes(server.srv, *host, 8, 100)
    resident = _collect(server.srv, 1)[0]["structure_id"]
    builds = [tuple(t.cpu().pin_memory() for t in _pack(*_strings(n, _mix_seed(seed, 10 + i))))
              for i, n in enumerate(_sizes(case["builds"], case["build_lo"], case["build_hi"]))]
    lookups = []
    for i, q in enumerate(_sizes(case["lookups"], case["q_lo"], case["q_hi"])):
        data, offsets = _pack(rows, lengths, _below(_mix_seed(seed, 30 + i), q, case["n"]))
        lookups.append((data.cpu().pin_memory(), offsets.cpu().pin_memory(),
                        torch.empty(q, dtype=torch.int64).pin_memory()))
    return {"case": case, "server": server, "resident": resident, "builds": builds, "lookups": lookups,
            "slabs": [_slab(offsets.shape[0] - 1) for _, offsets in builds]}


def _collect(srv, count):
    done = []
    while len(done) < count:
        done += rs.recsplit_server_poll(srv, 64, 1000)
    for c in done:
        if c["status"] != rs.OK:
            raise RuntimeError("request failed: %s" % rs.recsplit_strerror(c["status"]))
    return done


# ---------------------------------------------------------------- one pass
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "build":
        build = rs.Structure.build_perfect_u64 if case["key"] == "u64" else rs.Structure.build_perfect_bytes
        if not case["extra"]:
            build = rs.Structure.build_u64 if case["key"] == "u64" else rs.Structure.build_bytes
            s = build(*state["keys"], case["leaf"], case["bucket"])
        else:
            s = build(*state["keys"], case["leaf"], case["bucket"], case["extra"])
        words = s.serialize()
        s.free()
        return _store(words, state["slab"])
    if kind == "batch":
        handles = rs.recsplit_build_batch(state["sets"])
        words = [_store(rs.recsplit_serialize(h), slab) for h, slab in zip(handles, state["slabs"])]
        for h in handles:
            rs.recsplit_free(h)
        return words
    if kind == "lookup":
        look = state["s"].lookup_u64 if case["key"] == "u64" else state["s"].lookup_bytes
        return look(*state["queries"], state["out"])
    if kind == "lookup_batch":
        rs.recsplit_lookup_batch(state["owner"].handles, state["ids"], state["keys"], state["out"])
        return state["out"]
    srv = state["server"].srv
    ids = [rs.recsplit_server_submit_build_bytes(srv, data, offsets, 8, 100) for data, offsets in state["builds"]]
    for data, offsets, out in state["lookups"]:
        rs.recsplit_server_submit_lookup_bytes(srv, state["resident"], data, offsets, out)
    _collect(srv, len(ids) + len(state["lookups"]))
    words = []
    for i, slab in zip(ids, state["slabs"]):
        words.append(_store(rs.recsplit_serialize(rs.recsplit_server_structure(srv, i)), slab))
        rs.recsplit_server_release(srv, i)
    return {"structures": words, "values": [out for _, _, out in state["lookups"]]}


def exact(case, seed):
    return None  # structures and lookup values are whole numbers: they are equal or wrong


# ---------------------------------------------------------------- what a pass cannot do without
def _units(leaf):
    """Part sizes of the splitting strategy (Sec. 5.4): lower and upper aggregation."""
    s = max(2, (7 * leaf + 29) // 20)
    t = (21 * leaf + 189) // 100 if leaf >= 7 else 2
    return s * leaf, s * t * leaf


def _node_evaluations(m, leaf, extra, memo):
    """Expected evaluations below a node of m keys: per trial all keys of a split, and at a leaf the keys up to the
    first repeated value."""
    if m < 2:
        return 0.0
    if m in memo:
        return memo[m]
    if m <= leaf:
        r, p, e = m + extra, 1.0, 0.0
        for h in range(m):
            e += p
            p *= (r - h) / r
        memo[m] = e / p
        return memo[m]
    lower, upper = _units(leaf)
    if m > upper:
        unit = (m // 2 + upper - 1) // upper * upper
        parts = [unit, m - unit]
    else:
        unit = leaf if m <= lower else lower
        parts = [unit] * ((m + unit - 1) // unit - 1)
        parts.append(m - sum(parts))
    lp = math.lgamma(m + 1) - m * math.log(m)
    for k in parts:
        lp += k * math.log(k) - math.lgamma(k + 1)
    memo[m] = m * math.exp(-lp) + sum(_node_evaluations(k, leaf, extra, memo) for k in parts)
    return memo[m]


def _evaluations(n, leaf, bucket, extra):
    """Expected hash evaluations of a build: Poisson bucket sizes."""
    memo, total, spread = {}, 0.0, int(6 * math.sqrt(bucket)) + 6
    for m in range(max(0, bucket - spread), bucket + spread + 1):
        w = math.exp(m * math.log(bucket) - bucket - math.lgamma(m + 1))
        total += w * _node_evaluations(m, leaf, extra, memo)
    return total * n / bucket


# bytes of a key (a string has 20 on average, and an 8-byte offset), of a key's share of the structure (about two
# bits), of a lookup's result
def _key_bytes(key):
    return 8 if key == "u64" else 28


def work(case):
    kind = case["kind"]
    if kind == "build":
        return {"bytes": case["n"] * (_key_bytes(case["key"]) + 0.25),
                "flops": OPS * _evaluations(case["n"], case["leaf"], case["bucket"], case["extra"])}
    if kind == "batch":
        mean = (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])  # of a log-uniform size
        n = case["count"] * mean
        combos = [(leaf, b) for leaf in (5, 8, 12) for b in (5, 100, 2000)]
        return {"bytes": n * 8.25, "flops": OPS * sum(_evaluations(n / 9, leaf, b, 0) for leaf, b in combos)}
    if kind == "lookup":
        # of the structure no more than a cache line or so per query
        return {"bytes": case["q"] * (_key_bytes(case["key"]) + 8) + min(case["n"] * 0.25, case["q"] * 64.0), "flops": 0}
    if kind == "lookup_batch":
        return {"bytes": case["q"] * 20, "flops": 0}
    builds, queries = sum(_sizes(case["builds"], case["build_lo"], case["build_hi"])), sum(
        _sizes(case["lookups"], case["q_lo"], case["q_hi"]))
    return {"bytes": builds * 28.25 + queries * 36, "flops": OPS * _evaluations(builds, 8, 100, 0)}
