"""Performance cases of the join library: what is timed, on which inputs.

Every case is one call a user's program makes through
``paper_1904_11201_gb300.jn`` with the default tuning.  The order of a join's
pairs is unspecified, so a case that emits pairs puts them where its program
needs them: into a column of the table whose rows match at most once (the
lookup of a dimension row for every fact row, of the time window an event
falls into), -1 where nothing matches.  That column holds every pair and does
not depend on their order.  Cases whose result is not stored return the count
and the checksum of jn_aggregate.

Sizes are those of the benchmark (16K x 64K, 1M x 16M, 64K x 1M, a 64M-row
fact table with two 1M-row dimensions, 256M x 256M, Zipf keys over 2^28
ranks, batches of 1000-row to 4M-row joins) or ordinary odd ones between.
"""
import math
import random

import numpy as np
import torch

from paper_1904_11201_gb300 import datagen as dg
from paper_1904_11201_gb300 import jn

DEV = "cuda"


def listed():
    return [
        # the smallest call: a request's few thousand rows, bound by launches and latency
        {"name": "hash_16k_64k", "op": "hash", "r": 16384, "s": 65536, "i64": False, "pay": True, "match": 0.25},
        # an ordinary lookup: an odd-sized 1M-row dimension, every fact row matches, row indices as payload
        {"name": "hash_1m_4m", "op": "hash", "r": 1000003, "s": 4100011, "i64": False, "pay": False, "match": 1.0},
        # a large equi-join of two tables of the same size, half of the probing rows match
        {"name": "hash_64m_64m", "op": "hash", "r": 1 << 26, "s": 1 << 26, "i64": False, "pay": True, "match": 0.5},
        # 64-bit keys, and the fact table (many rows per key) given as the build side
        {"name": "hash_i64_24m_3m", "op": "hash_fact_r", "r": 24000011, "s": 3000017, "i64": True, "pay": True,
         "match": 0.7},
        # the benchmark's headline inputs (uniform keys, 2^28 rows a side), result counted and checksummed
        {"name": "aggregate_256m_256m", "op": "aggregate", "r": 1 << 28, "s": 1 << 28, "i64": False, "theta": 0.0},
        # skewed keys: Zipf(1) over 2^28 ranks, far more pairs than can be stored
        {"name": "aggregate_zipf_32m_64m", "op": "aggregate", "r": 1 << 25, "s": 1 << 26, "i64": False, "theta": 1.0},
        # the sort-merge join, odd sizes
        {"name": "sort_merge_16m_40m", "op": "sort", "r": 16000057, "s": 40000003, "i64": False, "pay": True,
         "match": 0.6},
        # a star schema: a 64M-row fact table against two 1M-row dimensions
        {"name": "star_64m_1m_1m", "op": "star", "r": 1 << 26, "s1": 1 << 20, "s2": 1 << 20, "i64": False,
         "match": 1.0},
        # a band join that finds the window of each event (with a second, ordered condition), pairs written
        {"name": "band_1m_16m", "op": "band", "r": 1 << 20, "s": 1 << 24, "i64": False, "gap": 16, "w": 7},
        # the benchmark's wide band (95 either side, about 1e8 pairs), counted and checksummed
        {"name": "band_aggregate_1m_16m", "op": "band_aggregate", "r": 1 << 20, "s": 1 << 24, "i64": False, "w": 95},
        # the nested loop, for predicates no index serves: every pair is compared on two columns
        {"name": "nested_64k_1m", "op": "nested", "r": 1 << 16, "s": 1 << 20, "i64": False, "gap": 256, "w": 127},
        # many small joins at once (what a server's coalesced requests become), half of them band joins
        {"name": "batch_256", "op": "batch", "joins": 256, "lo": 1000, "hi": 4000000, "i64": False, "mix": 1},
    ]


def _log(rng, lo, hi):
    """An integer log-uniform in [lo, hi], odd three times in four."""
    v = int(math.exp(rng.uniform(math.log(lo), math.log(hi))))
    return max(lo, min(hi, v | 1 if rng.random() < 0.75 else v))


def draw(rng):
    op = rng.choice(["hash", "hash", "hash_fact_r", "aggregate", "sort", "star", "band", "band_aggregate", "nested",
                     "batch"])
    i64 = rng.random() < 0.35
    match = rng.choice([0.1, 0.5, 0.8, 1.0])
    if op in ("hash", "sort"):
        return {"op": op, "r": _log(rng, 1000, 1 << 26), "s": _log(rng, 1000, 1 << 26), "i64": i64,
                "pay": rng.random() < 0.6, "match": match}
    if op == "hash_fact_r":
        return {"op": op, "r": _log(rng, 4000, 1 << 26), "s": _log(rng, 1000, 1 << 23), "i64": i64,
                "pay": rng.random() < 0.6, "match": match}
    if op == "aggregate":
        return {"op": op, "r": _log(rng, 1000, 1 << 27), "s": _log(rng, 1000, 1 << 27), "i64": i64,
                "theta": rng.choice([0.0, 0.0, 0.5, 1.0])}
    if op == "star":
        return {"op": op, "r": _log(rng, 10000, 1 << 26), "s1": _log(rng, 1000, 1 << 22),
                "s2": _log(rng, 1000, 1 << 22), "i64": i64, "match": match}
    if op == "band":
        gap = rng.randint(1, 64)
        return {"op": op, "r": _log(rng, 1000, 1 << 21), "s": _log(rng, 1000, 1 << 25), "i64": i64, "gap": gap,
                "w": rng.randint(0, (gap - 1) // 2)}
    if op == "band_aggregate":
        return {"op": op, "r": _log(rng, 1000, 1 << 20), "s": _log(rng, 1000, 1 << 24), "i64": i64,
                "w": rng.randint(0, 100)}
    if op == "nested":
        gap = rng.randint(1, 512)
        # 64-bit comparisons take about twice as long: half the rows
        return {"op": op, "r": _log(rng, 1000, 1 << 16), "s": _log(rng, 1000, 1 << (19 if i64 else 20)), "i64": i64,
                "gap": gap, "w": rng.randint(0, (gap - 1) // 2)}
    return {"op": op, "joins": _log(rng, 2, 256), "lo": 1000, "hi": _log(rng, 4000, 4000000), "i64": i64,
            "mix": rng.randint(0, 1)}


# ------------------------------------------------------------------- inputs --
def _bits(n):
    return max(1, int(n - 1).bit_length())


def _scramble(x, bits, seed):
    """A bijection of [0, 2^bits), chosen by the seed, applied to int64 values."""
    rng = random.Random(seed)
    mask = (1 << bits) - 1
    for _ in range(3):
        x = (x * (rng.getrandbits(62) | 1) + rng.getrandbits(62)) & mask
        x = x ^ (x >> max(1, (bits + 1) // 2))
    return x


def _key(rank, bits, seed, i64):
    """Distinct keys for distinct ranks of [0, 2^bits), positive and negative."""
    if i64:
        return dg.rank_to_key64(rank, seed)
    return (_scramble(rank, bits, seed) - (1 << (bits - 1))).to(torch.int32)


def _ranks(n, domain, seed, stream):
    return dg.uniform_int(n, 0, domain, seed, stream, DEV, torch.int64)


def _lookup(n_dim, n_fact, match, i64, seed, stream=0):
    """Keys of a dimension table without duplicates, keys of a fact table of
    which a share `match` is among them, and the facts' ranks (the dimension
    row of a rank below n_dim)."""
    domain = max(n_dim, int(n_dim / match))
    bits = _bits(domain)
    dim = _key(torch.arange(n_dim, dtype=torch.int64, device=DEV), bits, seed + stream, i64)
    rank = _ranks(n_fact, domain, seed, 10 + stream)
    return dim, _key(rank, bits, seed + stream, i64), rank


def _windows(n_r, n_s, gap, i64, seed, stream=0):
    """Columns (a, k) of windows centred `gap` apart and of events anywhere."""
    bits = _bits(n_r)
    dt = torch.int64 if i64 else torch.int32
    ids = _scramble(torch.arange(n_r, dtype=torch.int64, device=DEV), bits, seed + stream)
    rk = (ids * gap + gap // 2).to(dt)
    sk = dg.uniform_int(n_s, 0, gap << bits, seed, 20 + stream, DEV, dt)
    ra = dg.uniform_int(n_r, 0, 1 << 24, seed, 21 + stream, DEV, dt)
    sa = dg.uniform_int(n_s, 0, 1 << 24, seed, 22 + stream, DEV, dt)
    return ra, rk, sa, sk


def _pay(case, n):
    return dg.row_ids(n, DEV) if case["pay"] else None


def _equi(case, seed):
    """(R key, S key, the fact rows' ranks) of a lookup; the facts are S, or R."""
    if case["op"] == "hash_fact_r":
        dim, fact, rank = _lookup(case["s"], case["r"], case["match"], case["i64"], seed)
        return fact, dim, rank
    dim, fact, rank = _lookup(case["r"], case["s"], case["match"], case["i64"], seed)
    return dim, fact, rank


def _zipf_ranks(n, theta, bits, seed, stream):
    """Ranks of [0, 2^bits) with probability about proportional to (rank + 1)^-theta,
    by the inverse of the continuous distribution on [1, 2^bits + 1)."""
    u, top = dg.uniform_float(n, seed, stream, DEV), float((1 << bits) + 1)
    if theta == 1.0:
        x = torch.exp(u * math.log(top))
    else:
        x = (u * (top ** (1.0 - theta) - 1.0) + 1.0).pow(1.0 / (1.0 - theta))
    return (x.to(torch.int64) - 1).clamp_(0, (1 << bits) - 1)


def _batch_sizes(case):
    rng = random.Random("%d %d %d" % (case["joins"], case["lo"], case["hi"]))
    return [(_log(rng, case["lo"], case["hi"]), _log(rng, case["lo"], case["hi"])) for _ in range(case["joins"])]


def prepare(case, seed):
    op = case["op"]
    st = {"op": op, "ctx": jn.Context(0)}
    if op in ("hash", "hash_fact_r", "sort"):
        rk, sk, _ = _equi(case, seed)
        st["R"] = jn.table(rk, payload=_pay(case, case["r"]))
        st["S"] = jn.table(sk, payload=_pay(case, case["s"]))
        st["rows"] = case["r"] if op == "hash_fact_r" else case["s"]
    elif op == "star":
        k1, f1, _ = _lookup(case["s1"], case["r"], case["match"], case["i64"], seed)
        k2, f2, _ = _lookup(case["s2"], case["r"], case["match"], case["i64"], seed, 1)
        st["R"] = jn.table(f1, f2, dg.row_ids(case["r"], DEV))
        st["S1"], st["S2"] = jn.table(k1), jn.table(k2)
        st["rows"] = case["r"]
    elif op == "aggregate":
        if case["theta"] > 0:
            rk = _key(_zipf_ranks(case["r"], case["theta"], 28, seed, 1), 28, seed, case["i64"])
            sk = _key(_zipf_ranks(case["s"], case["theta"], 28, seed, 2), 28, seed, case["i64"])
        else:
            domain = max(case["r"], case["s"])
            rk = _key(_ranks(case["r"], domain, seed, 1), _bits(domain), seed, case["i64"])
            sk = _key(_ranks(case["s"], domain, seed, 2), _bits(domain), seed, case["i64"])
        st["R"] = jn.table(rk, payload=dg.row_ids(case["r"], DEV))
        st["S"] = jn.table(sk, payload=dg.row_ids(case["s"], DEV))
    elif op in ("band", "nested"):
        ra, rk, sa, sk = _windows(case["r"], case["s"], case["gap"], case["i64"], seed)
        st["R"] = jn.table(ra, rk, dg.row_ids(case["r"], DEV))
        st["S"] = jn.table(sa, sk, dg.row_ids(case["s"], DEV))
        st["w"], st["rows"] = case["w"], case["s"]
    elif op == "band_aggregate":
        dt = torch.int64 if case["i64"] else torch.int32
        ra, rk = dg.band_columns(case["r"], 24, seed, 0, DEV)
        sa, sk = dg.band_columns(case["s"], 24, seed, 1, DEV)
        st["R"] = jn.table(ra.to(dt), rk.to(dt), dg.row_ids(case["r"], DEV))
        st["S"] = jn.table(sa.to(dt), sk.to(dt), dg.row_ids(case["s"], DEV))
        st["w"] = case["w"]
    else:
        joins, base = [], 0
        for i, (nr, ns) in enumerate(_batch_sizes(case)):
            # the S payload is the row's place in the batch's one result column
            spay = torch.arange(base, base + ns, dtype=torch.int32, device=DEV)
            base += ns
            if case["mix"] and i % 2:
                ra, rk, sa, sk = _windows(nr, ns, 16, case["i64"], seed, 50 + 50 * i)
                joins.append((jn.table(ra, rk), jn.table(sa, sk, spay), jn.JN_LT, 7))
            else:
                rk, sk, _ = _lookup(nr, ns, 0.5, case["i64"], seed, 50 + 50 * i)
                joins.append((jn.table(rk), jn.table(sk, payload=spay), jn.JN_EQ, -1))
        st["joins"], st["rows"] = joins, base
    torch.cuda.synchronize()
    return st


# ---------------------------------------------------------------------- run --
def _column(pairs, rows, by, value):
    """The matching row of every row of one side, -1 where there is none."""
    col = torch.full((rows,), -1, dtype=torch.int32, device=DEV)
    col[pairs[:, by]] = pairs[:, value]
    return col


def run(st):
    op, ctx = st["op"], st["ctx"]
    if op == "hash":
        return _column(jn.jn_hash(ctx, st["R"], st["S"]), st["rows"], 1, 0)
    if op == "hash_fact_r":
        return _column(jn.jn_hash(ctx, st["R"], st["S"]), st["rows"], 0, 1)
    if op == "sort":
        return _column(jn.jn_sort_merge(ctx, st["R"], st["S"]), st["rows"], 1, 0)
    if op == "star":
        t = jn.jn_star(ctx, st["R"], st["S1"], st["S2"])
        cols = torch.full((st["rows"], 2), -1, dtype=torch.int32, device=DEV)
        cols[t[:, 0]] = t[:, 1:]
        return cols
    if op == "band":
        return _column(jn.jn_theta(ctx, st["R"], st["S"], jn.JN_LT, st["w"]), st["rows"], 1, 0)
    if op == "nested":
        pairs = jn.jn_nested_loop(ctx, st["R"], st["S"], jn.pred(jn.JN_LT, jn.JN_ANY, st["w"]))
        return _column(pairs, st["rows"], 1, 0)
    if op == "batch":
        pairs, first, count = jn.jn_batch(ctx, st["joins"])
        return [_column(pairs, st["rows"], 1, 0), np.array(first), np.array(count)]
    if op == "aggregate":
        count, chk = jn.jn_aggregate(ctx, jn.JN_ALGO_HASH, st["R"], st["S"])
    else:
        count, chk = jn.jn_aggregate(ctx, jn.JN_ALGO_THETA, st["R"], st["S"], jn.pred(jn.JN_LT, jn.JN_ANY, st["w"]))
    return [count, chk - (1 << 64) if chk >> 63 else chk]  # the checksum as a signed word


def exact(case, seed):
    """The lookups' column, from the ranks the keys were made of (no join)."""
    op = case["op"]
    if op in ("hash", "hash_fact_r", "sort"):
        n_dim = case["s"] if op == "hash_fact_r" else case["r"]
        _, _, rank = _equi(case, seed)
        return torch.where(rank < n_dim, rank, -1).to(torch.int32)
    if op == "star":
        _, _, r1 = _lookup(case["s1"], case["r"], case["match"], case["i64"], seed)
        _, _, r2 = _lookup(case["s2"], case["r"], case["match"], case["i64"], seed, 1)
        both = (r1 < case["s1"]) & (r2 < case["s2"])
        return torch.stack([torch.where(both, r1, -1), torch.where(both, r2, -1)], 1).to(torch.int32)
    return None


def work(case):
    """Bytes: every input column read once, the pairs and the column they go
    to written once.  Operations: the nested loop compares every pair of rows
    (a subtraction and a comparison for each of its two columns)."""
    op, kb = case["op"], 8 if case["i64"] else 4
    if op in ("hash", "hash_fact_r", "sort"):
        fact = case["r"] if op == "hash_fact_r" else case["s"]
        row = kb + (4 if case["pay"] else 0)
        return {"bytes": row * (case["r"] + case["s"]) + 8 * int(case["match"] * fact) + 4 * fact, "flops": 0}
    if op == "star":
        m = int(case["match"] ** 2 * case["r"])
        return {"bytes": (2 * kb + 4) * case["r"] + kb * (case["s1"] + case["s2"]) + 12 * m + 8 * case["r"], "flops": 0}
    if op == "aggregate":
        return {"bytes": (kb + 4) * (case["r"] + case["s"]), "flops": 0}
    if op == "band_aggregate":
        return {"bytes": (2 * kb + 4) * (case["r"] + case["s"]), "flops": 0}
    if op in ("band", "nested"):
        rows = case["r"] + case["s"]
        share = (2 * case["w"] + 1) / case["gap"] * case["r"] / (1 << _bits(case["r"])) / 2
        flops = 4 * case["r"] * case["s"] if op == "nested" else 0
        return {"bytes": (2 * kb + 4) * rows + 8 * int(share * case["s"]) + 4 * case["s"], "flops": flops}
    total = 0
    for i, (nr, ns) in enumerate(_batch_sizes(case)):
        band = case["mix"] and i % 2  # two compared columns; about 0.47 of the events lie in a window and pass
        m = 0.47 * nr / (1 << _bits(nr)) if band else 0.5
        total += (2 if band else 1) * kb * (nr + ns) + 4 * ns + int(8 * m * ns) + 4 * ns
    return {"bytes": total, "flops": 0}
