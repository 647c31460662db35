"""What the speed of this library is measured on: the work its users have it
do, through its public entry points, from one short array to the largest
benchmark workloads.

listed() names the fixed cases and draw() gives more of the same ranges.  A
case is a dict: `op` says which entry point (keys, pairs, pairs64, segmented,
segmented_pairs, served), `dtype` the key type, `n` the number of keys (`nseg`
and `max_len` for the segmented sorts, `requests` and `max_len` for the sort
server) and `dist` the distribution of the keys.  Distributions and sizes are
those of bench.py's workloads, and ragged sizes beside them.
"""
import math

import torch

from paper_2409_03970_gb300 import nsort as ns

KEY_BYTES = {"u32": 4, "i32": 4, "f32": 4, "i64": 8, "f64": 8}
CODE = {"u32": ns.U32, "i32": ns.I32, "f32": ns.F32, "i64": ns.I64, "f64": ns.F64}
# -0, +0, +Inf, -Inf, +qNaN, -qNaN, +sNaN as int32 patterns
SPECIALS = [-0x80000000, 0, 0x7F800000, -0x800000, 0x7FC00000, -0x400000, 0x7F800001]


def listed():
    return [
        # one short array, as a program with many small arrays sorts each: launch latency
        {"name": "keys_u32_1000", "op": "keys", "dtype": "u32", "n": 1000, "dist": "uniform"},
        # the small plain workload of the benchmark (2^20 uniform keys)
        {"name": "keys_u32_2p20", "op": "keys", "dtype": "u32", "n": 1 << 20, "dist": "uniform"},
        # a ragged array of measurements: floats with the odd infinity and NaN
        {"name": "keys_f32_3m", "op": "keys", "dtype": "f32", "n": 3000017, "dist": "normal"},
        # a large array with heavy duplicates, of no round size
        {"name": "keys_i32_100m_zipf", "op": "keys", "dtype": "i32", "n": 100000007,
         "dist": "zipf"},
        # the headline workload of the benchmark
        {"name": "keys_u32_2p28", "op": "keys", "dtype": "u32", "n": 1 << 28, "dist": "uniform"},
        # 64-bit keys (ids, time stamps)
        {"name": "keys_i64_20m", "op": "keys", "dtype": "i64", "n": 20000003, "dist": "uniform"},
        # a small table sorted by a column of few values, stably
        {"name": "pairs_i32_200k", "op": "pairs", "dtype": "i32", "n": 200003, "dist": "dup16"},
        # the stable pairs workload of the benchmark
        {"name": "pairs_f32_2p27", "op": "pairs", "dtype": "f32", "n": 1 << 27, "dist": "normal"},
        # 64-bit payloads (row ids, pointers)
        {"name": "pairs64_u32_30m", "op": "pairs64", "dtype": "u32", "n": 30000000,
         "dist": "uniform"},
        # the batched workload of the benchmark: 100,000 arrays of uneven length
        {"name": "segmented_u32_100k", "op": "segmented", "dtype": "u32", "nseg": 100000,
         "max_len": 65536, "dist": "uniform"},
        # rows of a batch of tables, each sorted stably with its payloads
        {"name": "segmented_pairs_f32_5k", "op": "segmented_pairs", "dtype": "f32", "nseg": 5000,
         "max_len": 65536, "dist": "normal"},
        # a burst of mixed requests to the sort server
        {"name": "served_32", "op": "served", "dtype": "mixed", "requests": 32,
         "max_len": 1 << 22, "dist": "uniform"},
    ]


def _log_uniform(rng, lo, hi):
    return min(hi, max(lo, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    op = rng.choice(["keys", "keys", "keys64", "pairs", "pairs64", "segmented",
                     "segmented_pairs", "served"])
    if op == "keys":
        dtype = rng.choice(["u32", "i32", "f32"])
        dist = rng.choice(["uniform", "sorted", "reverse", "dup16", "zipf"] +
                          (["normal"] if dtype == "f32" else []))
        return {"op": "keys", "dtype": dtype, "n": _log_uniform(rng, 500, 1 << 28), "dist": dist}
    if op == "keys64":
        return {"op": "keys", "dtype": rng.choice(["i64", "f64"]),
                "n": _log_uniform(rng, 2000, 1 << 27),
                "dist": rng.choice(["uniform", "sorted", "dup16"])}
    if op == "pairs":
        dtype = rng.choice(["u32", "i32", "f32"])
        dist = rng.choice(["uniform", "dup16", "zipf"] + (["normal"] if dtype == "f32" else []))
        return {"op": "pairs", "dtype": dtype, "n": _log_uniform(rng, 2000, 1 << 27),
                "dist": dist}
    if op == "pairs64":
        return {"op": "pairs64", "dtype": rng.choice(["u32", "i32", "f32"]),
                "n": _log_uniform(rng, 2000, 1 << 26),
                "dist": rng.choice(["uniform", "dup16", "zipf"])}
    if op == "segmented":
        return {"op": "segmented", "dtype": rng.choice(["u32", "i32", "f32"]),
                "nseg": _log_uniform(rng, 100, 100000),
                "max_len": _log_uniform(rng, 64, 65536), "dist": "uniform"}
    if op == "segmented_pairs":
        return {"op": "segmented_pairs", "dtype": rng.choice(["u32", "i32", "f32"]),
                "nseg": _log_uniform(rng, 100, 30000),
                "max_len": _log_uniform(rng, 64, 65536), "dist": rng.choice(["uniform", "dup16"])}
    return {"op": "served", "dtype": "mixed", "requests": rng.randint(4, 40),
            "max_len": _log_uniform(rng, 1 << 14, 1 << 22), "dist": "uniform"}


# ---- inputs ------------------------------------------------------------------

def _rng(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _bits(n, wide, g):
    """n draws that cover every bit pattern, as int32 or int64."""
    if not wide:
        return torch.randint(-(1 << 31), 1 << 31, (n,), dtype=torch.int32, device="cuda",
                             generator=g)
    hi = torch.randint(-(1 << 31), 1 << 31, (n,), dtype=torch.int64, device="cuda", generator=g)
    lo = torch.randint(0, 1 << 32, (n,), dtype=torch.int64, device="cuda", generator=g)
    return (hi << 32) | lo


def _to_keys(bits, dtype):
    """Draws to keys: the integers themselves, or floats in [-1, 1)."""
    if dtype == "f32":
        return bits.to(torch.float32) * 2.0 ** -31
    if dtype == "f64":
        return bits.to(torch.float64) * 2.0 ** -63
    return bits


def _keys(n, dtype, dist, g):
    """n keys; u32 keys as int32 patterns (the entry points take the dtype code)."""
    wide = KEY_BYTES[dtype] == 8
    if dist == "normal":
        k = torch.randn(n, device="cuda", generator=g)
        sp = torch.tensor(SPECIALS, dtype=torch.int32, device="cuda").view(torch.float32)
        m = max(1, n // 1000)
        at = torch.randint(0, n, (m,), device="cuda", generator=g)
        # one special by position, so that a position drawn twice gets one value
        k[at] = sp[at % len(SPECIALS)]
        return k
    if dist in ("sorted", "reverse"):
        # ascending in the dtype's order without a sort: one draw in each of n slices
        bits = 63 if wide else 32
        step = max(1, (1 << bits) // n)
        i = torch.arange(n, dtype=torch.int64, device="cuda")
        if dist == "reverse":
            i = i.flip(0)
        v = i * step + torch.randint(0, step, (n,), dtype=torch.int64, device="cuda", generator=g)
        del i
        if wide:
            return _to_keys(v - (1 << 62), dtype)
        if dtype != "u32":
            v -= 1 << 31
        return _to_keys(v.to(torch.int32), dtype)
    if dist == "dup16":
        table = _to_keys(_bits(16, wide, g), dtype)
        return table[torch.randint(0, 16, (n,), device="cuda", generator=g)]
    if dist == "zipf":
        ranks = 1 << 20
        w = 1.0 / torch.arange(1, ranks + 1, dtype=torch.float64, device="cuda")
        cdf = torch.cumsum(w, 0)
        cdf /= cdf[-1].clone()
        table = _to_keys(_bits(ranks, wide, g), dtype)
        out = torch.empty(n, dtype=table.dtype, device="cuda")
        for lo in range(0, n, 1 << 26):
            m = min(n - lo, 1 << 26)
            u = torch.rand(m, dtype=torch.float64, device="cuda", generator=g)
            out[lo:lo + m] = table[torch.searchsorted(cdf, u).clamp_(max=ranks - 1)]
        return out
    return _to_keys(_bits(n, wide, g), dtype)


def _offsets(nseg, max_len, g):
    """int64 offsets of nseg segments of log-uniform lengths in [1, max_len]:
    the lengths are the case's, their order the generator's."""
    u = torch.rand(nseg, dtype=torch.float64, device="cuda", generator=_rng(nseg))
    lens = torch.exp2(u * math.log2(max_len)).to(torch.int64).clamp_(1, max_len)
    lens = lens[torch.randperm(nseg, device="cuda", generator=g)]
    off = torch.zeros(nseg + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=off[1:])
    return off


class Served:
    """A sort server and the requests of one burst."""

    def __init__(self, reqs):
        self.reqs = reqs
        self.server = ns.SortServer(mem_budget_bytes=1 << 30, streams=4)

    def __del__(self):
        self.server.close()


def prepare(case, seed):
    g = _rng(seed)
    op = case["op"]
    if op == "served":
        reqs = []
        # the sizes are the case's, the keys the seed's
        u = torch.rand(case["requests"], dtype=torch.float64, device="cuda",
                       generator=_rng(case["requests"])).tolist()
        for i, x in enumerate(u):
            n = int(2 ** (10 + x * (math.log2(case["max_len"]) - 10)))
            dtype, pairs = [("u32", False), ("i32", False), ("f32", False), ("f32", True)][i % 4]
            k = _keys(n, dtype, case["dist"], g)
            v = torch.arange(n, dtype=torch.int32, device="cuda") if pairs else None
            reqs.append((k, torch.empty_like(k), v, torch.empty_like(v) if pairs else None,
                         CODE[dtype]))
        return {"op": op, "served": Served(reqs)}
    s = {"op": op, "code": CODE[case["dtype"]]}
    if op in ("segmented", "segmented_pairs"):
        s["off"] = _offsets(case["nseg"], case["max_len"], g)
        n = int(s["off"][-1])
        kind = ns.KIND_SEGMENTED if op == "segmented" else ns.KIND_SEGMENTED_PAIRS
        s["tmp"] = ns.scratch(kind, n, case["nseg"], dtype=s["code"])
    else:
        n = case["n"]
        kind = {"keys": ns.KIND_KEYS, "pairs": ns.KIND_PAIRS, "pairs64": ns.KIND_PAIRS64}[op]
        s["tmp"] = ns.scratch(kind, n, dtype=s["code"])
    s["n"] = n
    s["keys"] = _keys(n, case["dtype"], case["dist"], g)
    s["keys_out"] = torch.empty_like(s["keys"])
    s["vals"] = s["vals_out"] = None
    if op in ("pairs", "segmented_pairs"):
        s["vals"] = torch.arange(n, dtype=torch.int32, device="cuda")
    elif op == "pairs64":
        s["vals"] = torch.arange(n, dtype=torch.int64, device="cuda") * 0x10000001
    if s["vals"] is not None:
        s["vals_out"] = torch.empty_like(s["vals"])
    return s


# ---- one pass ----------------------------------------------------------------

def run(s):
    op = s["op"]
    if op == "served":
        served = s["served"]
        tickets = [ns.nsort_submit(served.server.ctx, ns.KIND_KEYS if v is None else ns.KIND_PAIRS,
                                   code, k.numel(), k, ko, v, vo)
                   for k, ko, v, vo, code in served.reqs]
        for t in tickets:
            rc = served.server.wait(t)
            if rc != ns.OK:
                raise ns.NsortError(rc, "nsort_wait")
        return [[ko] if vo is None else [ko, vo] for _, ko, _, vo, _ in served.reqs]
    k, ko, v, vo, n, tmp = (s["keys"], s["keys_out"], s["vals"], s["vals_out"], s["n"], s["tmp"])
    if op == "keys":
        rc = ns.nsort_keys(k, ko, n, s["code"], tmp, tmp.numel())
    elif op == "pairs":
        rc = ns.nsort_pairs(k, v, ko, vo, n, s["code"], tmp, tmp.numel())
    elif op == "pairs64":
        rc = ns.nsort_pairs64(k, v, ko, vo, n, s["code"], tmp, tmp.numel())
    else:
        rc = ns.nsort_segmented(k, ko, v, vo, s["off"], s["off"].numel() - 1, n, s["code"], tmp,
                                tmp.numel())
    if rc != ns.OK:
        raise ns.NsortError(rc, op)
    return [ko] if vo is None else [ko, vo]


def work(case):
    """Each key and payload read once and written once; a sort does no
    floating-point work."""
    op = case["op"]
    if op == "served":
        # log-uniform lengths in [2^10, max_len]; a quarter of the requests are pairs
        a, b = 1024.0, float(case["max_len"])
        return {"bytes": case["requests"] * (b - a) / math.log(b / a) * 8 * 1.25, "flops": 0}
    if op in ("segmented", "segmented_pairs"):
        # floor of log-uniform lengths in [1, max_len]
        b = float(case["max_len"])
        n = case["nseg"] * ((b - 1) / math.log(b) - 0.5 if b > 2 else 1.0)
        return {"bytes": n * (8 if op == "segmented" else 16) + 8 * case["nseg"], "flops": 0}
    payload = {"keys": 0, "pairs": 4, "pairs64": 8}[op]
    return {"bytes": 2 * case["n"] * (KEY_BYTES[case["dtype"]] + payload), "flops": 0}


# ---- the exact results -------------------------------------------------------

def _order(keys, code):
    """Signed integers in the key order: the integers themselves (u32 patterns
    offset), or the IEEE total order of floats."""
    if code == ns.U32:
        return keys ^ -0x80000000
    if code == ns.F32:
        b = keys.view(torch.int32)
        return b ^ ((b >> 31) & 0x7FFFFFFF)
    if code == ns.F64:
        b = keys.view(torch.int64)
        return b ^ ((b >> 63) & 0x7FFFFFFFFFFFFFFF)
    return keys


def _wide(x):
    return x.to(torch.float64) if x.is_floating_point() else x


def _exact_sort(k, v, code, off=None):
    idx = torch.sort(_order(k, code), stable=True)[1]
    if off is not None:   # segments in order, each one's keys in order
        seg = torch.searchsorted(off, idx, right=True)
        idx = idx[torch.sort(seg, stable=True)[1]]
    return [_wide(k[idx])] if v is None else [_wide(k[idx]), v[idx]]


def exact(case, seed):
    s = prepare(case, seed)
    if case["op"] == "served":
        return [_exact_sort(k, v, code) for k, _, v, _, code in s["served"].reqs]
    return _exact_sort(s["keys"], s["vals"], s["code"], s.get("off"))
