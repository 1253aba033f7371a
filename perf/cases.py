"""Workloads of the triangle counter, from the smallest call to the largest.

Each case is one use of the public entry points on synthetic pairs drawn on
the GPU: preprocess + count of one graph (device pairs or pinned host pairs),
counts of a graph that is kept, a batch of kept graphs, a disjoint union, a
burst of served requests, and a graph counted out of core.  Sizes are those of
bench.py's workloads and of the tests, or odd ones in between.
"""
import math

import numpy as np
import torch

from paper_1907_09575_gb300 import tc

A, AB, ABC = 0.57, 0.76, 0.95          # RMAT quadrants a, a+b, a+b+c
CHUNK = 1 << 26                        # pairs drawn at once


def listed():
    return [
        # the smallest call: a count that must not allocate, in a latency-critical loop
        {"name": "static_tiny", "kind": "static", "family": "rmat", "n": 600, "pairs": 4801, "pv": True},
        # bench.py rmat-s14: one small graph, latency and launches
        {"name": "step_rmat14", "kind": "step", "family": "rmat", "n": 1 << 14, "pairs": 1 << 18,
         "pv": False, "offsets": 32},
        # an even degree profile (no hubs, hardly a triangle), odd sizes
        {"name": "step_gnp", "kind": "step", "family": "gnp", "n": 100_003, "pairs": 1_600_021,
         "pv": True, "offsets": 0},
        # graph500 shape at an ordinary size (the tests' scale 20)
        {"name": "step_rmat20", "kind": "step", "family": "rmat", "n": 1 << 20, "pairs": 1 << 24,
         "pv": True, "offsets": 0},
        # bench.py chunglu: a social-network degree profile, totals
        {"name": "step_chunglu", "kind": "step", "family": "chunglu", "n": 50_000_000,
         "pairs": 1_000_000_000, "pv": False, "offsets": 64},
        # bench.py rmat-s26: the headline step, the largest graph
        {"name": "step_rmat26", "kind": "step", "family": "rmat", "n": 1 << 26, "pairs": 1 << 30,
         "pv": True, "offsets": 64},
        # a kept graph counted again and again (the counting kernel alone)
        {"name": "count_rmat22", "kind": "count", "family": "rmat", "n": 1 << 22, "pairs": 1 << 26,
         "pv": True, "offsets": 0},
        # bench.py batch4096 with an eighth of its graphs: many kept graphs of uneven size
        {"name": "batch_512", "kind": "batch", "graphs": 512},
        # what one serving tick is: requests of uneven size counted as one disjoint union
        {"name": "union_24", "kind": "union", "graphs": 24, "lo": 10, "hi": 20},
        # bench.py serve: requests submitted one by one to a server with three workers
        {"name": "serve_64", "kind": "serve", "graphs": 64, "lo": 10, "hi": 20},
        # host pairs to host results (bench.py e2e), an ordinary graph, pinned memory
        {"name": "triangles_rmat18", "kind": "triangles", "family": "rmat", "n": 1 << 18, "pairs": 1 << 22,
         "pv": True, "pinned": True},
        # a graph larger than its device budget (the tests' scale 20 within 1/8 of its arena)
        {"name": "tiled_rmat20", "kind": "tiled", "family": "rmat", "n": 1 << 20, "pairs": 1 << 24,
         "pv": True, "fraction": 8},
    ]


def _log(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    kind = rng.choice(["static", "step", "step", "step", "count", "batch", "union", "serve", "triangles", "tiled"])
    if kind == "batch":
        return {"kind": kind, "graphs": _log(rng, 16, 512)}
    if kind in ("union", "serve"):
        return {"kind": kind, "graphs": _log(rng, 2, 64), "lo": 10, "hi": rng.randint(14, 20)}
    top = {"static": tc.TC_STATIC_MAX_PAIRS, "step": 1 << 28, "count": 1 << 26, "triangles": 1 << 25,
           "tiled": 1 << 24}[kind]
    pairs = _log(rng, {"static": 64, "tiled": 1 << 20}.get(kind, 1 << 12), top)
    n = max(16, int(pairs / rng.uniform(8, 32)))
    case = {"kind": kind, "family": rng.choice(["rmat", "rmat", "gnp", "chunglu"]), "n": n, "pairs": pairs,
            "pv": rng.random() < 0.6}
    if kind == "static":
        case["n"] = min(case["n"], tc.TC_STATIC_MAX_VERTICES)
    elif kind == "triangles":
        case["pinned"] = rng.random() < 0.7
    elif kind == "tiled":
        case["fraction"] = rng.choice([4, 8])
    else:
        case["offsets"] = rng.choice([0, 0, 32, 64])
    return case


# --- inputs -----------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _rmat_chunk(g, scale, count, mul, xor):
    src = torch.zeros(count, dtype=torch.int32, device="cuda")
    dst = torch.zeros(count, dtype=torch.int32, device="cuda")
    u = torch.empty(count, dtype=torch.float32, device="cuda")
    for _ in range(scale):
        u.uniform_(generator=g)
        down = u >= AB                                   # quadrants c, d
        src.mul_(2).add_(down)
        dst.mul_(2).add_((u >= A) ^ down ^ (u >= ABC))   # quadrants b, d
    # seeded bijection of [0, 2^scale): hubs get ids all over the range
    mask = (1 << scale) - 1
    return [((x.to(torch.int64) * mul & mask) ^ xor).to(torch.int32) for x in (src, dst)]


def _rmat(g, n, pairs, seed):
    """RMAT pairs at the smallest scale that holds n; pairs with an id >= n are redrawn."""
    scale = max(1, (n - 1).bit_length())
    rs = np.random.RandomState(seed & 0x7FFFFFFF)
    mul, xor = int(rs.randint(0, 1 << 30)) * 2 + 1, int(rs.randint(0, 1 << scale))
    src = torch.empty(pairs, dtype=torch.int32, device="cuda")
    dst = torch.empty(pairs, dtype=torch.int32, device="cuda")
    at = 0
    while at < pairs:
        want = pairs - at
        s, d = _rmat_chunk(g, scale, min(CHUNK, want if n == 1 << scale else 2 * want + 64), mul, xor)
        if n < 1 << scale:
            keep = (s < n) & (d < n)
            s, d = s[keep], d[keep]
        k = min(want, s.numel())
        src[at:at + k], dst[at:at + k] = s[:k], d[:k]
        at += k
    return src, dst


def _chunglu(g, n, pairs, seed):
    """Power law of exponent 2.1 (weight (i+1)^(-1/1.1) up to a cap that the
    heaviest vertices share), both ends drawn by weight, ids shuffled."""
    a = 1.0 / 1.1
    h = max(1.0, n / 200_000.0)                  # the first h vertices have the capped weight
    head = h * h ** -a
    tail = (n ** (1 - a) - h ** (1 - a)) / (1 - a)
    mul = 2 * int(np.random.RandomState(seed & 0x7FFFFFFF).randint(1 << 20, 1 << 29)) + 1
    while math.gcd(mul, n) != 1:
        mul += 2
    out = []
    for _ in range(2):
        x = torch.empty(pairs, dtype=torch.int32, device="cuda")
        for at in range(0, pairs, CHUNK):
            k = min(CHUNK, pairs - at)
            u = torch.rand(k, dtype=torch.float64, device="cuda", generator=g) * (head + tail)
            v = torch.where(u < head, u * h ** a,
                            ((u - head).clamp_(min=0) * (1 - a) + h ** (1 - a)) ** (1 / (1 - a)))
            x[at:at + k] = (v.to(torch.int64).clamp_(0, n - 1) * mul % n).to(torch.int32)
        out.append(x)
    return out[0], out[1]


def _pairs(family, n, pairs, seed):
    g = _gen(seed)
    if family == "rmat":
        return _rmat(g, n, pairs, seed)
    if family == "chunglu":
        return _chunglu(g, n, pairs, seed)
    return tuple(torch.randint(0, n, (pairs,), generator=g, dtype=torch.int32, device="cuda") for _ in range(2))


def _members(case, seed):
    """(family, n, pairs, seed) of each graph of a batch, a union or a request stream."""
    rs = np.random.RandomState(seed & 0x7FFFFFFF)
    out = []
    for k in range(case["graphs"]):
        s = int(rs.randint(1, 1 << 31))
        if case["kind"] == "batch":              # n log-uniform in 2^8..2^16, mean degree 4..64
            n = int(2.0 ** rs.uniform(8, 16))
            out.append(("gnp" if k % 2 == 0 else "rmat", n, int(n * rs.uniform(4, 64) / 2), s))
        else:                                    # pairs log-uniform, edge factor 8..32
            m = int(2.0 ** rs.uniform(case["lo"], case["hi"]))
            out.append(("rmat", max(2, -(-m // int(rs.randint(8, 33)))), m, s))
    return out


def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind, "case": case}
    if kind == "serve":
        st["requests"] = [(s, max(1, (n - 1).bit_length()), n, m) for _, n, m, s in _members(case, seed)]
        st["server"] = tc.Server(hbm_budget_bytes=64 << 30, workers=3, max_batch=4096, max_tick_pairs=1 << 28)
        return st
    if kind == "batch":
        st["batch"] = tc.Batch([tc.preprocess(*_pairs(f, n, m, s), n, offsets=32)
                                for f, n, m, s in _members(case, seed)])
        return st
    if kind == "union":
        members = _members(case, seed)
        st["prefix"] = np.concatenate([[0], np.cumsum([n for _, n, _, _ in members])])
        both = [_pairs(f, n, m, s) for f, n, m, s in members]
        st["src"], st["dst"] = (torch.cat([p[e] + int(b) for p, b in zip(both, st["prefix"])]) for e in (0, 1))
        return st
    n = case["n"]
    src, dst = _pairs(case["family"], n, case["pairs"], seed)
    if kind == "triangles":
        host = [x.cpu().pin_memory() if case["pinned"] else x.cpu() for x in (src, dst)]
        out = torch.zeros(n, dtype=torch.int64)
        st["out"] = out.pin_memory() if case["pinned"] else out
        st["host"] = host
        st["src"], st["dst"] = (x.numpy() for x in host)
        return st
    if kind in ("count", "tiled"):
        st["graph"] = tc.preprocess(src, dst, n, offsets=case.get("offsets") or None)
        if kind == "tiled":
            st["budget"] = st["graph"].stats()["device_bytes"] // case["fraction"]
            st["graph"].offload()
        return st
    st["src"], st["dst"] = src, dst
    if kind == "static":
        st["out"] = torch.zeros(n, dtype=torch.int64, device="cuda")
    return st


# --- one pass ---------------------------------------------------------------

def run(st):
    kind, case = st["kind"], st["case"]
    pv = case.get("pv", False)
    if kind == "step":
        g = tc.preprocess(st["src"], st["dst"], case["n"], offsets=case["offsets"] or None)
        r = g.count(per_vertex=True if pv else None)
        g.free()
        return r
    if kind == "static":
        t = tc.triangles_static(st["src"], st["dst"], case["n"], per_vertex=st["out"] if pv else None)
        return (t, st["out"]) if pv else t
    if kind == "count":
        return st["graph"].count(per_vertex=True if pv else None)
    if kind == "batch":
        return st["batch"].count()
    if kind == "union":
        g = tc.preprocess_components(st["src"], st["dst"], st["prefix"])
        r = tc.count_components(g)
        g.free()
        return r
    if kind == "serve":
        srv = st["server"]
        tickets = [srv.submit_rmat(*q) for q in st["requests"]]
        srv.drain()
        got = {r["ticket"]: r["triangles"] for r in srv.poll()}
        return np.array([got[t] for t in tickets], dtype=np.int64)
    if kind == "triangles":
        r = tc.triangles(st["src"], st["dst"], case["n"], per_vertex=pv,
                         out=st["out"].numpy().view(np.uint64) if pv else None)
        return (r[0], r[1].view(np.int64)) if pv else r
    if kind == "tiled":
        total, t, _ = st["graph"].count_tiled(st["budget"], per_vertex=pv)
        return (total, t.view(np.int64)) if pv else total
    raise ValueError(kind)


# --- what a pass cannot do without ------------------------------------------

def work(case):
    """Each input pair (or kept edge) read once, each result written once."""
    kind = case["kind"]
    if kind in ("batch", "union", "serve"):
        members = _members(case, 1)
        pairs = sum(m for _, _, m, _ in members)
        # a batch keeps U (columns and offsets), a union has pairs, a request is a few words
        read = {"batch": 4 * pairs + 4 * sum(n for _, n, _, _ in members), "union": 8 * pairs, "serve": 64 * len(members)}
        return {"bytes": read[kind] + 8 * len(members), "flops": 0}
    per = 4 if kind in ("count", "tiled") else 8
    return {"bytes": per * case["pairs"] + (8 * case["n"] if case["pv"] else 8), "flops": 0}


# --- the same results by plain torch ----------------------------------------

def _triangles(src, dst, n, limit=4_000_000_000):
    """Triangles through each vertex (int64), or None where there are too many wedges."""
    a, b = torch.minimum(src, dst).long(), torch.maximum(src, dst).long()
    key = torch.unique((a * n + b)[a != b])
    a, b = key // n, key % n
    deg = torch.bincount(a, minlength=n) + torch.bincount(b, minlength=n)
    order = torch.sort(deg, stable=True).indices
    rank = torch.empty_like(order)
    rank[order] = torch.arange(n, device=order.device)
    a, b = rank[a], rank[b]
    key = torch.sort(torch.minimum(a, b) * n + torch.maximum(a, b)).values
    row, col = key // n, key % n
    m = key.numel()
    out = torch.zeros(n, dtype=torch.int64, device=key.device)
    if m == 0:
        return out
    end = torch.cumsum(torch.bincount(row, minlength=n), 0)[row]
    after = end - torch.arange(m, device=key.device) - 1     # wedges (row, col, k > col) of each edge
    upto = torch.cumsum(after, 0)
    if int(upto[-1]) > limit:
        return None
    at = 0
    while at < m:
        base = int(upto[at - 1]) if at else 0
        to = max(at + 1, int(torch.searchsorted(upto, base + (1 << 27), right=True)))
        e = torch.repeat_interleave(torch.arange(at, to, device=key.device), after[at:to])
        k = e + 1 + torch.arange(e.numel(), device=key.device) - (upto[e] - after[e] - base)
        want = col[e] * n + col[k]
        hit = key[torch.searchsorted(key, want).clamp_(max=m - 1)] == want
        e, k = e[hit], k[hit]
        for v in (row[e], col[e], col[k]):
            out += torch.bincount(v, minlength=n)
        at = to
    return out[rank]


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        return None                        # the requests' graphs are drawn by the server
    if kind in ("batch", "union"):
        members = _members(case, seed)
        base = np.concatenate([[0], np.cumsum([n for _, n, _, _ in members])])
        both = [_pairs(f, n, m, s) for f, n, m, s in members]
        src, dst = (torch.cat([p[e].long() + int(b) for p, b in zip(both, base)]) for e in (0, 1))
        t = _triangles(src, dst, int(base[-1]))
        if t is None:
            return None
        sums = torch.cat([torch.zeros(1, dtype=torch.int64, device=t.device), torch.cumsum(t, 0)])
        ends = sums[torch.from_numpy(base).to(t.device)]
        return (ends[1:] - ends[:-1]) // 3
    if case["pairs"] > 1 << 25:
        return None
    t = _triangles(*_pairs(case["family"], case["n"], case["pairs"], seed), case["n"])
    if t is None:
        return None
    total = int(t.sum()) // 3
    return (total, t) if case["pv"] else total
