"""Cases that time the library through its public entry points.

Every case is one piece of work as a program that uses the library gives it:
the exact distance of a string to one or a few versions of it, the distances
of a batch and of a burst of served requests, an optimal edit script, and a
prefix-hash table.  The listed sizes
are those of the single-pair, batch, serve and tuning workloads and of the
tests; ``draw`` gives more cases of the same ranges.

Inputs are drawn on the GPU from a seed alone: strings of the workloads'
alphabets (uniform, Zipf over 256 bytes, or two skewed symbols) with planted
insertions, deletions and substitutions, uniform or in bursts.
"""
from __future__ import annotations

import math
import time

import numpy as np
import torch

from paper_2306_17461_gb300 import binding as ed

Q61 = (1 << 61) - 1
CHUNK = 1 << 26
HASH_SEED = 20230617


# ---------------------------------------------------------------- the cases
def _pair(name, n, k, **kw):
    c = {"name": name, "kind": "pair", "n": n, "k": k, "sigma": 4, "p0": 0.0, "zipf": False, "bursts": False,
         "lcp": ed.ED_LCP_AUTO, "tune": True, "hint": True, "host": False, "off": 0, "versions": 3 if k < 10_000 else 1}
    c.update(kw)
    return c


def listed():
    return [
        # short strings in host memory, no tuning: calls that are all latency
        _pair("pair_1k_host", 1_000, 20, tune=False, hint=False, host=True),
        # the small single pair: about 100 edits in a million characters
        _pair("pair_1m", 1_000_000, 100),
        # the same search answered from prefix-hash tables, tables built by the call
        _pair("pair_10m_hash", 10_000_000, 1_000, lcp=ed.ED_LCP_HASH),
        # the mid-size pair: near-identical, ordinary and far apart strings
        _pair("pair_100m_k10", 100_000_000, 10),
        _pair("pair_100m_k1000", 100_000_000, 1_000),
        _pair("pair_100m_k100000", 100_000_000, 100_000),
        # the large pair: natural-language-like symbols, edits in bursts
        _pair("pair_1g_bursts", 1_000_000_000, 10_000, zipf=True, bursts=True),
        # the batch workload: thousands of uneven device pairs in one call
        {"name": "batch_4096", "kind": "batch", "pairs": 4096, "n_lo": 1e3, "n_hi": 1e6, "r_lo": 1e-4,
         "r_hi": 5e-2, "shapes": 4, "host": False},
        # many short host strings in one call (reads, records)
        {"name": "batch_short_host", "kind": "batch", "pairs": 1024, "n_lo": 1e2, "n_hi": 1e4, "r_lo": 1e-3,
         "r_hi": 5e-2, "shapes": 9, "host": True},
        # a burst of mixed requests submitted to the serving engine, each polled
        # until it is done
        {"name": "serve_64", "kind": "serve", "pairs": 64, "n_lo": 1e2, "n_hi": 1e6, "r_lo": 1e-3, "r_hi": 1e-1,
         "shapes": 5},
        # the prefix-hash table of a long string (hash LCP, or a caller's own use)
        {"name": "hash_table_100m", "kind": "hash", "n": 100_000_000, "block": 1, "off": 0},
        # an optimal edit script: the frontiers of every round and the walk back
        {"name": "script_1m", "kind": "script", "n": 1_000_000, "k": 500, "sigma": 4, "t_max": 1024, "off": 0},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    u = rng.random()
    off = rng.choice([0, 0, 1, 3, 7, 8, 13])
    if u < 0.5:
        n = int(_log_uniform(rng, 1e3, 3e8)) | 1
        k = max(8, int(min(_log_uniform(rng, 1e-7, 3e-2) * n, 3e4)))
        text = rng.choice(["dna", "dna", "bytes", "zipf", "binary"])
        c = _pair("", n, k, off=off, tune=rng.random() < 0.7, host=n < 10_000_000 and rng.random() < 0.3,
                  bursts=k > 50 and rng.random() < 0.3)
        c["hint"] = c["tune"] and rng.random() < 0.7
        if text == "bytes":
            c["sigma"] = 64
        elif text == "zipf":
            c["zipf"] = True
        elif text == "binary" and k <= 10_000:
            c["p0"] = rng.choice([0.5, 0.9])
        if n <= 10_000_000 and k <= 1_000 and c["p0"] == 0.0 and rng.random() < 0.2:
            c["lcp"] = rng.choice([ed.ED_LCP_HASH, ed.ED_LCP_BHASH])
    elif u < 0.7:
        host = rng.random() < 0.4
        c = {"kind": "batch", "pairs": int(_log_uniform(rng, 16, 2048)), "n_lo": 1e2 if host else 1e3,
             "n_hi": 1e4 if host else _log_uniform(rng, 1e4, 1e6), "r_lo": 1e-4, "r_hi": 5e-2,
             "shapes": rng.randrange(10, 1 << 30), "host": host}
    elif u < 0.8:
        c = {"kind": "serve", "pairs": int(_log_uniform(rng, 8, 64)), "n_lo": 1e2,
             "n_hi": _log_uniform(rng, 1e4, 5e5), "r_lo": 1e-3, "r_hi": 1e-1,
             "shapes": rng.randrange(10, 1 << 30)}
    elif u < 0.9:
        c = {"kind": "hash", "n": int(_log_uniform(rng, 1e3, 1e8)) | 1, "block": rng.choice([1, 1, 4, 32]),
             "off": off}
    else:
        n = int(_log_uniform(rng, 1e3, 1e7)) | 1
        k = max(1, int(min(_log_uniform(rng, 1e-5, 3e-2) * n, 900)))
        c = {"kind": "script", "n": n, "k": k, "sigma": rng.choice([4, 64]), "t_max": 1024, "off": off}
    c.pop("name", None)
    return c


# ---------------------------------------------------------------- inputs
def _gen(seed, device="cuda"):
    g = torch.Generator(device=device)
    g.manual_seed(seed)
    return g


def _lut(p):
    """65536 entries in which symbol i takes a share of about p[i]."""
    cdf = np.cumsum(p / p.sum())
    u = (np.arange(65536) + 0.5) / 65536.0
    return torch.from_numpy(np.minimum(np.searchsorted(cdf, u, side="right"), p.size - 1).astype(np.uint8)).cuda()


def _text(g, n, sigma=4, zipf=False, p0=0.0):
    if not zipf and not p0:
        return torch.randint(0, sigma, (n,), dtype=torch.uint8, device="cuda", generator=g)
    lut = _lut(np.arange(1, 257, dtype=np.float64) ** -1.1) if zipf else _lut(np.array([p0, 1.0 - p0]))
    out = torch.empty(n, dtype=torch.uint8, device="cuda")
    for lo in range(0, n, CHUNK):
        hi = min(n, lo + CHUNK)
        out[lo:hi] = lut[torch.randint(0, 65536, (hi - lo,), device="cuda", generator=g)]
    return out


def _plant(g, A, pos, sigma):
    """B = A with one edit (substitute, delete, insert: equally likely) at
    each of the sorted distinct positions pos; sigma is the alphabet size, one
    for all or one per edit.  Also returns the shift of the positions before
    each edit and after the last."""
    n, k = A.numel(), pos.numel()
    if k == 0:
        return A.clone(), torch.zeros(1, dtype=torch.int64, device="cuda")
    op = torch.randint(0, 3, (k,), device="cuda", generator=g)
    shift = torch.zeros(k + 1, dtype=torch.int64, device="cuda")
    shift[1:] = torch.cumsum((op == 2).long() - (op == 1).long(), 0)
    at = pos + shift[:-1]  # where each edit's output begins in B
    m = n + int(shift[-1])
    B = torch.empty(m, dtype=torch.uint8, device="cuda")
    for lo in range(0, m, CHUNK):
        j = torch.arange(lo, min(m, lo + CHUNK), device="cuda")
        src = j - shift[torch.searchsorted(at, j, right=True)]
        B[lo:lo + j.numel()] = A[src.clamp_(0, n - 1)]
    # a symbol of the text's own distribution, another one where it must differ
    sym = A[(pos + torch.randint(-64, 65, (k,), device="cuda", generator=g)).clamp_(0, n - 1)].long()
    old = A[pos].long()
    sym = torch.where((op == 0) & (sym == old), (old + 1) % sigma, sym)
    put = op != 1
    B[at[put]] = sym[put].to(torch.uint8)
    return B, shift


def _positions(g, n, k, bursts, seed):
    if not bursts:
        return torch.unique(torch.randint(0, n, (k,), device="cuda", generator=g))
    # bursts of mean 20 edits, mean gap 4, at uniform places
    r = np.random.default_rng(seed)
    size = r.geometric(1 / 20.0, size=k)
    size = size[: int(np.searchsorted(np.cumsum(size), k)) + 1]
    start = np.repeat(r.integers(0, n, size.size), size)
    gap = r.geometric(1 / 4.0, size=start.size)
    c = np.cumsum(gap)
    first = np.repeat(c[np.cumsum(size) - size], size)
    pos = np.unique(start + c - first)[:k]
    return torch.from_numpy(pos[pos < n]).cuda()


def _at_offset(t, off):
    """t at `off` bytes past an allocation's (aligned) start."""
    buf = torch.empty(t.numel() + off, dtype=torch.uint8, device="cuda")
    buf[off:] = t
    return buf[off:]


def _one_pair(case, seed):
    g = _gen(seed)
    A = _text(g, case["n"], case["sigma"])
    B, _ = _plant(g, A, _positions(g, case["n"], case["k"], False, seed), case["sigma"])
    return (A, _at_offset(B, case["off"])) if case["off"] else (A, B)


def _versions(case, seed):
    """A string and its versions, each with its own count of planted edits
    (k, give or take 7)."""
    g = _gen(seed)
    A = _text(g, case["n"], case["sigma"], case["zipf"], case["p0"])
    sigma = 256 if case["zipf"] else (2 if case["p0"] else case["sigma"])
    r = np.random.default_rng(seed)
    Bs = []
    for v in range(case["versions"]):
        k = case["k"] + int(r.integers(-7, 8))
        B, _ = _plant(g, A, _positions(g, case["n"], k, case["bursts"], (seed, v)), sigma)
        Bs.append(_at_offset(B, case["off"]) if case["off"] else B)
    return A, Bs


def _shapes(case):
    r = np.random.default_rng(case["shapes"])
    n = np.exp(r.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]), case["pairs"])).round().astype(np.int64)
    k = (n * np.exp(r.uniform(math.log(case["r_lo"]), math.log(case["r_hi"]), case["pairs"]))).round()
    return np.maximum(n, 1), k.astype(np.int64)


def _pairs(case, seed):
    """The set's pairs, packed one after another in two buffers; alphabets of
    4 and 64 symbols in turn (serving: 4)."""
    n, k = _shapes(case)
    sig = np.where(np.arange(n.size) % 2 == 0, 4, 4 if case["kind"] == "serve" else 64)
    g = _gen(seed)
    nt, kt, st = (torch.from_numpy(v).cuda() for v in (n, k, sig))
    total = int(n.sum())
    A = _text(g, total, 64)
    A &= torch.repeat_interleave((st - 1).to(torch.uint8), nt, output_size=total)
    a0 = torch.cumsum(nt, 0) - nt
    u = torch.rand(int(k.sum()), dtype=torch.float64, device="cuda", generator=g)
    nr = torch.repeat_interleave(nt, kt)
    pos = torch.unique(torch.repeat_interleave(a0, kt) + torch.minimum((u * nr).long(), nr - 1))
    whose = torch.searchsorted(a0, pos, right=True) - 1
    B, shift = _plant(g, A, pos, st[whose])
    ends = torch.cat([a0, torch.tensor([total], device="cuda")])
    b0 = (ends + shift[torch.searchsorted(pos, ends)]).tolist()
    a0 = ends.tolist()
    return ([A[a0[i]:a0[i + 1]] for i in range(n.size)], [B[b0[i]:b0[i + 1]] for i in range(n.size)])


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "case": dict(case)}
    if kind in ("pair", "script", "hash"):
        if kind == "hash":
            X = _text(_gen(seed), case["n"], 64)
            s["X"] = _at_offset(X, case["off"]) if case["off"] else X
        elif kind == "script":
            s["A"], s["B"] = _one_pair(case, seed)
        else:
            s["A"], s["B"] = _versions(case, seed)
            if case["host"]:
                s["A"], s["B"] = s["A"].cpu().numpy(), [B.cpu().numpy() for B in s["B"]]
        cfg = {"hash_seed": HASH_SEED}
        if kind == "pair":
            cfg["lcp_mode"] = case["lcp"]
            if case["tune"]:
                cfg["tune"] = 1
            if case["hint"]:
                cfg["distance_hint"] = case["k"]
        s["ctx"] = ed.Context(**cfg)
        return s
    s["A"], s["B"] = _pairs(case, seed)
    if kind == "serve" or case["host"]:
        s["A"] = [t.cpu().numpy() for t in s["A"]]
        s["B"] = [t.cpu().numpy() for t in s["B"]]
    s["ctx"] = ed.Context(mem_budget_bytes=16 << 30)
    return s


# ---------------------------------------------------------------- one pass
def run(state):
    kind, ctx, case = state["kind"], state["ctx"], state["case"]
    if kind == "pair":
        f = ctx.distance if case["host"] else ctx.distance_dev
        return {"distances": [f(state["A"], B) for B in state["B"]]}
    if kind == "batch":
        f = ed.ed_distance_batch if case["host"] else ed.ed_distance_batch_dev
        return {"distances": f(ctx.h, state["A"], state["B"])}
    if kind == "serve":
        return {"distances": _serve(ctx, state["A"], state["B"])}
    if kind == "hash":
        if case["block"] == 1:
            return {"table": ed.ed_prefix_hash_dev(ctx.h, state["X"])}
        return {"table": ed.ed_prefix_hash_blocked_dev(ctx.h, state["X"], case["block"])}
    k, ops = ed.ed_edit_script_dev(ctx.h, state["A"], state["B"], case["t_max"])
    return {"distance": k, "ops": ops}


def _serve(ctx, As, Bs):
    tickets = []
    for a, b in zip(As, Bs):
        while True:
            try:
                tickets.append(ed.ed_submit(ctx.h, a, b))
                break
            except ed.EdError as e:
                if e.code != ed.ED_EBUSY:
                    raise
                time.sleep(1e-4)
    out = np.zeros(len(tickets), dtype=np.int64)
    waiting = list(range(len(tickets)))
    while waiting:
        still = []
        for i in waiting:
            st, k = ed.ed_poll(ctx.h, tickets[i])
            if st == ed.ED_OK:
                out[i] = k
            else:
                still.append(i)
        waiting = still
        if waiting:
            time.sleep(5e-5)
    return out


# ---------------------------------------------------------------- the least work
def _ext(k):
    return (k + 1) * (k + 1)


def work(case):
    """Each string read once and each answer written once; per diagonal and
    round the three-way maximum, the bound and one comparison (6 integer
    operations), and per byte of a table one multiply-add of 61 bits."""
    kind = case["kind"]
    if kind == "hash":
        return {"bytes": case["n"] + 8 * (case["n"] // case["block"] + 1), "flops": 2 * case["n"]}
    if kind == "pair":
        v = case["versions"]
        return {"bytes": (1 + v) * case["n"] + 8 * v, "flops": 6 * v * _ext(case["k"])}
    if kind == "script":
        return {"bytes": 2 * case["n"] + 24 * case["k"], "flops": 6 * _ext(case["k"])}
    n, k = _shapes(case)
    return {"bytes": int(2 * n.sum() + 8 * n.size), "flops": int(6 * sum(_ext(int(x)) for x in k))}


# ---------------------------------------------------------------- exact values
def _lcp(A, B, x, y):
    """LCP of A[x..] and B[y..] for vectors of rows, in windows that grow."""
    n, m = A.numel(), B.numel()
    l = torch.zeros_like(x)
    todo = torch.arange(x.numel(), device=x.device)
    w = 8
    while todo.numel():
        xs, ys = x[todo] + l[todo], y[todo] + l[todo]
        o = torch.arange(w, device=x.device)
        lim = torch.minimum(n - xs, m - ys).clamp_(max=w)
        eq = A[(xs[:, None] + o).clamp_(max=n - 1)] == B[(ys[:, None] + o).clamp_(max=m - 1)]
        eq &= o < lim[:, None]
        run_ = torch.where(eq.all(1), torch.full_like(lim, w), (~eq).to(torch.uint8).argmax(1))
        l[todo] += run_
        todo = todo[run_ == w]
        w = min(w * 8, max(8, (1 << 22) // max(1, todo.numel())))
    return l


def _distance(A, B, k_max):
    """Unit-cost edit distance by furthest-reaching rows, in 64-bit integers."""
    n, m = A.numel(), B.numel()
    if n == 0 or m == 0:
        return max(n, m)
    R = k_max + 2
    NEG = -(1 << 40)
    d = torch.arange(-R, R + 1, device=A.device)
    cap = torch.minimum(torch.full_like(d, n), m - d)
    L = torch.full_like(d, NEG)
    for t in range(k_max + 1):
        lo, hi = R + max(-t, -n), R + min(t, m)
        if t == 0:
            c = torch.zeros(1, dtype=torch.int64, device=A.device)
        else:
            c = torch.maximum(L[lo - 1:hi], torch.maximum(L[lo:hi + 1], L[lo + 1:hi + 2]) + 1)
            c = torch.minimum(c, cap[lo:hi + 1])
        L = L.clone()
        L[lo:hi + 1] = c + _lcp(A, B, c, c + d[lo:hi + 1])
        if abs(m - n) <= t and int(L[R + m - n]) == n:
            return t
    return None


def _mul61(a, b):
    """a * b mod 2^61 - 1 of int64 tensors below it (b may be a number)."""
    a1, a0 = a >> 31, a & 0x7FFFFFFF
    b1, b0 = b >> 31, b & 0x7FFFFFFF
    mid = a1 * b0 + a0 * b1                    # < 2^62
    r = 2 * (a1 * b1) + (mid >> 30) + ((mid & ((1 << 30) - 1)) << 31)
    r = (r & Q61) + (r >> 61)
    r = r + a0 * b0
    r = (r & Q61) + (r >> 61)
    return torch.where(r >= Q61, r - Q61, r)


def _hash_base(seed):
    z = (seed + 0x9E3779B97F4A7C15) & ((1 << 64) - 1)
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & ((1 << 64) - 1)
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & ((1 << 64) - 1)
    z ^= z >> 31
    return 256 + z % (Q61 - 2 - 256)


def _table(X, base):
    """sum of (X[j] + 1) base^(i-1-j), j < i, for every i, by doubling."""
    h = X.long() + 1
    s, p = 1, base
    while s < h.numel():
        g = h.clone()
        for lo in range(s, h.numel(), CHUNK):
            hi = min(h.numel(), lo + CHUNK)
            v = _mul61(h[lo - s:hi - s], p) + h[lo:hi]
            g[lo:hi] = torch.where(v >= Q61, v - Q61, v)
        h = g
        s, p = 2 * s, p * p % Q61
    return torch.cat([torch.zeros(1, dtype=torch.int64, device=X.device), h])


def exact(case, seed):
    kind = case["kind"]
    if kind == "hash":
        X = _text(_gen(seed), case["n"], 64)
        return {"table": _table(X, _hash_base(HASH_SEED))[::case["block"]].contiguous()}
    if kind == "pair":
        if case["k"] * case["versions"] > 10_000:
            return None
        A, Bs = _versions(case, seed)
        return {"distances": [_distance(A, B, case["k"] + 7) for B in Bs]}
    if kind == "script":
        return {"distance": _distance(*_one_pair(case, seed), case["k"]), "ops": None}
    _, k = _shapes(case)
    if int(k.sum()) > 30_000:
        return None
    As, Bs = _pairs(case, seed)
    return {"distances": np.array([_distance(a, b, int(x)) for a, b, x in zip(As, Bs, k)], dtype=np.int64)}
