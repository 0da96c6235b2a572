"""The workloads by which this library's speed is judged.

Every case is one call (or one planned batch) through the public binding, on
int32 column pairs that lie on the GPU, as a program that keeps its relations
there would make it.  Inputs are seeded and generated on the GPU; their shapes
are those of the benchmark, the tests and the planner's training range:
uniform keys, ids spread over the whole int32 range, Zipf keys, power-law
friend graphs, star schemas and batches of small joins.
"""
from __future__ import annotations

import math

import torch

from paper_1905_13376_gb300 import binding

FM_BITMAPS = 16
FM_SEED = 0x5BD1E995
FM_PHI = 0.77351
FM_BITS = 28          # a sketch's bitmaps use bits 0 .. 27


def listed():
    return [
        # the smallest calls: a lookup-sized join inside a larger program
        # (the planner's smallest instances), where launches and latency count
        {"name": "linear_1k_count", "kind": "linear", "nr": 1021, "ns": 1024, "nt": 1537, "a": 4096, "b": 256,
         "c": 301, "keys": "uniform", "mode": "count"},
        # the paper's uniform workload: 2^16 tuples per relation
        {"name": "linear_64k_groupby", "kind": "linear", "nr": 65536, "ns": 65536, "nt": 65536, "a": 1 << 20,
         "b": 4096, "c": 4096, "keys": "uniform", "mode": "group_by_a"},
        # relations keyed by ids that are spread over the whole int32 range
        # (hashed or external identifiers), in no order, ragged sizes
        {"name": "linear_ids_6m_groupby", "kind": "linear", "nr": 6000011, "ns": 8388593, "nt": 5000087,
         "a": 1 << 20, "b": 1500007, "c": 2000003, "keys": "ids", "mode": "group_by_a"},
        # skewed join keys: the top B value holds more than a third of R and S
        {"name": "linear_zipf_4m_groupby", "kind": "linear", "nr": 1 << 22, "ns": 1 << 22, "nt": 1 << 22,
         "a": 1 << 20, "b": 1 << 20, "c": 1 << 22, "keys": "zipf", "s": 1.5, "mode": "group_by_a"},
        # result tuples written out and put in order: a fact relation with two
        # R tuples and one T tuple per key, two rows per S tuple
        {"name": "linear_4m_rows", "kind": "linear", "nr": 1 << 21, "ns": 1 << 22, "nt": 1 << 20, "a": 4096,
         "b": 1 << 20, "c": 1 << 20, "keys": "balanced", "mode": "rows"},
        # friends of friends of friends of every person (the headline):
        # an edge list sorted by source joined with itself twice
        {"name": "friends_1m_groupby", "kind": "friends", "vertices": 1 << 20, "degree": 32.0, "op": "linear",
         "order": "sorted", "mode": "group_by_a"},
        # one hop more: the chain of four relations
        {"name": "friends_1m_chain4", "kind": "friends", "vertices": 1 << 20, "degree": 32.0, "op": "chain4",
         "order": "sorted", "mode": "group_by_a"},
        # distinct friends of friends of friends, by sketches
        {"name": "friends_1m_sketch", "kind": "friends", "vertices": 1 << 20, "degree": 32.0, "op": "sketch",
         "order": "sorted", "mode": "group_by_a"},
        # a data-warehouse star: a large fact relation, two dimensions
        {"name": "star_64m_groupby", "kind": "star", "fact": 1 << 26, "dim": 1 << 20, "attr": 1 << 16,
         "order": "sorted", "mode": "group_by_a"},
        # triangle counting on a large power-law graph (the largest case)
        {"name": "triangles_4m_count", "kind": "triangles", "vertices": 1 << 22, "degree": 32.0, "cap": 4096.0,
         "mode": "count"},
        # the triangle list of a smaller graph, written out and put in order
        {"name": "triangles_1m_rows", "kind": "triangles", "vertices": 1 << 20, "degree": 24.0, "cap": 1024.0,
         "mode": "rows"},
        # many joins of uneven sizes in one planned launch
        {"name": "batch_1024", "kind": "batch", "queries": 1024, "lo": 1 << 8, "hi": 1 << 18},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["linear", "linear", "linear", "friends", "friends", "star", "triangles", "batch"])
    if kind == "linear":
        mode = rng.choice(["count", "group_by_a", "group_by_a", "rows"])
        if mode == "rows":
            # up to 2^22 tuples per relation, a few matches per tuple
            b, c = _log_int(rng, 1 << 10, 1 << 20), _log_int(rng, 1 << 10, 1 << 20)
            n = [b * rng.randint(1, 3), _log_int(rng, 1 << 10, 1 << 22), c * rng.randint(1, 3)]
            keys = "balanced"
        else:
            keys = rng.choice(["uniform", "ids", "zipf"])
            base = _log_int(rng, 1 << 10, 1 << 23)
            n = [max(64, int(base * rng.uniform(0.4, 1.0)) | 1) for _ in range(3)]
            b = _log_int(rng, max(64, base // 64), max(128, base))
            c = _log_int(rng, max(64, base // 64), max(128, base))
        a = _log_int(rng, 1 << 8, 1 << 12) if mode == "rows" else _log_int(rng, 1 << 10, 1 << 20)
        case = {"kind": "linear", "nr": n[0], "ns": n[1], "nt": n[2], "a": a, "b": b,
                "c": c, "keys": keys, "mode": mode}
        if keys == "zipf":
            case["s"] = round(rng.uniform(0.8, 1.5), 2)
        return case
    if kind == "friends":
        return {"kind": "friends", "vertices": _log_int(rng, 1 << 12, 1 << 20),
                "degree": round(rng.uniform(4.0, 32.0), 2), "op": rng.choice(["linear", "linear", "chain4", "sketch"]),
                "order": rng.choice(["sorted", "shuffled"]), "mode": "group_by_a"}
    if kind == "star":
        dim = _log_int(rng, 1 << 10, 1 << 20)
        return {"kind": "star", "fact": dim * rng.randint(8, 64) + rng.randint(0, 63), "dim": dim,
                "attr": _log_int(rng, 1 << 8, 1 << 16), "order": rng.choice(["sorted", "shuffled"]),
                "mode": "group_by_a"}
    if kind == "triangles":
        mode = rng.choice(["count", "group_by_a", "rows"])
        rows = mode == "rows"
        return {"kind": "triangles", "vertices": _log_int(rng, 1 << 12, 1 << (20 if rows else 21)),
                "degree": round(rng.uniform(4.0, 24.0 if rows else 32.0), 2),
                "cap": float(_log_int(rng, 64, 1024 if rows else 4096)), "mode": mode}
    return {"kind": "batch", "queries": _log_int(rng, 64, 1024), "lo": 1 << 8, "hi": 1 << 18}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed, part):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + part * 7919 + 12345) & ((1 << 62) - 1))
    return g


def _uniform(g, n, domain):
    return torch.randint(0, domain, (n,), generator=g, device="cuda", dtype=torch.int64)


def _zipf_cdf(domain, s):
    w = torch.arange(1, domain + 1, device="cuda", dtype=torch.float64).pow_(-s)
    return torch.cumsum(w, 0)


def _zipf(g, n, cdf, mult, off):
    """Zipf ranks through the bijection rank -> (rank * mult + off) mod domain."""
    domain = cdf.numel()
    u = torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * cdf[-1]
    k = torch.searchsorted(cdf, u, right=True).clamp_(max=domain - 1)
    return (k * mult + off) % domain


def _bijection(domain, seed, part):
    """(mult, off) of an affine bijection of [0, domain)."""
    x = (int(seed) * 2654435761 + part * 40503 + 97) & 0xFFFFFFFF
    mult = 1 + x % max(1, domain - 1)
    while math.gcd(mult, domain) != 1:
        mult = mult + 1 if mult + 1 < domain else 1
    return mult, (x >> 7) % domain


def _i32(x):
    return x.to(torch.int32)


def _spread(x):
    """Dense ids spread over the int32 range by an odd multiplier (a bijection of 32-bit words)."""
    y = (x * 2246822519 + 374761393) & 0xFFFFFFFF
    return torch.where(y >= 1 << 31, y - (1 << 32), y)


def _linear_inputs(case, seed):
    nr, ns, nt, a, b, c = (case[k] for k in ("nr", "ns", "nt", "a", "b", "c"))
    g = _gen(seed, 1)
    ra, td = _uniform(g, nr, a), _uniform(g, nt, a)
    if case["keys"] == "zipf":
        # B Zipf in R and S through one bijection (heavy keys meet), C uniform
        cdf = _zipf_cdf(b, case["s"])
        mult, off = _bijection(b, seed, 2)
        rb, sb = _zipf(g, nr, cdf, mult, off), _zipf(g, ns, cdf, mult, off)
    else:
        rb, sb = _uniform(g, nr, b), _uniform(g, ns, b)
    sc, tc = _uniform(g, ns, c), _uniform(g, nt, c)
    if case["keys"] == "balanced":   # every key equally often in R and in T, in random order
        rb = torch.randperm(nr, generator=g, device="cuda") % b
        tc = torch.randperm(nt, generator=g, device="cuda") % c
    if case["keys"] == "ids":
        rb, sb, sc, tc = _spread(rb), _spread(sb), _spread(sc), _spread(tc)
    return (_i32(ra), _i32(rb)), (_i32(sb), _i32(sc)), (_i32(tc), _i32(td))


def _power_law_cdf(vertices, degree, s=1.1, cap=4096.0):
    """Cumulative weights min(cap, c r^-s) with mean `degree` (c by bisection)."""
    base = torch.arange(1, vertices + 1, device="cuda", dtype=torch.float64).pow_(-s)
    lo, hi = 1e-6, 1e12
    for _ in range(60):
        mid = math.sqrt(lo * hi)
        if float((base * mid).clamp_(max=cap).mean()) < degree:
            lo = mid
        else:
            hi = mid
    return torch.cumsum((base * hi).clamp_(max=cap), 0)


def _by_weight(g, cdf, m):
    u = torch.rand(m, generator=g, device="cuda", dtype=torch.float64) * cdf[-1]
    return torch.searchsorted(cdf, u, right=True).clamp_(max=cdf.numel() - 1)


def _friends(case, seed):
    """Directed power-law edge list (src, dst): distinct, no self loops, sorted by
    (src, dst) or in random order."""
    v, d = case["vertices"], case["degree"]
    g = _gen(seed, 3)
    cdf = _power_law_cdf(v, d)
    m = int(round(v * d))
    po = torch.randperm(v, generator=g, device="cuda")
    pi = torch.randperm(v, generator=g, device="cuda")
    src, dst = po[_by_weight(g, cdf, m)], pi[_by_weight(g, cdf, m)]
    code = torch.unique((src * v + dst)[src != dst])
    if case["order"] == "shuffled":
        code = code[torch.randperm(code.numel(), generator=g, device="cuda")]
    return _i32(code // v), _i32(code % v)


def _triangle_inputs(case, seed):
    """Undirected power-law edges once as a < b: R = S = (a, b), T = (b, a).  For
    the triangle list the seed relabels one graph, so that the list's length is
    the case's own."""
    v, d = case["vertices"], case["degree"]
    g = _gen(0 if case["mode"] == "rows" else seed, 4)
    cdf = _power_law_cdf(v, d, cap=case["cap"])
    m = int(round(v * d / 2))
    p = torch.randperm(v, generator=_gen(seed, 8), device="cuda")
    x, y = p[_by_weight(g, cdf, m)], p[_by_weight(g, cdf, m)]
    lo, hi = torch.minimum(x, y), torch.maximum(x, y)
    code = torch.unique((lo * v + hi)[lo != hi])
    a, b = _i32(code // v), _i32(code % v)
    return (a, b), (a, b), (b, a)


def _star_inputs(case, seed):
    n, dim, attr = case["fact"], case["dim"], case["attr"]
    g = _gen(seed, 5)
    rb = torch.randperm(dim, generator=g, device="cuda")
    tc = torch.randperm(dim, generator=g, device="cuda")
    ra, td = _uniform(g, dim, attr), _uniform(g, dim, attr)
    sb, sc = _uniform(g, n, dim), _uniform(g, n, dim)
    if case["order"] == "sorted":
        sb, _ = torch.sort(sb)
    return (_i32(ra), _i32(rb)), (_i32(sb), _i32(sc)), (_i32(tc), _i32(td))


def _batch_inputs(case, seed):
    """Linear and cyclic joins in turn, sizes and key domains log-uniform, keys
    uniform or Zipf(1.0)."""
    g = _gen(seed, 6)
    queries = case["queries"]
    # the sizes are the case's own; the keys are the seed's
    u = torch.rand((queries, 8), generator=_gen(0, 7), device="cuda", dtype=torch.float64).cpu().tolist()
    cdf = _zipf_cdf(1 << 20, 1.0)
    lo, hi = math.log(case["lo"]), math.log(case["hi"])
    dlo, dhi = math.log(1 << 6), math.log(1 << 20)
    out = []
    for q in range(queries):
        n = [int(round(math.exp(lo + x * (hi - lo)))) for x in u[q][:3]]
        dom = [int(round(math.exp(dlo + x * (dhi - dlo)))) for x in u[q][3:7]]
        zipf = u[q][7] < 0.5

        def column(k, domain, part):
            if not zipf:
                return _i32(_uniform(g, k, domain))
            mult, off = _bijection(domain, seed, 64 * q + part)
            return _i32(_zipf(g, k, cdf[:domain], mult, off))

        A, B, C, D = dom
        last = D if q % 2 == 0 else A
        R = (column(n[0], A, 0), column(n[0], B, 1))
        S = (column(n[1], B, 2), column(n[1], C, 3))
        T = (column(n[2], C, 4), column(n[2], last, 5))
        out.append((binding.MWJ_LINEAR if q % 2 == 0 else binding.MWJ_CYCLIC, R, S, T))
    return out


# ---------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------

def prepare(case, seed):
    ctx = binding.Context(torch.cuda.current_device())
    kind = case["kind"]
    st = {"case": case, "ctx": ctx}
    if kind == "friends":
        st["F"] = _friends(case, seed)
    elif kind == "batch":
        st["batch"] = binding.Batch(ctx, _batch_inputs(case, seed))
    else:
        make = {"linear": _linear_inputs, "triangles": _triangle_inputs, "star": _star_inputs}[kind]
        st["rel"] = make(case, seed)
        if case["mode"] == "rows":
            # a program that writes rows out counts them first
            join = ctx.join3_linear if kind == "linear" else ctx.join3_cyclic
            st["rows"] = int(join(*st["rel"], "count")["total"].item())
    return st


def _packed(rows, bases):
    code = rows[:, 0].to(torch.int64)
    for k in range(1, len(bases)):
        code = code.mul_(bases[k]).add_(rows[:, k])
    return code


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    if kind == "batch":
        return state["batch"].launch()
    if kind == "friends":
        F, v = state["F"], case["vertices"]
        if case["op"] == "linear":
            return ctx.join3_linear(F, F, F, case["mode"], a_domain=v, sync=False)
        if case["op"] == "chain4":
            return ctx.join4_linear(F, F, F, F, case["mode"], a_domain=v, sync=False)
        return ctx.fm_linear(F, F, F, v, sync=False)
    R, S, T = state["rel"]
    mode = case["mode"]
    if kind == "star":
        return ctx.join3_star(R, S, T, mode, a_domain=case["attr"], sync=False)
    join, dom = (ctx.join3_linear, case.get("a")) if kind == "linear" else (ctx.join3_cyclic, case["vertices"])
    if mode == "rows":
        # rows come in no order: a program that compares or stores them sorts
        # them, here as one packed word per row
        out = join(R, S, T, mode, capacity=state["rows"], sync=False)
        bases = (case["a"], case["b"], case["c"], case["a"]) if kind == "linear" else (dom, dom, dom)
        return {"n_rows": out["n_rows"], "rows": torch.sort(_packed(out["rows"], bases)).values}
    return join(R, S, T, mode, a_domain=dom, sync=False)


def work(case):
    """Each input column read once (an edge list that plays several relations is
    one input), each output written once; one addition per input tuple of
    each relation, and for rows one written tuple each."""
    kind = case["kind"]
    group = case.get("mode") == "group_by_a"
    if kind == "linear":
        n = case["nr"] + case["ns"] + case["nt"]
        out = 8 * case["a"] if group else 8
        if case["mode"] == "rows":
            out = 8 * int(case["nr"] * case["ns"] / case["b"] * case["nt"] / case["c"])   # as packed words
        return {"bytes": 8 * n + out, "flops": n}
    if kind == "friends":
        e = int(case["vertices"] * case["degree"] * 0.98)
        out = {"linear": 8, "chain4": 8, "sketch": 4 * FM_BITMAPS + 4}[case["op"]] * case["vertices"]
        return {"bytes": 8 * e + out, "flops": (4 if case["op"] == "chain4" else 3) * e}
    if kind == "star":
        n = case["fact"] + 2 * case["dim"]
        return {"bytes": 8 * n + (8 * case["attr"] if group else 8), "flops": n}
    if kind == "triangles":
        # R, S and T are three relations over the same two columns
        e = int(case["vertices"] * case["degree"] / 2 * 0.98)
        return {"bytes": 8 * e + (8 * case["vertices"] if group else 8), "flops": 3 * e}
    mean = (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
    n = int(3 * mean * case["queries"])
    return {"bytes": 8 * n + 8 * case["queries"], "flops": n}


# ---------------------------------------------------------------------------
# the same numbers from plain torch, in 64 bits
# ---------------------------------------------------------------------------

def _sums_at(keys, weights, at):
    """Sum of weights[i] over keys[i] == at[j], for every j (exact int64)."""
    k, o = torch.sort(keys.to(torch.int64))
    pre = torch.zeros(k.numel() + 1, dtype=torch.int64, device=k.device)
    pre[1:] = torch.cumsum(weights[o], 0)
    at = at.to(torch.int64)
    return pre[torch.searchsorted(k, at, right=True)] - pre[torch.searchsorted(k, at)]


def _chain(rels, mode, a_domain):
    w = torch.ones_like(rels[-1][0], dtype=torch.int64)
    for left, right in zip(reversed(rels[:-1]), reversed(rels[1:])):
        w = _sums_at(right[0], w, left[1])
    out = {"total": w.sum().reshape(1)}
    if mode == "group_by_a":
        cnt = torch.zeros(a_domain, dtype=torch.int64, device=w.device)
        out["counts"] = cnt.index_add_(0, rels[0][0].to(torch.int64), w)
    return out


def _sketches(F, v):
    """The sketches of every vertex by reachability: a bit is set where the number
    of paths to a value that sets it is not zero."""
    src, dst = F[0].to(torch.int64), F[1].to(torch.int64)
    h = (dst ^ FM_SEED) & 0xFFFFFFFF
    h = h ^ (h >> 16)
    h = (h * 0x85EBCA6B) & 0xFFFFFFFF
    h = h ^ (h >> 13)
    h = (h * 0xC2B2AE35) & 0xFFFFFFFF
    h = h ^ (h >> 16)
    j, q = h & (FM_BITMAPS - 1), h >> 4
    r = torch.where(q == 0, torch.full_like(q, 27), torch.log2((q & -q).clamp_(min=1).to(torch.float64)).round().to(torch.int64))
    width = FM_BITMAPS * FM_BITS
    bits = torch.zeros(v * width, dtype=torch.float32, device=src.device)
    bits[src * width + j * FM_BITS + r] = 1.0
    bits = bits.view(v, width)
    o = torch.argsort(src, stable=True)
    crow = torch.zeros(v + 1, dtype=torch.int64, device=src.device)
    crow[1:] = torch.cumsum(torch.bincount(src, minlength=v), 0)
    adj = torch.sparse_csr_tensor(crow, dst[o], torch.ones_like(src, dtype=torch.float32), (v, v))
    for _ in range(2):
        bits = (adj @ bits).clamp_(max=1.0)
    bits = bits.view(v, FM_BITMAPS, FM_BITS)
    words = torch.zeros(v, FM_BITMAPS, dtype=torch.int64, device=src.device)
    low = torch.full((v, FM_BITMAPS), FM_BITS, dtype=torch.int64, device=src.device)
    for k in range(FM_BITS - 1, -1, -1):
        on = bits[:, :, k] > 0
        words |= on.to(torch.int64) << k
        low = torch.where(on, low, torch.full_like(low, k))
    est = (FM_BITMAPS / FM_PHI) * torch.exp2(low.sum(1).to(torch.float64) / FM_BITMAPS)
    return {"sketches": words.to(torch.int32), "estimates": est}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("triangles", "batch") or case["mode"] == "rows":
        return None
    if kind == "friends":
        F = _friends(case, seed)
        if case["op"] == "sketch":
            return _sketches(F, case["vertices"])
        return _chain([F] * (4 if case["op"] == "chain4" else 3), case["mode"], case["vertices"])
    make = _linear_inputs if kind == "linear" else _star_inputs
    return _chain(list(make(case, seed)), case["mode"], case["a"] if kind == "linear" else case["attr"])
