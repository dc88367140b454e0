"""What this framework's speed is measured on: calls of its public entry points as a user makes them.

The graphs are the ones of gen/workloads.py in shape: G(n, m) and R-MAT (0.57, 0.19, 0.19, 0.05) with
permuted ids, duplicates and self-loops among the raw edges.  They are drawn here with torch from the
seed, so that a case needs nothing but this file and the package.

Kinds of case:
  build_export    graph_build of a COO on the device, then the CSC back on the host
  build_wcc       graph_build, then weakly connected components
  build_pagerank  graph_build, then PageRank on the fresh graph (the paper's headline workload)
  pagerank        PageRank on a resident graph
  hits            HITS on a resident graph
  ppr             ppr_batch: personalised PageRank, `graphs` graphs with `seeds` seed nodes each
  serve           requests to a running server, all answers fetched
"""
import math

import numpy as np
import torch

import paper_1606_07550_gb300 as gpr

DTYPES = {"fp32": gpr.FP32, "bf16": gpr.BF16}
DAMPING = 0.85


# ---- cases ------------------------------------------------------------------------------------------

def listed():
    return [
        # The smallest calls: a G(10,000, 100,000) graph, where launches and latency count.
        {"name": "build-er-10k", "kind": "build_export", "model": "er", "n": 10_000, "m": 100_000},
        {"name": "pagerank-er-10k", "kind": "pagerank", "model": "er", "n": 10_000, "m": 100_000, "iters": 50,
         "dtype": "fp32"},
        # One graph of the size of the serving pool's middle, odd n, 16-bit contributions.
        {"name": "pagerank-rmat-18-bf16", "kind": "pagerank", "model": "rmat", "n": 250_007, "m": 4_000_003, "iters": 50,
         "dtype": "bf16"},
        # Social-network scale (LiveJournal's shape): a resident graph ranked, and one loaded and taken apart.
        {"name": "pagerank-rmat-lj", "kind": "pagerank", "model": "rmat", "n": 4_800_000, "m": 69_000_000, "iters": 100,
         "dtype": "fp32"},
        {"name": "build-wcc-rmat-lj", "kind": "build_wcc", "model": "rmat", "n": 4_800_000, "m": 69_000_000},
        # The headline workload, the largest: R-MAT scale 25, edge factor 32, built and ranked.
        {"name": "build-pagerank-rmat-25", "kind": "build_pagerank", "model": "rmat", "n": 1 << 25, "m": 1 << 30,
         "iters": 100, "dtype": "fp32"},
        # Another analytic on the same steps, both edge directions: the pool's largest graph.
        {"name": "hits-rmat-22", "kind": "hits", "model": "rmat", "n": 1 << 22, "m": 16 << 22, "iters": 20},
        # Who is near this node?  One seed on a middling graph: the latency of a single query.
        {"name": "ppr-one-seed", "kind": "ppr", "graphs": 1, "n_lo": 100_000, "n_hi": 100_000, "deg_lo": 16, "deg_hi": 16,
         "seeds": 1, "iters": 50, "dtype": "fp32"},
        # The same for a group of nodes of one large graph.
        {"name": "ppr-one-graph-64", "kind": "ppr", "graphs": 1, "n_lo": 1 << 20, "n_hi": 1 << 20, "deg_lo": 16,
         "deg_hi": 16, "seeds": 64, "iters": 50, "dtype": "fp32"},
        # Many small and middling graphs at once (the batched workload, a sixteenth of its 4,096 graphs).
        {"name": "ppr-batch-256", "kind": "ppr", "graphs": 256, "n_lo": 1_000, "n_hi": 200_000, "deg_lo": 4,
         "deg_hi": 32, "seeds": 64, "iters": 50, "dtype": "fp32"},
        # The same with 16-bit contributions, a smaller batch.
        {"name": "ppr-batch-64-bf16", "kind": "ppr", "graphs": 64, "n_lo": 1_000, "n_hi": 200_000, "deg_lo": 4,
         "deg_hi": 32, "seeds": 64, "iters": 50, "dtype": "bf16"},
        # A burst of requests to the server, over a pool with one graph of each of its scales 14 to 22.
        {"name": "serve-burst", "kind": "serve", "scale_lo": 14, "scale_hi": 22, "requests": 32, "budget_gb": 40},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["build_export", "pagerank", "pagerank", "build_wcc", "build_pagerank", "hits", "ppr", "ppr", "ppr",
                       "serve"])
    if kind == "serve":
        lo = rng.randint(14, 18)
        return {"kind": kind, "scale_lo": lo, "scale_hi": rng.randint(lo, 22), "requests": rng.randint(5, 32),
                "budget_gb": 40}
    if kind == "ppr":
        c = {"kind": kind, "seeds": rng.choice([1, rng.randint(2, 63), 64]), "iters": rng.choice([20, 50]),
             "dtype": rng.choice(["fp32", "bf16"])}
        if rng.random() < 0.5:  # one graph
            n, deg = _log(rng, 1_000, 1 << 20), rng.randint(4, 32)
            deg = min(deg, max(4, (16 << 20) // n))
            return dict(c, graphs=1, n_lo=n, n_hi=n, deg_lo=deg, deg_hi=deg)
        return dict(c, graphs=_log(rng, 2, 256), n_lo=1_000, n_hi=_log(rng, 20_000, 200_000), deg_lo=4, deg_hi=32)
    model = rng.choice(["er", "rmat", "rmat"])
    lo, hi = {"build_export": (1_000, 300_000), "pagerank": (1_000, 4_800_000), "build_wcc": (100_000, 4_800_000),
              "build_pagerank": (1_000_000, 1 << 24), "hits": (10_000, 1 << 22)}[kind]
    n = _log(rng, lo, hi)
    c = {"kind": kind, "model": model, "n": n, "m": int(n * rng.uniform(4, 14 if kind != "build_pagerank" else 32))}
    if kind in ("pagerank", "build_pagerank"):
        c["iters"], c["dtype"] = rng.choice([10, 50, 100]), rng.choice(["fp32", "bf16"])
    if kind == "hits":
        c["iters"] = 20
    return c


# ---- inputs -----------------------------------------------------------------------------------------

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _levels(count, levels, gen):
    """`levels` R-MAT quadrant draws for each of `count` edges, packed into source and destination bits."""
    s = torch.zeros(count, dtype=torch.int32, device="cuda")
    d = torch.zeros(count, dtype=torch.int32, device="cuda")
    for _ in range(levels):
        r = torch.rand(count, device="cuda", generator=gen)
        sb = r >= 0.76
        db = (r >= 0.57) ^ sb ^ (r >= 0.95)
        s.mul_(2).add_(sb)
        d.mul_(2).add_(db)
    return s, d


def _rmat(n_of, m_of, gen):
    """R-MAT edges of graphs of n_of[i] nodes with m_of[i] raw edges each, one after another: every edge takes as
    many of its quadrant draws as its graph has levels, is drawn again until both ends are nodes, and the nodes of
    each graph are permuted.  Ids are local to their graph."""
    total, most = sum(m_of), max(n_of)
    top = max(1, (most - 1).bit_length())
    src = torch.empty(total, dtype=torch.int32, device="cuda")
    dst = torch.empty(total, dtype=torch.int32, device="cuda")
    one = len(n_of) == 1
    if not one:
        which = torch.repeat_interleave(torch.arange(len(n_of), device="cuda"), torch.tensor(m_of, device="cuda"))
        shift = torch.tensor([top - max(1, (n - 1).bit_length()) for n in n_of], dtype=torch.int32, device="cuda")
        size = torch.tensor(n_of, dtype=torch.int32, device="cuda")
    for a in range(0, total, 1 << 26):
        b = min(total, a + (1 << 26))
        at = None
        for _ in range(64):
            s, d = _levels(b - a if at is None else at.numel(), top, gen)
            if not one:
                w = which[a:b] if at is None else which[a + at]
                s >>= shift[w]
                d >>= shift[w]
            if at is None:
                src[a:b], dst[a:b] = s, d
            else:
                src[a + at], dst[a + at] = s, d
            if one and most == 1 << top:
                break
            lim = most if one else size[w]
            bad = ((s >= lim) | (d >= lim)).nonzero().flatten()
            at = bad if at is None else at[bad]
            if at.numel() == 0:
                break
        if at is not None and at.numel():
            lim = most if one else size[which[a + at]]
            src[a + at] %= lim
            dst[a + at] %= lim
    e = 0
    for n, m in zip(n_of, m_of):
        perm = torch.randperm(n, dtype=torch.int32, device="cuda", generator=gen)
        for ids in (src, dst):
            for a in range(e, e + m, 1 << 27):
                b = min(e + m, a + (1 << 27))
                ids[a:b] = perm[ids[a:b]]
        e += m
    return src, dst


def _edges(case, seed):
    """The raw COO of a case with one graph."""
    gen = _generator(seed)
    n, m = case["n"], case["m"]
    if case["model"] == "er":
        return tuple(torch.randint(0, n, (m,), dtype=torch.int32, device="cuda", generator=gen) for _ in range(2))
    return _rmat([n], [m], gen)


def _ppr_inputs(case, seed):
    """Per graph (n, src, dst, seed nodes).  The graphs' sizes belong to the case, their edges to the seed."""
    rng = np.random.default_rng(seed)
    u = np.random.default_rng(case["graphs"]).random((case["graphs"], 2))
    lo, hi = math.log(case["n_lo"]), math.log(case["n_hi"])
    n_of = [int(round(math.exp(lo + (hi - lo) * a))) for a in u[:, 0]]
    m_of = [int(round(n * (case["deg_lo"] + (case["deg_hi"] - case["deg_lo"]) * b))) for n, b in zip(n_of, u[:, 1])]
    src, dst = _rmat(n_of, m_of, _generator(seed))
    out, e = [], 0
    for n, m in zip(n_of, m_of):
        out.append((n, src[e:e + m], dst[e:e + m], rng.integers(0, n, case["seeds"]).astype(np.int32)))
        e += m
    return out


def _serve_inputs(case, seed):
    """The pool's graphs (n, src, dst), and requests (graph, seeds, damping, tol, dtype name).  Which graph a request
    names, how many seeds it has and to what tolerance belong to the case; the rest to the seed."""
    pool = []
    for j, s in enumerate(range(case["scale_lo"], case["scale_hi"] + 1)):
        pool.append((1 << s, *_rmat([1 << s], [16 << s], _generator(seed + 1000 * j))))
    rng, mix = np.random.default_rng(seed), np.random.default_rng(case["requests"])
    reqs = []
    for _ in range(case["requests"]):
        g = int(mix.integers(len(pool)))
        k = int(mix.integers(1, 65))
        tol = 1e-6 if mix.random() < 0.5 else 1e-3
        dtype = "bf16" if tol == 1e-3 and mix.random() < 0.5 else "fp32"
        reqs.append((g, rng.integers(0, pool[g][0], k).astype(np.int32), float(np.float32(rng.uniform(0.8, 0.9))), tol,
                     dtype))
    return pool, reqs


# ---- a pass -----------------------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "kind": kind}
    if kind == "ppr":
        inputs = _ppr_inputs(case, seed)
        k = case["seeds"]
        st["x"] = torch.empty(sum(n for n, *_ in inputs) * k, dtype=torch.float32, device="cuda")
        st["requests"], at = [], 0
        for n, s, d, seeds in inputs:
            g = gpr.graph_build(s.contiguous(), d.contiguous(), n)
            st["requests"].append((g, seeds, DAMPING, st["x"][at:at + n * k].view(n, k)))
            at += n * k
        return st
    if kind == "serve":
        pool, reqs = _serve_inputs(case, seed)
        st["pool"] = [gpr.graph_build(s, d, n) for n, s, d in pool]
        st["server"] = gpr.Server(st["pool"], case["budget_gb"] << 30)
        st["x"] = torch.empty(sum(pool[g][0] * len(seeds) for g, seeds, *_ in reqs), dtype=torch.float32, device="cuda")
        st["requests"], at = [], 0
        for g, seeds, damping, tol, dtype in reqs:
            size = pool[g][0] * len(seeds)
            st["requests"].append((g, seeds, damping, tol, DTYPES[dtype], st["x"][at:at + size]))
            at += size
        return st
    src, dst = _edges(case, seed)
    n = case["n"]
    st["n"] = n
    if kind in ("build_export", "build_wcc", "build_pagerank"):
        st["src"], st["dst"] = src, dst
    if kind == "build_export":
        st["rows"] = np.zeros(case["m"], np.int32)  # distinct edges are at most the raw ones
    else:
        st["g"] = gpr.graph_build(src, dst, n)
    if kind == "build_wcc":
        st["labels"] = torch.empty(n, dtype=torch.int32, device="cuda")
    if kind in ("pagerank", "build_pagerank"):
        st["x"] = torch.empty(n, dtype=torch.float32, device="cuda")
    if kind == "hits":
        st["hub"], st["auth"] = (torch.empty(n, dtype=torch.float32, device="cuda") for _ in range(2))
    return st


def run(st):
    case, kind = st["case"], st["kind"]
    if kind == "build_export":
        g = gpr.graph_build(st["src"], st["dst"], st["n"])
        col_ptr, row_idx, outdeg = g.export()
        g.free()
        st["rows"][:len(row_idx)] = row_idx
        return col_ptr, st["rows"], outdeg
    if kind == "build_wcc":
        g = gpr.graph_build(st["src"], st["dst"], st["n"])
        info = g.info()
        count = gpr.wcc(g, st["labels"])
        g.free()
        return st["labels"], count, info.m, info.n_dangling, info.max_in_degree, info.max_out_degree
    if kind == "build_pagerank":
        g = gpr.graph_build(st["src"], st["dst"], st["n"])
        gpr.pagerank(g, st["x"], damping=DAMPING, iters=case["iters"], dtype=DTYPES[case["dtype"]], stats=True)
        g.free()
        return st["x"]
    if kind == "pagerank":
        gpr.pagerank(st["g"], st["x"], damping=DAMPING, iters=case["iters"], dtype=DTYPES[case["dtype"]])
        return st["x"]
    if kind == "hits":
        gpr.hits(st["g"], st["hub"], st["auth"], iters=case["iters"])
        return st["hub"], st["auth"]
    if kind == "ppr":
        done = gpr.ppr_batch(st["requests"], max_iters=case["iters"], dtype=DTYPES[case["dtype"]])
        return st["x"], np.concatenate([iters for iters, _ in done])
    if kind == "serve":
        server = st["server"]
        tickets = [server.submit(g, seeds, damping=damping, tol=tol, max_iters=200, dtype=dtype)
                   for g, seeds, damping, tol, dtype, _ in st["requests"]]
        for ticket, (*_, out) in zip(tickets, st["requests"]):
            while server.poll(ticket, timeout_us=1_000_000) is None:
                pass
            server.fetch(ticket, out)
            server.release(ticket)
        return st["x"]
    raise ValueError(kind)


# ---- what a pass cannot do without -----------------------------------------------------------------

def _step(n, m, k):
    """One step on k columns: the in-adjacency (sources and offsets), the rank vectors read and written."""
    return {"bytes": 4 * m + 4 * (n + 1) + 8 * n * k, "flops": 2 * m * k}


def work(case):
    """Raw edges stand for distinct ones.  A step reads the graph and the ranks once and writes the ranks once;
    every step counts."""
    kind = case["kind"]
    if kind == "ppr":
        lo, hi = math.log(case["n_lo"]), math.log(case["n_hi"])
        mean_n = case["n_lo"] if hi == lo else (case["n_hi"] - case["n_lo"]) / (hi - lo)
        one = _step(mean_n, mean_n * (case["deg_lo"] + case["deg_hi"]) / 2, case["seeds"])
        return {u: v * case["graphs"] * case["iters"] for u, v in one.items()}
    if kind == "serve":
        # steps of a column: half the requests to 1e-6, half to 1e-3, at the mean damping; columns of one graph share
        # its in-adjacency in groups of 64
        steps = sum(math.log(tol * 0.15 / 0.85 / 2) / math.log(0.85) for tol in (1e-6, 1e-3)) / 2
        scales = range(case["scale_lo"], case["scale_hi"] + 1)
        cols = 32.5 * case["requests"] / len(scales)
        all_ = [_step(1 << s, 16 << s, cols) for s in scales]
        extra = max(0.0, cols / 64 - 1)
        return {"bytes": steps * sum(w["bytes"] + extra * (68 << s) for w, s in zip(all_, scales)),
                "flops": steps * sum(w["flops"] for w in all_)}
    n, m = case["n"], case["m"]
    build = 8 * m + 4 * m + 8 * n  # the COO read, the CSC and degrees written
    if kind == "build_export":
        return {"bytes": build, "flops": 0}
    if kind == "build_wcc":
        return {"bytes": build + 4 * m + 4 * n, "flops": 0}
    one = _step(n, m, 1)
    steps = case["iters"] * (2 if kind == "hits" else 1)
    return {"bytes": steps * one["bytes"] + (build if kind == "build_pagerank" else 0), "flops": steps * one["flops"]}


# ---- the same in 64 bits ----------------------------------------------------------------------------

def _simple(n, src, dst):
    """The distinct edges without self-loops, by (destination, source)."""
    key = dst.to(torch.int64) * n + src
    key = key[src != dst]
    key = torch.unique_consecutive(torch.sort(key).values)
    v = torch.div(key, n, rounding_mode="floor")
    return key - v * n, v


def _matrix(n, src, dst, weight):
    """The sparse matrix with weight[i] at (dst[i], src[i]); the edges are in order of (dst, src)."""
    at = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(torch.bincount(dst, minlength=n), 0, out=at[1:])
    return torch.sparse_csr_tensor(at, src, weight, (n, n), dtype=torch.float64)


def _walk_matrix(n, src, dst):
    """The column-stochastic matrix (but for dangling nodes) and the mask of dangling nodes."""
    src, dst = _simple(n, src, dst)
    deg = torch.bincount(src, minlength=n)
    return _matrix(n, src, dst, 1.0 / deg.to(torch.float64)[src]), deg == 0


def _pagerank64(n, src, dst, iters):
    P, dangling = _walk_matrix(n, src, dst)
    x = torch.full((n,), 1.0 / n, dtype=torch.float64, device="cuda")
    for _ in range(iters):
        x = DAMPING * (P @ x + x[dangling].sum() / n) + (1 - DAMPING) / n
    return x


def _ppr64(n, src, dst, seeds, damping, iters, tol=0.0):
    P, dangling = _walk_matrix(n, src, dst)
    k = len(seeds)
    x = torch.zeros(n, k, dtype=torch.float64, device="cuda")
    at = (torch.as_tensor(seeds, dtype=torch.int64, device="cuda"), torch.arange(k, device="cuda"))
    x[at] = 1.0
    going = torch.ones(k, dtype=torch.bool, device="cuda")
    for _ in range(iters):
        y = damping * (P @ x)
        y[at] += (1 - damping) + damping * x[dangling].sum(0)
        off = (y - x).abs().sum(0)
        x = torch.where(going, y, x)
        if tol > 0:
            going = going & (damping / (1 - damping) * off > tol)
            if not bool(going.any()):
                break
    return x


def _hits64(n, src, dst, iters):
    src, dst = _simple(n, src, dst)
    ones = torch.ones(src.numel(), dtype=torch.float64, device="cuda")
    to_auth = _matrix(n, src, dst, ones)
    order = torch.sort(src, stable=True).indices
    to_hub = _matrix(n, dst[order], src[order], ones)
    hub = torch.full((n,), n ** -0.5, dtype=torch.float64, device="cuda")
    auth = hub.clone()
    for _ in range(iters):
        auth = to_auth @ hub
        auth = auth / auth.norm().clamp_min(1e-300)
        hub = to_hub @ auth
        hub = hub / hub.norm().clamp_min(1e-300)
    return hub, auth


def exact(case, seed):
    kind = case["kind"]
    if kind in ("build_export", "build_wcc"):
        return None  # whole numbers
    if kind == "ppr":
        return torch.cat([_ppr64(n, s, d, seeds, DAMPING, case["iters"]).flatten()
                          for n, s, d, seeds in _ppr_inputs(case, seed)]), None
    if kind == "serve":
        pool, reqs = _serve_inputs(case, seed)
        return torch.cat([_ppr64(*pool[g], seeds, damping, 200, tol).flatten() for g, seeds, damping, tol, _ in reqs])
    src, dst = _edges(case, seed)
    if kind == "hits":
        return _hits64(case["n"], src, dst, case["iters"])
    return _pagerank64(case["n"], src, dst, case["iters"])
