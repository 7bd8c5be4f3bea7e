"""What a user of this framework has it do, as measurable cases.

A case is a graph with an influence model and one use of it:

  query        one influence query on resident sketches (host seeds in, host estimate out)
  query_batch  a block of queries in one call
  serve        a burst of queries through the continuous-batching server
  build        every node's combined bottom-k sketch (Algorithm 2) on a context the program keeps
  batch        the same over many graphs in one context
  greedy       SKIM seed selection with its thresholds (Algorithm 1)
  step         all of it from host edges: context, sketches, seeds, queries, context destroyed

Graphs are Erdos-Renyi or R-MAT (0.57, 0.19, 0.19, 0.05), drawn on the GPU from the case's seed, without
duplicates and self-loops.  Influence models: uniform p, weighted cascade ("wc"), trivalency ("tv").
"""
import math
import random

import numpy as np
import torch

import paper_1408_6282_gb300 as pkg

MODELS = {"uniform": pkg.PROB_UNIFORM, "wc": pkg.PROB_WC, "tv": pkg.PROB_TRIVALENCY}
RANKS = {"uniform": pkg.RANKS_UNIFORM, "perm": pkg.RANKS_PERMUTATION, "ic": pkg.RANKS_IC_MODEL}
M64 = (1 << 64) - 1


def _case(name, op, graph, n, m, model, p, l, k, ranks="uniform", rows=True, seeds=0, queries=0, graphs=1):
    c = {"op": op, "graph": graph, "n": n, "m": m, "model": model, "p": p, "l": l, "k": k, "ranks": ranks,
         "rows": rows, "seeds": seeds, "queries": queries, "graphs": graphs}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one question to an oracle over a small network: latency and launches
        _case("query_er4096", "query", "er", 4096, 32768, "uniform", 0.1, 16, 16, seeds=10),
        # an analyst's block of 1000 questions, |S| from 1 to 1000, over a million-node network
        _case("queries_rmat20_wc", "query_batch", "rmat", 1 << 20, 16 << 20, "wc", 0.0, 64, 64, queries=1000),
        # a burst of requests at a serving process
        _case("serve_rmat18_wc", "serve", "rmat", 1 << 18, 16 << 18, "wc", 0.0, 64, 64, queries=3000),
        # sketches of a small network: the smallest build
        _case("build_er4096", "build", "er", 4096, 32768, "uniform", 0.1, 16, 16),
        # odd sizes everywhere (n, m, l, k), structured permutation ranks
        _case("build_er50021_perm", "build", "er", 50021, 400009, "uniform", 0.12, 37, 21, ranks="perm"),
        # the headline build: weighted cascade, searches of a few nodes each
        _case("build_rmat20_wc", "build", "rmat", 1 << 20, 16 << 20, "wc", 0.0, 64, 64),
        # the largest: uniform p, hub-heavy searches that reach thousands of nodes
        _case("build_rmat22_p01", "build", "rmat", 1 << 22, 16 << 22, "uniform", 0.01, 64, 64),
        # a fresh instance per rank: coins are drawn in the searches
        _case("build_rmat15_ic", "build", "rmat", 1 << 15, 16 << 15, "uniform", 0.01, 1, 64, ranks="ic"),
        # many small graphs in one context (trivalency, k = 32)
        _case("batch24_tv", "batch", "rmat", 1 << 14, 16 << 14, "tv", 0.0, 64, 32, graphs=24),
        # seed selection on a quarter-million-node network
        _case("greedy_rmat18_wc", "greedy", "rmat", 1 << 18, 16 << 18, "wc", 0.0, 64, 64, seeds=50),
        # seed selection where the first seeds cover a giant component
        _case("greedy_rmat20_p01", "greedy", "rmat", 1 << 20, 16 << 20, "uniform", 0.01, 64, 64, seeds=50),
        # everything from host edges to answers, the context included
        _case("step_rmat20_wc", "step", "rmat", 1 << 20, 16 << 20, "wc", 0.0, 64, 64, seeds=50, queries=1000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    op = rng.choice(["query", "query_batch", "build", "build", "build", "batch", "greedy", "greedy", "step"])
    graph = rng.choice(["er", "rmat", "rmat"])
    n = _log(rng, 4096, 1 << 20)
    if graph == "rmat":  # scales of the generator, sizes between them as in a trimmed crawl
        n = rng.choice([1 << (n.bit_length() - 1), n])
    m = n * rng.choice([4, 8, 16, 16]) + rng.randrange(0, 97)
    model = rng.choice(["uniform", "wc", "wc", "tv"])
    p = rng.choice([0.01, 0.03, 0.1]) if model == "uniform" else 0.0
    if p * (m // n) > (1.2 if n <= 1 << 17 else 0.5):  # live graphs stay as sparse as in the networks that are studied
        p = 0.01
    l = rng.choice([64, 64, 64, 37, 16])
    k = rng.choice([64, 64, 32, 21, 16])
    c = _case(None, op, graph, n, m, model, p, l, k)
    if op == "build":
        c["ranks"] = rng.choice(["uniform", "uniform", "perm"])
        c["rows"] = n > (1 << 17) or rng.random() < 0.8
    elif op == "batch":
        c.update(n=_log(rng, 1024, 1 << 15), graphs=rng.randrange(3, 33))
        c["m"] = c["n"] * 16 + 1
    elif op == "greedy":
        c["seeds"] = rng.randrange(5, 81)
    elif op == "step":
        c.update(seeds=rng.randrange(1, 51), queries=_log(rng, 10, 1000))
    elif op == "query":
        c["seeds"] = _log(rng, 1, 1000)
    else:
        c["queries"] = _log(rng, 10, 2000)
    return c


# ---- inputs --------------------------------------------------------------------

def _edges(graph, n, m, seed, device="cuda"):
    """Canonical (src, dst) int32 tensors: sorted, distinct, no self-loops."""
    g = torch.Generator(device=device)
    g.manual_seed(seed)
    if graph == "er":
        u = torch.randint(0, n, (m,), generator=g, device=device)
        v = torch.randint(0, n, (m,), generator=g, device=device)
    else:
        u = torch.zeros(m, dtype=torch.int64, device=device)
        v = torch.zeros(m, dtype=torch.int64, device=device)
        for _ in range((n - 1).bit_length()):
            x = torch.rand(m, generator=g, device=device)
            u = 2 * u + (x >= 0.76)
            v = 2 * v + (((x >= 0.57) & (x < 0.76)) | (x >= 0.95))
        keep = (u < n) & (v < n)
        u, v = u[keep], v[keep]
    key = torch.unique(((u << 32) | v)[u != v])
    return (key >> 32).to(torch.int32), (key & 0xFFFFFFFF).to(torch.int32)


def _keys(seed):
    r = random.Random(seed * 7919 + 1)
    return [r.getrandbits(64) for _ in range(3)]  # coins, ranks, trivalency classes


def _context(case, src, dst, seed):
    coin, rank, prob = _keys(seed)
    return pkg.Skim(case["n"], src, dst, case["l"], case["k"], MODELS[case["model"]], case["p"], coin, rank, prob,
                    rank_mode=RANKS[case["ranks"]])


def _query_sets(n, count, seed):
    """|S| = 10^(3U), seeds distinct; as CSR arrays."""
    rng = np.random.default_rng(seed)
    size = np.minimum(np.clip(np.floor(10.0 ** (3.0 * rng.random(count))).astype(np.int64), 1, 1000), n)
    off = np.zeros(count + 1, np.uint64)
    off[1:] = np.cumsum(size)
    flat = np.concatenate([rng.choice(n, int(s), replace=False) for s in size]).astype(np.uint32)
    return off, flat


def _batch_graphs(case, seed):
    """(n, src, dst) host arrays of a batch's graphs: sizes from a sixteenth of case n up to it."""
    r = random.Random(case["graphs"])  # the sizes are the case's, the graphs the seed's
    out = []
    for i in range(case["graphs"]):
        n = max(64, int(case["n"] * 2.0 ** r.uniform(-4, 0)))
        src, dst = _edges(case["graph"], n, case["m"] * n // case["n"], seed * 131 + i)
        out.append((n, src.cpu().numpy().view(np.uint32), dst.cpu().numpy().view(np.uint32)))
    return out


def prepare(case, seed):
    op, n, k = case["op"], case["n"], case["k"]
    s = {"case": case, "op": op}
    if op == "batch":
        gs = _batch_graphs(case, seed)
        keys = [_keys(seed * 1009 + i) for i in range(len(gs))]
        sk = pkg.Skim.batch(gs, case["l"], k, [MODELS[case["model"]]] * len(gs), [case["p"]] * len(gs),
                            [x[0] for x in keys], [x[1] for x in keys], [x[2] for x in keys])
        n = sk.n
    else:
        src, dst = _edges(case["graph"], n, case["m"], seed)
        if op == "step":
            s["src"] = src.cpu().pin_memory().numpy().view(np.uint32)
            s["dst"] = dst.cpu().pin_memory().numpy().view(np.uint32)
            s["seed"] = seed
            s["off"], s["flat"] = _query_sets(n, case["queries"], seed)
            return s
        sk = _context(case, src, dst, seed)
        torch.cuda.synchronize()
    s["sk"] = sk
    if op in ("build", "batch"):
        sk.set_live_rows(case["rows"])
        s["x"] = torch.empty((n, k), dtype=torch.int64, device="cuda")
        s["len"] = torch.empty(n, dtype=torch.int32, device="cuda")
    elif op != "greedy":
        sk.build_sketches()
        if op == "query":
            s["set"] = np.random.default_rng(seed).choice(n, case["seeds"], replace=False).astype(np.uint32)
        else:
            s["off"], s["flat"] = _query_sets(n, case["queries"], seed)
        if op == "serve":
            s["sets"] = np.split(s["flat"], s["off"][1:-1].astype(np.int64))
            s["arrive"] = np.zeros(case["queries"])
            s["srv"] = _Serving(sk)
    return s


class _Serving:
    """A server that is stopped before its context goes."""

    def __init__(self, sk):
        self.sk = sk
        self.server = sk.server()

    def __del__(self):
        try:
            self.server.stop()
        except Exception:
            pass


# ---- one pass ------------------------------------------------------------------

def _signed(a):
    return a.view(np.int64 if a.dtype == np.uint64 else np.int32) if a.dtype.kind == "u" else a


def _queries(sk, off, flat):
    est = np.empty(off.shape[0] - 1)
    pkg.skim_oracle_query_batch(sk.ctx, off, est.shape[0], flat, est, 0)
    return est


def run(s):
    op, case = s["op"], s["case"]
    if op == "query":
        return s["sk"].query(s["set"])
    if op == "query_batch":
        return _queries(s["sk"], s["off"], s["flat"])
    if op == "serve":
        return s["srv"].server.replay(s["arrive"], s["sets"])[1]
    if op in ("build", "batch"):
        s["sk"].build_sketches()
        pkg.skim_get_sketches(s["sk"].ctx, s["x"], s["len"], 1)
        return {"x": s["x"], "len": s["len"]}
    if op == "greedy":
        s["sk"].greedy_reset()
        return [_signed(a) for a in s["sk"].greedy_stops(case["seeds"])]
    with _context(case, s["src"], s["dst"], s["seed"]) as sk:
        sk.build_sketches()
        seeds, cov = sk.greedy(case["seeds"])
        est = _queries(sk, s["off"], s["flat"])
        nodes = sk.node_estimates()
    return {"seeds": _signed(seeds), "cov": _signed(cov), "est": est, "nodes": nodes}


def work(case):
    """Stored instances (a row entry per node and instance, live edges), the rank order and the outputs, each once;
    where coins are drawn in the searches, the edges with their coins in their place (27 integer operations a coin)."""
    n, m, l, k = case["n"] * case["graphs"], case["m"] * case["graphs"], case["l"], case["k"]
    per_query = 1000 / math.log(1000) * (8 * k + 4)  # mean |S| of 10^(3U)
    live = {"uniform": m * l * case["p"], "wc": n * l * 0.55, "tv": m * l * 0.037}[case["model"]]
    stored = 4 * live + 4 * n * l
    sketches = 8 * n * k + 4 * n
    op = case["op"]
    if op == "query":
        return {"bytes": case["seeds"] * (8 * k + 4) + 8, "flops": 0}
    if op in ("query_batch", "serve"):
        return {"bytes": case["queries"] * per_query, "flops": 0}
    if op in ("build", "batch"):
        if case["ranks"] == "ic":
            return {"bytes": 12 * m + 12 * n * k + sketches, "flops": 27 * m * k}
        positions = n * (min(k, l) if case["ranks"] == "perm" else l)
        if not case["rows"]:
            return {"bytes": 12 * m + 12 * positions + sketches, "flops": 27 * m * l}
        return {"bytes": stored + 12 * positions + sketches, "flops": 0}
    if op == "greedy":
        return {"bytes": stored + 12 * n, "flops": 0}
    return {"bytes": 8 * m + stored + 12 * n * l + sketches + case["queries"] * per_query, "flops": 27 * m * l}


# ---- what the estimates are, in 64 bits ------------------------------------------

def _fmix(z):
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


_G = np.uint64(0x9E3779B97F4A7C15)


def _plain_sketches(case, seed):
    """Sketches of a small case from the definitions: pair ranks, live edges by their coins, and bottom-k merges
    along live edges until nothing changes."""
    n, l, k = case["n"], case["l"], case["k"]
    src, dst = (t.cpu().numpy().astype(np.uint64) for t in _edges(case["graph"], n, case["m"], seed))
    coin, rank, prob = (np.uint64(x) for x in _keys(seed))
    if case["model"] == "uniform":
        thr = np.full(src.shape, int(math.ldexp(case["p"], 64)) - 1, np.uint64)
    elif case["model"] == "wc":
        thr = np.uint64(M64) // np.bincount(dst.astype(np.int64), minlength=n).astype(np.uint64)[dst.astype(np.int64)]
    else:
        cls = np.array([int(math.ldexp(q, 64)) - 1 for q in (0.1, 0.01, 0.001)], np.uint64)
        thr = cls[(_fmix(prob ^ ((src << np.uint64(32)) | dst)) % np.uint64(3)).astype(np.int64)]
    state = _fmix(coin ^ ((src << np.uint64(32)) | dst))
    tails, heads = [], []
    for i in range(l):
        live = _fmix(state + _G * np.uint64(i + 1)) <= thr
        tails.append(src[live].astype(np.int64) * l + i)
        heads.append(dst[live].astype(np.int64) * l + i)
    tails, heads = torch.from_numpy(np.concatenate(tails)), torch.from_numpy(np.concatenate(heads))
    own = _fmix(rank + _G * np.arange(n * l, dtype=np.uint64))
    order = np.argsort(own)
    place = torch.empty(n * l, dtype=torch.int64)  # ranks as positions of the rank order
    place[torch.from_numpy(order)] = torch.arange(n * l)

    def bottom(owner, value, groups):
        key = torch.unique(owner * (n * l + 1) + value)
        owner, value = key // (n * l + 1), key % (n * l + 1)
        first = torch.searchsorted(owner, torch.arange(groups))
        at = torch.arange(owner.shape[0]) - first[owner]
        keep = at < k
        return owner[keep], value[keep]

    po, pv = torch.arange(n * l), place
    heads, by_head = torch.sort(heads)
    tails = tails[by_head]
    while True:
        lo = torch.searchsorted(heads, po)
        cnt = torch.searchsorted(heads, po, right=True) - lo
        rep = torch.repeat_interleave(torch.arange(po.shape[0]), cnt)
        e = torch.arange(rep.shape[0]) - torch.repeat_interleave(torch.cumsum(cnt, 0) - cnt, cnt) + lo[rep]
        no, nv = bottom(torch.cat([po, tails[e]]), torch.cat([pv, pv[rep]]), n * l)
        if no.shape == po.shape and torch.equal(no, po) and torch.equal(nv, pv):
            break
        po, pv = no, nv
    owner, value = bottom(po // l, pv, n)
    return owner.numpy(), own[order[value.numpy()]], k


def _plain_query(sketch, seeds, l):
    owner, ranks, k = sketch
    best = {}
    for u in seeds:
        x = ranks[np.searchsorted(owner, u):np.searchsorted(owner, u, side="right")]
        full = x.shape[0] == k
        tau = int(x[-1]) if full else 1 << 64
        for z in (x[:-1] if full else x).tolist():
            best[z] = max(best.get(z, 0), tau)
    return math.fsum(2.0 ** 64 / t for t in best.values()) / l


def exact(case, seed):
    small = case["n"] * case["l"] <= 1 << 18 and case["m"] * case["l"] <= 1 << 22 and case["ranks"] == "uniform"
    if not small or case["op"] not in ("query", "query_batch"):
        return None  # whole numbers, or too large for a plain computation
    with np.errstate(over="ignore"):
        sketch = _plain_sketches(case, seed)
    if case["op"] == "query":
        chosen = np.random.default_rng(seed).choice(case["n"], case["seeds"], replace=False)
        return _plain_query(sketch, chosen.tolist(), case["l"])
    off, flat = _query_sets(case["n"], case["queries"], seed)
    at = off.astype(np.int64)
    return np.array([_plain_query(sketch, flat[a:b].tolist(), case["l"]) for a, b in zip(at, at[1:])])
