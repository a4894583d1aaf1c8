"""Cases for timing the framework through its public entry points: what a user of the influence
minimization library has it do, from one small Alg. 2 call to a greedy run on a graph larger than
the L2 cache. The graphs are the families of the repository's workloads (directed Chung-Lu and
R-MAT; weighted-cascade, trivalency and linear-threshold weights) at their sizes and in between.

    listed()            the cases
    draw(rng)           one more case of the same ranges
    prepare(case, seed) what a program holds before the call: loaded graphs, seed sets, buffers
    run(state)          one call (or one burst of requests), and its results
    work(case)          bytes and integer operations one pass cannot do without
    exact(case, seed)   the results of a small case, recomputed in numpy
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2302_13529_gb300 import imin
from paper_2302_13529_gb300 import workloads as W

RMAT = "rmat"
CHUNG_LU = "chung-lu"


def listed():
    return [
        # One Alg. 2 call with few samples on a small graph, counters left on the device: the
        # latency a program pays that calls the estimator in its own loop.
        _case("estimate-small", "estimate", CHUNG_LU, 2_000, 10_000, "wc", seeds=10, theta=256),
        # AdvancedGreedy on the small workload (2,000 vertices, b = 10, theta = 10^4): launches count.
        _case("greedy-small", "greedy", CHUNG_LU, 2_000, 10_000, "wc", seeds=10, b=10, theta=10_000),
        # Alg. 2 with blockers on an odd-sized trivalency graph, host output: many tiny cascades
        # (the graph of the sweep over the number of sampled graphs).
        _case("estimate-blocked-odd", "estimate", CHUNG_LU, 100_003, 999_983, "tr", seeds=10, blocked=7,
              theta=100_000, host=True),
        # The headline: AdvancedGreedy on R-MAT 2^17 / 2^20, weighted cascade, |S| = 50, b = 50.
        _case("greedy-mid", "greedy", RMAT, 1 << 17, 1 << 20, "wc", seeds=50, b=50, theta=100_000),
        # GreedyReplace under trivalency (b = 20, |S| = 10): heavy-tailed cascades of up to tens of
        # thousands of vertices, where dominators weigh as much as the search.
        _case("replace-mid-tr", "replace", RMAT, 1 << 17, 1 << 20, "tr", seeds=10, b=20, theta=10_000),
        # The first rounds of AdvancedGreedy on R-MAT 2^22 / 2^26, |S| = 200: a 528 MB graph.
        _case("greedy-large", "greedy", RMAT, 1 << 22, 1 << 26, "wc", seeds=200, b=4, theta=100_000),
        # One batched call over many independent trivalency queries of all sizes (10^3 to 2*10^5
        # vertices), as an evaluation over many graphs makes it.
        _case("batch", "batch", CHUNG_LU, 1_000, 5_000, "tr", seeds=100, b=5, theta=20_000, queries=48),
        # The evaluation of a blocker set: 10^5 simulated cascades on the mid graph.
        _case("spread-mid", "spread", RMAT, 1 << 17, 1 << 20, "wc", seeds=50, blocked=50, theta=100_000),
        # The triggering model: AdvancedGreedy on linear-threshold samples of the mid graph.
        _case("greedy-mid-lt", "greedy", RMAT, 1 << 17, 1 << 20, "lt", seeds=50, b=5, theta=20_000),
        # BaselineGreedy, the comparison algorithm that simulates every candidate.
        _case("baseline-small", "baseline", CHUNG_LU, 2_000, 10_000, "wc", seeds=10, b=2, theta=2_000),
        # Alg. 2 for a caller that must not allocate, on a ragged graph near its size limit.
        _case("estimate-noalloc", "noalloc", CHUNG_LU, 50_021, 400_009, "wc", seeds=50, blocked=11, theta=10_000),
        # A burst of requests of both drivers, different sizes, through the request server.
        _case("serving", "serving", RMAT, 1 << 17, 1 << 20, "wc", seeds=500, b=20, theta=30_000, queries=8),
    ]


def _case(name, op, family, n, m, probs, *, seeds, theta, b=0, blocked=0, host=False, queries=0):
    c = dict(op=op, family=family, n=n, m=m, probs=probs, seeds=seeds, theta=theta, b=b, blocked=blocked,
             host=host, queries=queries)
    return dict(c, name=name) if name else c


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["estimate", "greedy", "greedy", "replace", "batch", "spread", "baseline", "noalloc", "serving"])
    family = rng.choice([CHUNG_LU, RMAT])
    if op in ("batch", "serving"):
        family = CHUNG_LU if op == "batch" else RMAT
    if op == "baseline":
        family = CHUNG_LU
        n = _log_int(rng, 300, 2_000)
    elif op == "batch":
        n = 1_000
    elif family == RMAT:  # a power of two
        n = 1 << rng.randint(14 if op == "serving" else 11, 16 if op == "noalloc" else 17 if op == "serving" else 20)
    else:
        n = _log_int(rng, 1_000, 65_536 if op == "noalloc" else 200_000)
    probs = "tr" if op == "batch" else rng.choice(["wc", "wc", "tr", "lt"])
    if family == RMAT and probs == "tr":
        # huge cascades: within the limits of the entry points that have no whole-graph fallback
        n = min(n, 1 << 17)
        probs = "wc" if op == "noalloc" else probs
    m = int(n * rng.uniform(4.0, 8.0 if probs == "tr" or family == RMAT else 20.0))
    seeds = min(_log_int(rng, 5, 200), n // 20)
    b = rng.randint(1, 20) if op in ("greedy", "replace", "batch", "serving") else 2 if op == "baseline" else 0
    queries = rng.randint(4, 48) if op == "batch" else rng.randint(2, 8) if op == "serving" else 0
    theta = 2_000 if op == "baseline" else _log_int(rng, 100, 100_000)
    c = _case(None, op, family, n, m, probs, seeds=seeds, theta=theta, b=b,
              blocked=rng.randint(0, min(60, n // 10)) if op in ("estimate", "spread", "noalloc") else 0,
              host=op == "estimate" and rng.random() < 0.3, queries=queries)
    # a drawn case examines at most as many edges as the headline
    most = 0.5 * _edges(listed()[3])
    while _edges(c) > most and c["theta"] > 100:
        c["theta"] = max(100, c["theta"] // 2)
    return c


def _edges(case):
    """Out-edges of reached vertices over all samples of one pass: the mean cascade of the family
    (measured at the listed sizes, scaled with the square root of the edges) times the samples."""
    per_seed = (0.7 if case["probs"] == "tr" else 7.0) * case["m"] / case["n"]
    if case["family"] == RMAT:
        # trivalency on the heavy-tailed graph is near its threshold: few samples, huge cascades
        per_seed = (10_000.0 if case["probs"] == "tr" else 110.0) * math.sqrt(case["m"] / (1 << 20))
    rounds = {"greedy": case["b"], "replace": 1.3 * case["b"], "batch": case["b"], "serving": 0.6 * case["b"],
              "baseline": case["b"] * float(case["n"])}.get(case["op"], 1.0)
    if case["queries"]:
        rounds *= 0.5 * case["queries"]
    if case["op"] == "batch":  # log-uniform sizes; the trivalency cascades stay near their seeds
        per_seed = 25.0
    return per_seed * case["seeds"] * case["theta"] * max(rounds, 1.0)


def work(case):
    """Bytes: every graph read once, every output written once. Operations: one Philox4x32-10 draw
    (10 rounds of 2 wide multiplications, 4 xors and 2 key additions) per 4 examined edges, and the
    comparison of each edge's word; a linear-threshold edge draws its target's word instead."""
    graphs = 1
    n, m = case["n"], case["m"]
    if case["op"] == "batch":  # mean of the log-uniform sizes, mean degree 12.5
        n, graphs = 37_000, case["queries"]
        m = 462_500
    bytes_ = graphs * (4.0 * (n + 1) + (12.0 if case["probs"] == "lt" else 8.0) * m) + 4.0 * case["seeds"]
    bytes_ += 8.0 * n if case["op"] in ("estimate", "noalloc") else 4.0 * case["b"] * max(case["queries"], 1)
    per_edge = 82.0 if case["probs"] == "lt" else 21.0
    return {"bytes": bytes_, "flops": _edges(case) * per_edge}


# ---- inputs ----------------------------------------------------------------------------------

def _rmat_gpu(n, m, seed):
    """R-MAT (0.57, 0.19, 0.19, 0.05) on the GPU: exactly m distinct non-loop edges, vertices
    relabelled at random. Returns device (row_ptr, col)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    scale = n.bit_length() - 1
    a, b, c, _ = W.RMAT_ABCD
    keys = torch.empty(0, dtype=torch.int64, device="cuda")
    while keys.numel() < m:
        k = int(1.15 * (m - keys.numel())) + 1024
        src = torch.zeros(k, dtype=torch.int64, device="cuda")
        dst = torch.zeros(k, dtype=torch.int64, device="cuda")
        for _ in range(scale):
            r = torch.rand(k, generator=g, device="cuda")
            src = src * 2 + (r >= a + b)
            dst = dst * 2 + (((r >= a) & (r < a + b)) | (r >= a + b + c))
        new = (src * n + dst)[src != dst]
        keys = torch.unique(torch.cat([keys, new]))
        del src, dst, r, new
    keep = torch.randperm(keys.numel(), generator=g, device="cuda")[:m]
    keys = keys[keep]
    label = torch.randperm(n, generator=g, device="cuda")
    keys = torch.sort(label[keys // n] * n + label[keys % n]).values
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.cumsum(torch.bincount(keys // n, minlength=n), 0)
    return row_ptr.to(torch.int32), (keys % n).to(torch.int32)


def _graph(family, n, m, probs, seed):
    """(n, row_ptr, col, weights) of one graph, as int32 / int32 / uint32 arrays."""
    if family == RMAT:
        row_ptr, col = _rmat_gpu(n, m, seed)
        if probs == "tr":
            g = torch.Generator(device="cuda").manual_seed(seed + 1)
            t = torch.tensor(W.TR_THRESHOLDS.astype(np.int64), device="cuda")
            w = t[torch.randint(0, 3, (m,), generator=g, device="cuda")]
        else:
            d = torch.bincount(col.long(), minlength=n)[col.long()]
            w = (1 << 32) // d - 1 if probs == "lt" else ((1 << 32) - 1) // d
        low = torch.where(w >= 1 << 31, w - (1 << 32), w).to(torch.int32)  # the same 32 bits
        return n, row_ptr, col, low.view(torch.uint32)
    row_ptr, col = W.chung_lu(n, m, 2.1, seed)
    if probs == "tr":
        w = W.tr_thresholds(m, seed + 1)
    else:
        w = W.lt_wc_weights(col, n) if probs == "lt" else W.wc_thresholds(col, n)
    return n, row_ptr, col, w


def _load(g, probs):
    return imin.GraphHandle(*g, model="lt" if probs == "lt" else "ic")


class _Serving(imin.Server):
    """A server that is closed with the state that holds it."""

    def __del__(self):
        self.close()


def _batch_items(case, seed):
    rng = np.random.default_rng(seed)
    items = []
    for _ in range(case["queries"]):
        n = int(math.exp(rng.uniform(math.log(1e3), math.log(2e5))))
        m = int(round(n * rng.uniform(5.0, 20.0)))
        gh = _load(_graph(CHUNG_LU, n, m, "tr", int(rng.integers(1 << 31))), "tr")
        seeds = W.uniform_seeds(n, int(rng.integers(5, case["seeds"] + 1)), int(rng.integers(1 << 31)))
        items.append((gh, seeds, case["b"], case["theta"], W.query_key(int(rng.integers(1 << 31)))))
    return items


def prepare(case, seed):
    op = case["op"]
    if op == "batch":
        return {"op": op, "items": _batch_items(case, seed)}
    g = _graph(case["family"], case["n"], case["m"], case["probs"], seed)
    gh = _load(g, case["probs"])
    if op == "serving":
        # both drivers, mixed budgets, |S| and theta uniform up to the case's
        rng = np.random.default_rng(seed)
        reqs = []
        for i in range(case["queries"]):
            k = int(rng.integers(min(10, case["seeds"]), case["seeds"] + 1))
            seeds = W.uniform_seeds(case["n"], k, int(rng.integers(1 << 30)))
            reqs.append((i % 2, gh, seeds, max(1, case["b"] * (4 - i % 4) // 4),
                         int(rng.integers((case["theta"] + 2) // 3, case["theta"] + 1)), int(rng.integers(1 << 62))))
        return {"op": op, "server": _Serving(), "reqs": reqs}
    ids = W.uniform_seeds(case["n"], case["seeds"] + case["blocked"], seed + 7)
    st = {"op": op, "graph": gh, "seeds": ids[:case["seeds"]], "blocked": ids[case["seeds"]:],
          "theta": case["theta"], "b": case["b"], "key": W.query_key(seed + 11), "out": None}
    if op in ("estimate", "noalloc") and not case["host"]:
        st["out"] = torch.zeros(case["n"], dtype=torch.uint64, device="cuda")
    return st


# ---- one pass --------------------------------------------------------------------------------

def run(st):
    op = st["op"]
    if op == "batch":
        return imin.batch_advanced_greedy(st["items"])
    if op == "serving":
        srv = st["server"]
        tickets = [(srv.submit(*r), r[3]) for r in st["reqs"]]
        return [_padded(srv.wait(t, b)[0], b) for t, b in tickets]
    g, seeds, key, theta = st["graph"], st["seeds"], st["key"], st["theta"]
    if op == "estimate":
        return imin.estimate_decrease(g, seeds, st["blocked"], theta, key, out=st["out"])
    if op == "noalloc":
        return imin.estimate_decrease_noalloc(g, seeds, st["blocked"], theta, key, out=st["out"])
    if op == "spread":
        return imin.estimate_spread(g, seeds, st["blocked"], theta, key)
    driver = {"greedy": imin.advanced_greedy, "replace": imin.greedy_replace, "baseline": imin.baseline_greedy}[op]
    found = driver(g, seeds, st["b"], theta, key)
    return [_padded(found, st["b"]), len(found)]


def _padded(found, b):
    """The blockers in an array of the budget's length (GreedyReplace may find fewer)."""
    out = np.full(b, -1, dtype=np.int32)
    out[:len(found)] = found
    return out


# ---- the results of a small case in numpy ----------------------------------------------------

def _philox(q, j, key):
    """Philox4x32-10 words [len(q), 4] at counters (q, j, 0, 0)."""
    lo = np.uint64(0xFFFFFFFF)
    x = [q.astype(np.uint64), np.full(len(q), j, np.uint64), np.zeros(len(q), np.uint64), np.zeros(len(q), np.uint64)]
    k = [key & 0xFFFFFFFF, key >> 32]
    for _ in range(10):
        p, r = np.uint64(0xD2511F53) * x[0], np.uint64(0xCD9E8D57) * x[2]
        x = [(r >> np.uint64(32)) ^ x[1] ^ np.uint64(k[0]), r & lo, (p >> np.uint64(32)) ^ x[3] ^ np.uint64(k[1]), p & lo]
        k = [(k[0] + 0x9E3779B9) & 0xFFFFFFFF, (k[1] + 0xBB67AE85) & 0xFFFFFFFF]
    return np.stack(x, 1)


def _reach(adj, start, without):
    """Vertices reached from start in the live graph without vertex `without`."""
    seen, todo = set(start), list(start)
    while todo:
        for v in adj.get(todo.pop(), ()):
            if v != without and v not in seen:
                seen.add(v)
                todo.append(v)
    return seen


def exact(case, seed):
    """The counters of one small independent-cascade Alg. 2 call: vertex u's is the number of
    vertices (u included) that the seeds no longer reach once u is deleted, summed over the samples."""
    if case["op"] not in ("estimate", "noalloc") or case["probs"] == "lt" or case["theta"] * case["m"] > 20_000_000:
        return None
    if case["family"] == RMAT or _edges(case) > 1e6:
        return None
    n, row_ptr, col, thr = _graph(case["family"], case["n"], case["m"], case["probs"], seed)
    ids = W.uniform_seeds(n, case["seeds"] + case["blocked"], seed + 7)
    seeds, shut = ids[:case["seeds"]].tolist(), np.zeros(n, bool)
    shut[ids] = True
    src = np.repeat(np.arange(n), np.diff(row_ptr))
    out = np.zeros(n, np.uint64)
    for j in range(case["theta"]):
        words = _philox(np.arange((len(col) + 3) // 4), j, W.query_key(seed + 11)).reshape(-1)[:len(col)]
        live = np.nonzero((words <= thr) & ~shut[col])[0]
        adj = {}
        for e in live.tolist():
            adj.setdefault(int(src[e]), []).append(int(col[e]))
        reached = _reach(adj, seeds, -1)
        for u in reached.difference(seeds):
            out[u] += np.uint64(len(reached) - len(_reach(adj, seeds, u)))
    return out
