"""The workloads this library is timed on, through its public calls.

Graphs, weights, suspects and walk seeds are synthetic and made on the GPU from one seed: R-MAT (a, b, c = 0.57, 0.19,
0.19) and directed Chung-Lu (gamma 2.1) edge lists with weighted-cascade or random LT weights, the classes and sizes of
bench.py and tests/.  `steps` (a throughput counter) is not among the outputs; everything else a call returns is.
"""
import math

import numpy as np
import torch

import paper_1702_05854_gb300 as hs

U32 = (1 << 32) - 1


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # The smallest call: a host loop that asks for the hits of a short attempt range and may not allocate.
        dict(name="static-4k", op="static", graph="chung-lu", n=16384, m=131072, weights="wc", sources=16, coin=False,
             attempts=4096),
        # The plain eSI query on a graph that fits the L2 cache (bench.py --workload c1).
        dict(name="fixed-edge-16k", op="fixed", graph="chung-lu", n=16384, m=131072, weights="wc", sources=16,
             coin=False, mode="edge", k=10, hits=200_000),
        # The paper's experimental query on its smallest graph: many suspects of random probability, nSI, stopping
        # rule (first point of bench.py --mode sweep).  Launches and round trips count.
        dict(name="stop-node-8k", op="stop", graph="rmat", n=1 << 13, m=5 << 13, weights="wc", sources=1000, coin=True,
             mode="node", k=100, eps=0.1),
        # nSI with unequal LT weights and few suspects: rare hits, short walks (bench.py --workload c2, tenth of its N).
        dict(name="fixed-node-1m-lt", op="fixed", graph="rmat", n=1 << 20, m=16 << 20, weights="lt", sources=100,
             coin=False, mode="node", k=100, hits=1_000_000),
        # The large eSI query with the stopping rule on a graph far beyond L2 (bench.py's headline, two scales down so
        # that its graph can be made for each seed).
        dict(name="stop-edge-16m", op="stop", graph="rmat", n=1 << 24, m=16 << 24, weights="wc", sources=1000,
             coin=False, mode="edge", k=1000, eps=0.1),
        # A served query: the graph is resident with a walk pool of the query's seed (bench.py --mode serve).
        dict(name="pool-edge-256k", op="pool", graph="rmat", n=1 << 18, m=16 << 18, weights="wc", sources=300,
             coin=False, mode="edge", k=300, eps=0.1, attempts=1 << 25),
        # What the spread is after an interdiction: the same stream on the graph without 1,000 edges.
        dict(name="spread-edge-4m", op="spread", graph="rmat", n=1 << 22, m=16 << 22, weights="wc", sources=1000,
             coin=False, mode="edge", removed=1000, hits=100_000),
        # A graph loaded from an edge list that lies on the GPU, and one query on it.
        dict(name="ingest-device-4m", op="ingest", graph="rmat", n=1 << 22, m=16 << 22, weights="wc", sources=4000,
             coin=False, form="edges", host=False, mode="edge", k=50, hits=10_000),
        # The same from pinned host arrays, the end-to-end path of bench.py.
        dict(name="ingest-host-1m", op="ingest", graph="rmat", n=1 << 20, m=16 << 20, weights="lt", sources=4000,
             coin=False, form="edges", host=True, mode="node", k=50, hits=10_000),
        # The ordered stream itself, for a program that does its own counting in buffers of its own: an odd number
        # of hits, coins.
        dict(name="stream-node-1m", op="stream", graph="rmat", n=1 << 20, m=16 << 20, weights="wc", sources=1000,
             coin=True, mode="node", hits=300_001),
        # Selection on a stream that is there already: greedy on one half, coverage of the picks on the other.
        dict(name="select-edge-4m", op="select", graph="rmat", n=1 << 22, m=16 << 22, weights="wc", sources=4000,
             coin=False, mode="edge", k=1000, hits=300_000),
        # Many small instances in one call (bench.py --mode batch with small graphs).
        dict(name="batch-32", op="batch", graph="chung-lu", count=32, n_min=1000, n_max=10000, coin=False, k=100,
             hits=20_000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the same calls over the sizes between the smallest and the largest above, odd ones among them."""
    op = rng.choice(["static", "fixed", "fixed", "stop", "stop", "pool", "spread", "ingest", "stream", "select",
                     "batch"])
    if op == "batch":
        return dict(op=op, graph="chung-lu", count=rng.randint(4, 32), n_min=1000, n_max=_log(rng, 2000, 10000),
                    coin=rng.random() < 0.3, k=_log(rng, 10, 200), hits=_log(rng, 2000, 20000))
    top = {"static": 1 << 20, "fixed": 1 << 20, "stop": 1 << 23, "pool": 1 << 18, "spread": 1 << 22, "ingest": 1 << 22,
           "stream": 1 << 20, "select": 1 << 21}[op]
    n = _log(rng, 2000, top)
    c = dict(op=op, graph=rng.choice(["rmat", "chung-lu"]), n=n, m=n * rng.randint(5, 16) + rng.randint(0, n),
             weights=rng.choice(["wc", "lt"]))
    # suspects: enough of them that a hit takes at most some ten thousand attempts
    c["sources"] = max(8, min(n // 8, _log(rng, max(1, n / 5000), max(2, n / 50))))
    c["coin"] = op != "static" and rng.random() < 0.4
    if op == "static":
        c.update(attempts=_log(rng, 256, 1 << 18))
        return c
    c["mode"] = rng.choice(["edge", "node"])
    if op in ("fixed", "spread", "stream", "select"):
        c["hits"] = _log(rng, 1000, 100_000)
    if op in ("fixed", "stop", "pool", "select"):
        c["k"] = _log(rng, 5, 1000)
    if op in ("stop", "pool"):
        c["eps"] = rng.choice([0.1, 0.2])
    if op == "pool":
        c["attempts"] = _log(rng, 1 << 20, 1 << 25)
    if op == "spread":
        c["removed"] = _log(rng, 1, 1000)
    if op == "ingest":
        c.update(k=_log(rng, 5, 100), form=rng.choice(["edges", "csr"]), host=rng.random() < 0.5, hits=_log(rng, 1000, 10_000))
    return c


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _rmat(n, m, gen):
    """R-MAT on the next power of two, folded onto [0, n)."""
    bits = max(1, (n - 1).bit_length())
    src = torch.zeros(m, dtype=torch.int32, device="cuda")
    dst = torch.zeros(m, dtype=torch.int32, device="cuda")
    for _ in range(bits):
        r = torch.rand(m, device="cuda", generator=gen)
        src.mul_(2).add_(r >= 0.57 + 0.19)
        dst.mul_(2).add_(((r >= 0.57) & (r < 0.57 + 0.19)) | (r >= 0.57 + 0.19 + 0.19))
        del r
    if n != 1 << bits:
        src = ((src.long() * n) >> bits).int()
        dst = ((dst.long() * n) >> bits).int()
    return src, dst


def _chung_lu(n, m, gen, gamma=2.1):
    w = torch.arange(1, n + 1, dtype=torch.float64, device="cuda") ** (-1.0 / (gamma - 1.0))
    cdf = torch.cumsum((w * (1 << 40)).long(), 0)  # whole numbers: the same sums in any order
    ends = []
    for _ in range(2):
        at = torch.searchsorted(cdf, torch.randint(int(cdf[-1]), (m,), device="cuda", generator=gen), right=True)
        ends.append(torch.randperm(n, device="cuda", generator=gen)[at].int())
    return ends


def _u32_bits(x):
    """int64 values below 2^32 as the int32 tensor of the same bits."""
    return torch.where(x > 0x7FFFFFFF, x - (1 << 32), x).int()


def _weights(kind, n, dst, gen):
    """uint32 in-weights as int64: weighted cascade, or uniform shares of a node in-sum U(0.5, 1)."""
    if kind == "wc":
        deg = torch.bincount(dst, minlength=n)
        return (U32 // deg.clamp_(min=1))[dst]
    x = torch.randint(1, 1 << 20, (dst.numel(),), device="cuda", generator=gen)
    total = torch.zeros(n, dtype=torch.int64, device="cuda").index_add_(0, dst, x)
    insum = (torch.rand(n, dtype=torch.float64, device="cuda", generator=gen) * 0.5 + 0.5).mul_(U32).long()
    return x * insum[dst] // total[dst]


def _edges(case, gen):
    make = _rmat if case["graph"] == "rmat" else _chung_lu
    src, dst = make(case["n"], case["m"], gen)
    return src, dst, _weights(case["weights"], case["n"], dst, gen)


def _suspects(n, count, coin, gen):
    """(suspects, increasing, and their probabilities or None), host arrays."""
    s = torch.randperm(n, device="cuda", generator=gen)[:count].sort().values.int().cpu().numpy()
    p = torch.randint(0, 1 << 32, (count,), device="cuda", generator=gen) if coin else None
    return s, None if p is None else p.cpu().numpy().astype(np.uint32)


def _removed(case, src, dst, sus, gen):
    """CSR ids of up to case["removed"] elements next to the suspects: their out-edges, or their out-neighbours."""
    flag = torch.zeros(case["n"], dtype=torch.bool, device="cuda")
    flag[torch.from_numpy(sus).cuda().long()] = True
    if case["mode"] == "node":
        ids = torch.unique(dst[flag[src]].long())
    else:
        ids = torch.nonzero(flag[src[torch.sort(dst, stable=True).indices]]).reshape(-1)
    return ids[torch.randperm(ids.numel(), device="cuda", generator=gen)[: case["removed"]]].sort().values.cpu().numpy()


def _query(case, sus, p, seed, **more):
    mode = hs.HSAW_NODE if case.get("mode") == "node" else hs.HSAW_EDGE
    rule = hs.HSAW_STOP_RULE if "eps" in case else hs.HSAW_FIXED_N
    return hs.Query(sources=sus, p_fixed=p, mode=mode, k=case.get("k", 1), sampling=rule, n_hsaw=case.get("hits", 0),
                    eps=case.get("eps", 0.1), seed=seed, **more)


def _to_csr(n, src, dst, w):
    order = torch.sort(dst, stable=True).indices
    row = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row[1:] = torch.cumsum(torch.bincount(dst, minlength=n), 0)
    return row, src[order], w[order]


def _batch_graphs(case, gen):
    got = []
    for _ in range(case["count"]):
        u = torch.rand(4, generator=gen, device="cuda").tolist()
        n = int(case["n_min"] * (case["n_max"] / case["n_min"]) ** u[0])
        c = dict(graph="chung-lu", n=n, m=int(n * (8 + 24 * u[1])), weights="wc")
        src, dst, w = _edges(c, gen)
        sus, p = _suspects(n, max(8, int(8 * (n / 64.0) ** u[2])), case["coin"], gen)
        got.append((c, src, dst, w, sus, p, "edge" if u[3] < 0.5 else "node"))
    return got


def prepare(case, seed):
    gen, op = _gen(seed), case["op"]
    if op == "batch":
        graphs, queries = [], []
        for i, (c, src, dst, w, sus, p, mode) in enumerate(_batch_graphs(case, gen)):
            graphs.append(hs.hsaw_graph_from_edges(c["n"], src, dst, _u32_bits(w)))
            queries.append(_query(dict(case, mode=mode), sus, p, seed + i))
        return dict(op=op, graphs=graphs, queries=queries)
    n = case["n"]
    src, dst, w = _edges(case, gen)
    sus, p = _suspects(n, case["sources"], case["coin"], gen)
    state = dict(op=op, n=n, query=_query(case, sus, p, seed), hits=case.get("hits", 0), k=case.get("k", 1))
    if op == "ingest":
        parts = (src, dst, w) if case["form"] == "edges" else _to_csr(n, src, dst, w)
        parts = [*parts[:2], _u32_bits(parts[2])]
        if case["host"]:
            parts = [t.cpu().pin_memory().numpy() for t in parts]
            parts[2] = parts[2].view(np.uint32)
        load = hs.hsaw_graph_from_edges if case["form"] == "edges" else hs.hsaw_graph_from_csr
        return dict(state, load=load, parts=parts)
    if op == "spread":
        state["removed"] = _removed(case, src, dst, sus, gen)
    state["graph"] = hs.hsaw_graph_from_edges(n, src, dst, _u32_bits(w))
    if op == "pool":
        state["graph"].build_walk_pool(seed, case["attempts"])
    elif op == "stream":
        h = case["hits"]
        state["keep"] = [torch.zeros(c, dtype=t, device="cuda") for c, t in (
            (h, torch.int64), (h + 1, torch.int64), (16 * h, torch.int32), (16 * h, torch.int32))]
    elif op == "select":
        state["walks"] = hs.hsaw_sample(state["graph"], state["query"], 0, case["hits"])
    elif op == "static":
        bits = np.zeros((n + 31) // 32, np.uint32)
        np.bitwise_or.at(bits, sus >> 5, np.uint32(1) << (sus & 31).astype(np.uint32))
        state.update(bits=torch.from_numpy(bits.view(np.int32)).cuda(), attempts=case["attempts"], seed=seed,
                     aid=torch.zeros(case["attempts"], dtype=torch.int64, device="cuda"),
                     len=torch.zeros(case["attempts"], dtype=torch.int32, device="cuda"))
    return state


# ------------------------------------------------------------------ one pass
RESULT = ("n_selected", "rounds_t", "hits", "attempts", "cov_R", "cov_Rprime", "hits_Rprime", "attempts_Rprime",
          "spread_base_est", "spread_reduction_est", "eps_t")


def _solved(ids, gains, r):
    return dict({f: r[f] for f in RESULT}, ids=ids, gains=gains)


def run(state):
    op = state["op"]
    if op in ("fixed", "stop", "pool"):
        return _solved(*hs.hsaw_solve(state["graph"], state["query"]))
    if op == "static":
        hits = hs.hsaw_sample_hits_static(state["graph"], state["bits"], state["seed"], 0, state["attempts"],
                                          state["aid"], state["len"])
        return dict(hits=hits, aid=state["aid"], len=state["len"])
    if op == "spread":
        spread, std_err = hs.hsaw_estimate_spread(state["graph"], state["query"], state["removed"])
        return dict(spread=spread, std_err=std_err)
    if op == "select":
        half = state["hits"] // 2
        mode, graph, walks = state["query"].mode, state["graph"], state["walks"]
        ids, gains = hs.hsaw_greedy(walks, graph, mode, 0, half, state["k"])
        return dict(ids=ids, gains=gains, cov=hs.hsaw_coverage(walks, mode, half, state["hits"] - half, ids))
    if op == "batch":
        done = hs.hsaw_solve_batch(state["graphs"], state["queries"])
        out = [_solved(ids, gains, r) for _, ids, gains, r in done]
        return dict({f: np.array([o[f] for o in out]) for f in RESULT}, status=np.array([d[0] for d in done]),
                    ids=np.concatenate([o["ids"] for o in out]), gains=np.concatenate([o["gains"] for o in out]))
    if op == "ingest":
        graph = state["load"](state["n"], *state["parts"])
        out = _solved(*hs.hsaw_solve(graph, state["query"]))
        graph.close()
        return out
    # stream: the first hits, and as many of their nodes and edges as the program has room for
    walks = hs.hsaw_sample(state["graph"], state["query"], 0, state["hits"])
    for keep, got in zip(state["keep"], walks.export_device()):
        room = min(keep.numel(), got.numel())
        keep[:room].copy_(got[:room])
    walks.close()
    return dict(zip(("aid", "node_off", "nodes", "edges"), state["keep"]))


# ------------------------------------------------------------------ what a pass cannot do without
PHILOX = 80  # integer operations of one Philox4x32-10 block


def _walk(case):
    """(attempts per hit, live-edge draws per attempt), about: means seen on these graph classes."""
    far = case["graph"] == "rmat" and case["n"] >= 1 << 17
    per = 2.5 if case["weights"] == "lt" else (40.0 if far else 10.0)
    share = case["sources"] / case["n"] * (0.5 if case["coin"] else 1.0)
    return 1.0 / min(0.9, per * share), per


def _rule_hits(case):
    """Hits the stopping rule takes, about: R and R' of its usual last round."""
    elements = case["m"] if case["mode"] == "edge" else case["n"]
    most = 3072 if _walk(case)[1] > 10.0 else 128  # short walks share more elements: fewer rounds
    return most * (0.1 / case["eps"]) ** 2 * math.log(elements) * math.sqrt(case["k"])


def work(case):
    """Bytes: each live-edge draw reads one 32-byte record of its own, each walk element of the hits is written and
    read once (counting), inputs and outputs move once.  Operations: the generator's."""
    op = case["op"]
    if op == "batch":
        n = math.sqrt(case["n_min"] * case["n_max"])
        one = dict(op="fixed", graph="chung-lu", n=n, m=20 * n, weights="wc", sources=0.02 * n, coin=case["coin"], mode="edge",
                   k=case["k"], hits=case["hits"])
        w = work(one)
        return {f: v * case["count"] for f, v in w.items()}
    per_hit, draws = _walk(case)
    if op == "static":
        return {"bytes": case["attempts"] * draws * 32 + case["n"] / 8 + case["attempts"] / per_hit * 12,
                "flops": PHILOX * case["attempts"] * draws}
    hits = _rule_hits(case) if op in ("stop", "pool") else case["hits"]
    out = hits * (16 + 8 * draws)
    attempts = hits * per_hit
    if op == "select":
        return {"bytes": hits * draws * 8.0, "flops": hits * draws}
    if op == "pool":
        return {"bytes": attempts / 8 + hits * draws * 32 + out, "flops": PHILOX * hits * draws}
    total = attempts * draws * 32 + out
    if op == "ingest":
        total += case["m"] * (12 + 4 + 32)
    return {"bytes": total, "flops": PHILOX * attempts * draws}


# ------------------------------------------------------------------ the same numbers in 64 bits
def _mulhilo(a, b):
    lo = a * b  # the low 64 bits, as int64
    return (lo >> 32) & U32, lo & U32


def _philox(c0, c1, c2, c3, seed):
    """Words 0 and 1 of Philox4x32-10 (Salmon et al., SC'11) on int64 tensors."""
    k0, k1 = seed & U32, (seed >> 32) & U32
    for _ in range(10):
        h0, l0 = _mulhilo(c0, 0xD2511F53)
        h1, l1 = _mulhilo(c2, 0xCD9E8D57)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & U32, (k1 + 0xBB67AE85) & U32
    return c0, c1


class _World:
    """Live-edge worlds of one query in plain int64 torch."""

    def __init__(self, case, seed, src, dst, w, sus, p, removed=None):
        self.n, self.seed = case["n"], seed
        order = torch.sort(dst, stable=True).indices
        d = dst[order].long()
        self.src = src[order].long()
        run = torch.cumsum(w[order], 0)
        deg = torch.bincount(d, minlength=self.n)
        first = torch.cumsum(deg, 0) - deg
        base = torch.where(first > 0, run[(first - 1).clamp(min=0)], torch.zeros_like(first))
        thr = run - base[d]
        self.keys = (d << 32) | thr
        last = (first + deg - 1).clamp(min=0)
        self.insum = torch.where(deg > 0, thr[last], torch.zeros_like(deg))
        self.p = torch.zeros(self.n, dtype=torch.int64, device="cuda")
        s = torch.from_numpy(sus).cuda().long()
        self.p[s] = U32 if p is None else torch.from_numpy(p.astype(np.int64)).cuda()
        self.sus = torch.zeros(self.n, dtype=torch.bool, device="cuda")
        self.sus[s] = True
        self.node = case.get("mode") == "node"
        self.gone = None
        if removed is not None:
            self.gone = torch.zeros(self.n if self.node else src.numel(), dtype=torch.bool, device="cuda")
            self.gone[torch.from_numpy(removed).cuda()] = True

    def start(self, a):
        z = torch.zeros_like(a)
        return (_philox(a & U32, a >> 32, z, z + 1, self.seed)[0] * self.n) >> 32

    def step(self, a, v):
        """(hit, in-edge or -1) of node v in attempt a."""
        z = torch.zeros_like(a)
        x0, x1 = _philox(a & U32, a >> 32, v, z, self.seed)
        hit = self.sus[v] & ((self.p[v] == U32) | (x1 < self.p[v]))
        e = torch.searchsorted(self.keys, (v << 32) | x0, right=True)
        e = torch.where(x0 < self.insum[v], e, torch.full_like(e, -1))
        return hit, e

    def hits(self, first, count):
        """Attempt ids of the hits among [first, first + count), increasing."""
        a = torch.arange(first, first + count, device="cuda")
        v = self.start(a)
        if self.gone is not None and self.node:
            keep = ~self.gone[v]
            a, v = a[keep], v[keep]
        old, at, power, found = v, 0, 1, []
        while a.numel():
            hit, e = self.step(a, v)
            found.append(a[hit])
            go = ~hit & (e >= 0)
            a, e, old = a[go], e[go], old[go]
            u = self.src[e]
            go = u != old  # Brent: a revisit of the kept node closes the cycle
            if self.gone is not None:
                go &= ~self.gone[u if self.node else e]
            a, v, old = a[go], u[go], old[go]
            at += 1
            if at == power:
                old, at, power = v, 0, power * 2
        return torch.sort(torch.cat(found)).values if found else a

    def walks(self, a):
        """(walk index, element) of every walk element of hits a."""
        idx, v = torch.arange(a.numel(), device="cuda"), self.start(a)
        where, what = [], []
        if self.node:
            where.append(idx)
            what.append(v)
        while a.numel():
            hit, e = self.step(a, v)
            go = ~hit
            idx, a, e = idx[go], a[go], e[go]
            v = self.src[e]
            where.append(idx)
            what.append(v if self.node else e)
        return torch.cat(where), torch.cat(what)

    def first_hits(self, count, block=1 << 22):
        """Attempt ids of the first `count` hits."""
        got, have, at = [], 0, 0
        while have < count:
            got.append(self.hits(at, block))
            have, at = have + got[-1].numel(), at + block
        return torch.cat(got)[:count]


def _greedy(where, what, walks, k):
    """(ids, coverage) of the greedy: largest gain, smallest id; without a gain, the smallest ids not taken yet."""
    left, ids, cov = torch.ones(walks, dtype=torch.bool, device="cuda"), [], 0
    for _ in range(k):
        live = left[where]
        if not bool(live.any()):
            break
        u, c = torch.unique(what[live], return_counts=True)
        best = int(u[int(torch.nonzero(c == c.max())[0])])
        ids.append(best)
        cov += int(c.max())
        left[where[what == best]] = False
    taken, x = set(ids), 0
    while len(ids) < k:
        if x not in taken:
            ids.append(x)
        x += 1
    return ids, cov


def _estimates(world, case):
    """The result's floating fields, from the paper's formulas (Alg. 4-9)."""
    n, k = case["n"], case["k"]
    if "hits" in case:
        a = world.first_hits(case["hits"])
        _, cov = _greedy(*world.walks(a), a.numel(), k)
        tried = int(a[-1]) + 1
        return n * float(case["hits"]) / tried, n * float(cov) / tried, math.nan
    eps, delta, size = case["eps"], 1.0 / n, case["n"] if world.node else case["m"]
    ln_c = math.lgamma(size + 1.0) - math.lgamma(k + 1.0) - math.lgamma(size - k + 1.0)
    a1 = 2.0 + 2.0 * eps / 3.0
    n_max = (2.0 - 1.0 / math.e) ** 2 * a1 * size * (math.log(6.0 / delta) + ln_c) / (k * eps * eps)
    t_max = max(1.0, math.ceil(math.log2(2.0 * n_max / (a1 * math.log(3.0 / delta) / (eps * eps)))))
    lam = a1 * math.log(3.0 * t_max / delta) / (eps * eps)
    et, t = math.nan, 0
    while True:
        t += 1
        half = math.ceil(lam) << (t - 1)
        last = half >= n_max or t >= t_max
        if half < 1.0 + (1.0 + eps) * lam and not last:
            continue
        a = world.first_hits(2 * half)
        ids, c = _greedy(*world.walks(a[:half]), half, k)
        where, what = world.walks(a[half:])
        picked = torch.isin(what, torch.tensor(ids, device="cuda"))
        cp = int(torch.unique(where[picked]).numel())
        ok = False
        if cp >= 1.0 + (1.0 + eps) * lam:
            gap, scale = 1.0 - 1.0 / math.e - eps, 2.0 ** (t - 1)
            e1 = c / cp - 1.0
            e2 = eps * math.sqrt(half * (1.0 + eps) / (scale * cp))
            e3 = eps * math.sqrt(half * (1.0 + eps) * gap / ((1.0 + eps / 3.0) * scale * cp))
            et = (e1 + e2 + e1 * e2) * gap + (1.0 - 1.0 / math.e) * e3
            ok = et <= eps
        if ok or last:
            tried = int(a[-1]) + 1
            return n * float(2 * half) / tried, n * float(c + cp) / tried, et


def exact(case, seed):
    """The floating results (estimates); the other outputs are whole numbers."""
    op = case["op"]
    if op not in ("fixed", "stop", "pool", "spread"):
        return None
    per_hit, draws = _walk(case)
    hits = case.get("hits") or _rule_hits(case)
    if hits * per_hit * draws > 2.5e9 or (op != "spread" and (hits * case["k"] > 2.5e8 or case["n"] > 1 << 15)):
        return None  # minutes in plain torch
    gen = _gen(seed)
    src, dst, w = _edges(case, gen)
    sus, p = _suspects(case["n"], case["sources"], case["coin"], gen)
    removed = _removed(case, src, dst, sus, gen) if op == "spread" else None
    world = _World(case, seed, src, dst, w, sus, p, removed)
    if op == "spread":
        tried = int(world.first_hits(case["hits"], 1 << 23)[-1]) + 1
        f = case["hits"] / tried
        return dict(spread=case["n"] * float(case["hits"]) / tried,
                    std_err=case["n"] * math.sqrt(f * (1.0 - f) / tried))
    base, reduction, et = _estimates(world, case)
    return dict({f: None for f in RESULT}, spread_base_est=base, spread_reduction_est=reduction, eps_t=et, ids=None,
                gains=None)
