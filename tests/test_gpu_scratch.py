"""Scratch device memory: what calls hold at most, and what is left when an allocation fails.

Counted by an allocator of the tests' own (hsaw_set_allocator) over torch's caching allocator; failures are made on the
host, by that allocator or by the library's own hook.
"""
import threading

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
hs = pytest.importorskip("paper_1702_05854_gb300")

MB = 1 << 20


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.init()


class Scratch:
    """Installs an allocator that counts the bytes held and refuses what `refuse(nbytes, held)` says."""

    def __init__(self, refuse=lambda nbytes, held: False):
        self.live, self.held, self.peak, self.asked, self.refuse = {}, 0, 0, 0, refuse
        self.lock = threading.Lock()

    def alloc(self, nbytes, stream):
        with self.lock:
            self.asked += 1
            if self.refuse(nbytes, self.held):
                return 0
            p = torch.cuda.caching_allocator_alloc(nbytes, stream=stream)
            self.live[p] = nbytes
            self.held += nbytes
            self.peak = max(self.peak, self.held)
            return p

    def release(self, ptr, stream):
        with self.lock:
            self.held -= self.live.pop(ptr)
            torch.cuda.caching_allocator_delete(ptr)

    def __enter__(self):
        hs.hsaw_set_allocator(self.alloc, self.release)
        return self

    def __exit__(self, *exc):
        torch.cuda.synchronize()
        hs.hsaw_set_allocator()


def test_server_budget_bounds_scratch():
    """Queries of few walks on 2^24 edges: the counts by edge id, the slab and the sampler's records, not the walks, are
    what they hold; together they stay within the budget."""
    d = synth.workload_rmat(20, "wc", 1000, 50, "edge")
    g = hs.hsaw_graph_from_edges(d["n"], d["src"], d["dst"], d["w"])
    queries = [hs.Query(sources=d["sources"], mode=hs.HSAW_EDGE, k=50, n_hsaw=2000, seed=s) for s in range(48)]
    alone = [hs.hsaw_solve(g, q) for q in queries]
    budget = 700 * MB
    with Scratch() as a:
        srv = hs.Server([g], mem_budget=budget, workers=8)
        tickets = [srv.submit(0, q) for q in queries]
        got = [srv.poll(t) for t in tickets]
        srv.close()
        assert 128 * MB < a.peak <= budget, a.peak / MB
    for (ids, gains, r), (ids2, gains2, r2, *_) in zip(alone, got):
        assert np.array_equal(ids, ids2) and np.array_equal(gains, gains2) and r["attempts"] == r2["attempts"]


def test_server_takes_what_its_walks_fit():
    """A query whose walks fit the budget is served, alone, though its scratch does not."""
    d = synth.workload_rmat(20, "wc", 1000, 50, "edge")
    g = hs.hsaw_graph_from_edges(d["n"], d["src"], d["dst"], d["w"])
    srv = hs.Server([g], mem_budget=80 * MB, workers=2)
    q = hs.Query(sources=d["sources"], mode=hs.HSAW_EDGE, k=50, n_hsaw=2000, seed=1)
    ids, gains = hs.hsaw_solve(g, q)[:2]
    for t in [srv.submit(0, q) for _ in range(4)]:
        got = srv.poll(t)
        assert np.array_equal(got[0], ids) and np.array_equal(got[1], gains)
    srv.close()


def test_scratch_while_no_attempt_hits():
    """One suspect among 2^25 isolated nodes: launches grow to tens of millions of attempts before the first hit, and have
    room for the few hits that can be expected, not for one an attempt (8 bytes each: 268 MB and more)."""
    n = 1 << 25
    one = np.zeros(1, np.int32)
    g = hs.hsaw_graph_from_edges(n, one, one + 1, np.ones(1, np.uint32))
    og = oracle.Graph(n, one, one + 1, np.ones(1, np.uint32))
    sources = np.array([12_345_678], np.int32)
    with Scratch() as a:
        ids, gains, r = hs.hsaw_solve(g, hs.Query(sources=sources, mode=hs.HSAW_NODE, k=1, n_hsaw=2, seed=8))
        assert a.peak < 192 * MB, a.peak / MB
    st = oracle.Stream(oracle.Query(og, sources, seed=8)).extend_threads(2, threads=8)
    aid = st.export().aid
    assert r["attempts"] == aid[1] + 1 and r["attempts"] > 1 << 24 and ids[0] == sources[0] and gains[0] == 2


def test_walks_handle_keeps_no_checkpoints():
    """What a handle holds: its walks and the sampler's records of one launch of 2^20 attempts (8 bytes each)."""
    d = synth.workload_c1()
    g = hs.hsaw_graph_from_edges(d["n"], d["src"], d["dst"], d["w"])
    with Scratch() as a:
        w = hs.hsaw_sample(g, hs.Query(sources=d["sources"], seed=4), 0, 1000)
        i = w.info()
        walks = 20 * i["count"] + 8 + 8 * i["total_nodes"]  # ids, lengths, offsets; nodes and edges
        assert a.held <= 2 * walks + (8 << 20) + 2 * MB, (a.held / MB, walks / MB)
        w.close()
        assert not a.live


def test_injected_failure_reaches_the_caller():
    """The n-th allocation fails as if memory were out, and the call with it, the first too."""
    d = synth.workload_c1()
    g = hs.hsaw_graph_from_edges(d["n"], d["src"], d["dst"], d["w"])
    q = hs.Query(sources=d["sources"], mode=hs.HSAW_EDGE, k=10, n_hsaw=1000, seed=4)
    walks = hs.hsaw_sample(g, q, 0, 1000)
    calls = [lambda: hs.hsaw_solve(g, q), lambda: hs.hsaw_estimate_spread(g, q, [3]),
             lambda: hs.hsaw_greedy(walks, g, hs.HSAW_EDGE, 0, 1000, 10), lambda: hs.hsaw_sample(g, q, 0, 1000)]
    try:
        for call in calls:
            for n in (1, 2, 3):
                hs.hsaw_debug_fail_alloc_after(n)
                with pytest.raises(hs.HsawError) as e:
                    call()
                assert e.value.status == -4
    finally:
        hs.hsaw_debug_fail_alloc_after(0)
        walks.close()


def test_nothing_is_held_after_a_failed_call():
    """Allocations of a call refused from the n-th on, for every n, with and without room for the slab: the call ends
    with HSAW_E_NOMEM and gives everything back."""
    d = synth.workload_c1()
    g = hs.hsaw_graph_from_edges(d["n"], d["src"], d["dst"], d["w"])
    kw = dict(sources=d["sources"], mode=hs.HSAW_EDGE, seed=4)
    fixed = hs.Query(k=10, n_hsaw=1000, **kw)
    walks = hs.hsaw_sample(g, fixed, 0, 1000)
    calls = [lambda: hs.hsaw_solve(g, fixed), lambda: hs.hsaw_solve(g, hs.Query(k=5, sampling=hs.HSAW_STOP_RULE, eps=0.4, **kw)),
             lambda: hs.hsaw_greedy(walks, g, hs.HSAW_EDGE, 0, 1000, 10), lambda: hs.hsaw_histogram(walks, hs.HSAW_NODE, 0, 1000),
             lambda: hs.hsaw_coverage(walks, hs.HSAW_EDGE, 0, 1000, [3, 5]), lambda: hs.hsaw_estimate_spread(g, fixed, [3]),
             lambda: hs.hsaw_sample(g, fixed, 0, 1000, edge_removed=np.zeros(d["m"], np.uint8)).close(),
             lambda: hs.hsaw_classify(g, fixed, 0, 1000),
             lambda: hs.hsaw_solve_batch([g, g], [fixed, fixed], concurrency=1)]
    walks.close()  # its blocks are of the allocator of before: made again below
    for greedy in (None, "cluster", "grid"):
        for slab in (True, False):
            for i, call in enumerate(calls):
                if (greedy and i > 2) or (not slab and i in (3, 4, 7)):  # the latter have no slab
                    continue
                nth = 0
                while True:
                    nth += 1
                    with pytest.MonkeyPatch.context() as mp, Scratch() as a:
                        if greedy:
                            mp.setenv("HSAW_GREEDY", greedy)
                        walks = hs.hsaw_sample(g, fixed, 0, 1000)
                        held, first = set(a.live), a.asked
                        a.refuse = lambda b, h: (not slab and b >= 32 * MB) or a.asked - first >= nth
                        done = False
                        try:
                            out = call()
                            done = i != len(calls) - 1 or all(s == 0 for s, *_ in out)
                            if i == len(calls) - 1 and not done:
                                assert all(s in (0, -4) for s, *_ in out)
                        except hs.HsawError as e:
                            assert e.status == -4
                        torch.cuda.synchronize()
                        assert set(a.live) == held, (i, nth, len(a.live) - len(held))
                        used = a.asked - first
                        walks.close()
                    if done and used < nth:
                        break
                    assert nth < 400, (greedy, slab, i, used)


@pytest.mark.parametrize("call", ["solve", "greedy", "spread", "sample", "batch", "graph"])
def test_calls_do_with_less_scratch(call):
    """With too little memory for the scratch that only buys time (slab, counts by id, checkpoints, the edge sort's
    payload) a call does without and gives the same."""
    d = synth.workload_c1() if call in ("spread", "sample") else synth.workload_rmat(20, "wc", 1000, 20, "edge")
    g = hs.hsaw_graph_from_edges(d["n"], d["src"], d["dst"], d["w"])
    q = hs.Query(sources=d["sources"], mode=hs.HSAW_EDGE, k=20, n_hsaw=2000, seed=4)
    dev = [torch.from_numpy(x.view(np.int32)).cuda() for x in (d["src"], d["dst"], d["w"])]

    def run():
        if call == "solve":
            return hs.hsaw_solve(g, q)[:2]
        if call == "greedy":
            return hs.hsaw_greedy(walks, g, hs.HSAW_EDGE, 0, 2000, 20)
        if call == "spread":
            return hs.hsaw_estimate_spread(g, q, [5, 8])
        if call == "sample":
            w = hs.hsaw_sample(g, q, 0, 2000)
            out = [x[:2000] for x in w.export()]
            w.close()
            return out
        if call == "batch":
            return [x for s, ids, gains, _ in hs.hsaw_solve_batch([g, g], [q, q], concurrency=1) for x in (s, ids, gains)]
        h = hs.hsaw_graph_from_edges(d["n"], *dev)
        out = h.export()
        h.close()
        return out

    walks = hs.hsaw_sample(g, q, 0, 2000) if call == "greedy" else None
    ref = run()
    if walks:
        walks.close()
    # bytes held at most: the payload's 8 of 24 an edge less for the graph
    limit = {"solve": 60, "greedy": 90, "spread": 24, "sample": 24, "batch": 60, "graph": 300}[call] * MB
    with Scratch(lambda nbytes, held: held + nbytes > limit) as a:
        walks = hs.hsaw_sample(g, q, 0, 2000) if call == "greedy" else None
        got = run()
        if walks:
            walks.close()
        assert a.peak <= limit and not a.live
    for x, y in zip(ref, got):
        assert np.array_equal(x, y)
