"""The GPU kernels at the sizes where their tiles, words and dispatch rules change, against the oracle.

Everything compared is a whole number, so equality is exact.
"""
import re

import numpy as np
import pytest

import oracle
import synth
from tinygraphs import ONE, random_tiny

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
hs = pytest.importorskip("paper_1702_05854_gb300")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.init()


def assert_same_stream(walks, ost, hits):
    """The first `hits` walks of a GPU stream equal the oracle's, walk by walk."""
    aid, off, nodes, edges = walks.export()
    o = ost.export()
    assert np.array_equal(aid[:hits], o.aid[:hits])
    assert np.array_equal(off[:hits + 1], o.node_off[:hits + 1])
    assert np.array_equal(nodes[:off[hits]], o.nodes[:off[hits]])
    assert np.array_equal(edges[:off[hits] - hits], o.edges[:off[hits] - hits])


def hub_graph(d, w):
    """Hub 0 with d equal in-edges of weight w from leaves 1..d, and an edge from the hub to every leaf."""
    leaves = np.arange(1, d + 1, dtype=np.int32)
    hub = np.zeros(d, np.int32)
    src, dst = np.concatenate([leaves, hub]), np.concatenate([hub, leaves])
    return d + 1, src, dst, np.concatenate([np.full(d, w, np.uint32), np.full(d, ONE, np.uint32)])


@pytest.mark.parametrize("d,share", [(1, 1.0), (2, 1.0), (3, 1.0), (255, 1.0), (256, 0.3), (4097, 1.0), (70001, 1.0),
                                     (70001, 0.25), (600_000, 1.0)])
def test_equal_weight_pick(d, share):
    """j = floor(r / w) at small, large and not-weighted-cascade equal weights (16-byte walk records)."""
    n, src, dst, w = hub_graph(d, int(ONE * share) // d)
    sources = np.arange(1, d + 1, 7, dtype=np.int32)
    g, og = hs.hsaw_graph_from_edges(n, src, dst, w), oracle.Graph(n, src, dst, w)
    q = hs.Query(sources=sources, seed=11)
    walks = hs.hsaw_sample(g, q, 0, 300)
    assert_same_stream(walks, oracle.Stream(oracle.Query(og, sources, seed=11)).extend(300), 300)


@pytest.mark.parametrize("m", [1, 2, 31, 33, 511, 513, 4095, 4096, 4097, 8193, 70_000])
def test_ingest_sort_tiles(m):
    """Stable order by destination around the radix sort's batches and tiles, in graphs of few and many nodes."""
    rng = np.random.default_rng(m)
    for n in (1, 3, 257, 100_000):
        src, dst = rng.integers(0, n, m).astype(np.int32), rng.integers(0, n, m).astype(np.int32)
        w = synth.wc_weights(n, dst)
        g, og = hs.hsaw_graph_from_edges(n, src, dst, w), oracle.Graph(n, src, dst, w)
        for x, y in zip(g.export(), og.arrays()):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("deg", [31, 32, 33, 1023, 1024, 1025, 4096, 4097, 8192, 50_001])
@pytest.mark.parametrize("kind", ["equal", "unequal", "zeros"])
def test_hub_lists(deg, kind):
    """Running sums, node records and guide records around the hub threshold and its tiles."""
    rng = np.random.default_rng(deg)
    n, src, dst, w = hub_graph(deg, int(ONE * 0.8) // deg)
    if kind != "equal":  # the hub's in-weights differ; with "zeros" half of them are 0
        x = rng.random(deg) + 0.01
        if kind == "zeros":
            x[rng.random(deg) < 0.5] = 0.0
            x[0] = 0.5
        w[:deg] = np.floor(x / x.sum() * 0.8 * ONE).astype(np.uint32)
    order = rng.permutation(src.size)
    src, dst, w = src[order], dst[order], w[order]
    g, og = hs.hsaw_graph_from_edges(n, src, dst, w), oracle.Graph(n, src, dst, w)
    for x, y in zip(g.export(), og.arrays()):
        assert np.array_equal(x, y)
    rp, s, _, _, _ = og.arrays()
    gc = hs.hsaw_graph_from_csr(n, rp, s, w[og.arrays()[4]])
    sources = np.arange(1, deg + 1, 5, dtype=np.int32)
    ost = oracle.Stream(oracle.Query(og, sources, seed=9)).extend(300)
    for graph in (g, gc):
        assert_same_stream(hs.hsaw_sample(graph, hs.Query(sources=sources, seed=9), 0, 300), ost, 300)


@pytest.mark.parametrize("n", [1, 31, 32, 33, 1000])
def test_running_sums_of_neighbours(n):
    """In-lists of every kind side by side in one warp's 32 nodes: none, up to 8 edges, up to and beyond 32 at a time,
    and hubs around their tiles of 2,048; equal weights, equal but one, weights of 0, and all different."""
    rng = np.random.default_rng(n)
    degs = [0, 1, 2, 7, 8, 9, 31, 32, 33, 63, 64, 65, 96, 1023, 1024, 1025]
    big = iter([2047, 2048, 2049, 4096, 4097, 8193])
    dst, w = [], []
    for v in range(n):
        deg = next(big, 0) if v % 13 == 12 else int(rng.choice(degs))
        x = np.full(deg, 1.0)
        kind = rng.integers(4)
        if kind == 1 and deg:
            x[rng.integers(deg)] = 2.0
        elif kind == 2:
            x[rng.random(deg) < 0.5] = 0.0
        elif kind == 3:
            x = rng.random(deg)
        dst.append(np.full(deg, v, np.int32))
        w.append(np.floor(x / max(1.0, x.sum()) * ONE * (1.0 - 2.0 ** -20)).astype(np.uint32))
    dst, w = np.concatenate(dst), np.concatenate(w)
    order = rng.permutation(dst.size)
    dst, w = dst[order], w[order]
    src = rng.integers(0, n, dst.size).astype(np.int32)
    og = oracle.Graph(n, src, dst, w)
    rp, s, _, _, index = og.arrays()
    for g in (hs.hsaw_graph_from_edges(n, src, dst, w), hs.hsaw_graph_from_csr(n, rp, s, w[index])):
        for x, y in zip(g.export()[:4], og.arrays()[:4]):
            assert np.array_equal(x, y)


def test_small_tables_unequal():
    """Graphs whose records would not fit L2 are walked through edges and a guide of one entry per four in-edges:
    in-lists of every length around the guide's groups, the sector and the hub threshold, with weights from uniform to
    one that takes nearly all."""
    rng = np.random.default_rng(3)
    parts, base = [], 0
    for deg in [*range(1, 14), 31, 32, 33, 63, 64, 65, 1023, 1024, 1025, 1027, 4096, 4099, 50_001, 600_000]:
        for skew in (0.0, 3.0):
            _, src, dst, w = hub_graph(deg, 1)
            x = (rng.random(deg) + 1e-3) ** (1.0 + skew)
            if skew:
                x[rng.integers(deg)] = 20.0 * deg
            w[:deg] = np.floor(x / x.sum() * rng.uniform(0.6, 1.0) * ONE).astype(np.uint32)
            parts.append((src + base, dst + base, w))
            base += deg + 1
    src, dst, w = (np.concatenate(p) for p in zip(*parts))
    order = rng.permutation(src.size)
    src, dst, w = src[order], dst[order], w[order]
    g, og = hs.hsaw_graph_from_edges(base, src, dst, w), oracle.Graph(base, src, dst, w)
    sources = np.arange(1, base, 11, dtype=np.int32)
    for first in (0, (1 << 32) - 500):
        ost = oracle.Stream(oracle.Query(og, sources, seed=2), first_aid=first).extend(4000)
        assert_same_stream(hs.hsaw_sample(g, hs.Query(sources=sources, seed=2), first, 4000), ost, 4000)


def test_small_tables_equal():
    """Equal weights beyond L2 as records: tails and node records."""
    n, m = 400_003, 9_500_001
    src, dst = synth.chung_lu_graph(n, m, 2.1, 6)
    w = synth.wc_weights(n, dst)
    g, og = hs.hsaw_graph_from_edges(n, src, dst, w), oracle.Graph(n, src, dst, w)
    sources, p = synth.sources(n, 20_000, 8), synth.probabilities(20_000, 9)
    ost = oracle.Stream(oracle.Query(og, sources, p_fixed=p, seed=2)).extend(3000)
    assert_same_stream(hs.hsaw_sample(g, hs.Query(sources=sources, p_fixed=p, seed=2), 0, 3000), ost, 3000)


@pytest.mark.parametrize("deg", [1024, 1025, 9000])
def test_hub_overweight(deg):
    """An in-sum of 2^32 is refused, 2^32 - 1 accepted, above and below the hub threshold."""
    n, src, dst, w = hub_graph(deg, ONE // deg)
    w[0] += np.uint32(ONE - (ONE // deg) * deg)
    hs.hsaw_graph_from_edges(n, src, dst, w).close()
    w[deg // 2] += np.uint32(1)
    with pytest.raises(hs.HsawError) as e:
        hs.hsaw_graph_from_edges(n, src, dst, w)
    assert e.value.status == -2


@pytest.mark.parametrize("m", [1, 7, 31, 32, 33, 63, 64, 65, 200])
@pytest.mark.parametrize("kind", ["edge", "node", "both"])
def test_removal_mask_words(m, kind):
    """Removal masks (any nonzero byte) around the 32-bit words they are packed into."""
    n, src, dst, w = random_tiny(m, n=max(2, m), m=m)
    rng = np.random.default_rng(m)
    er = (rng.random(m) < 0.3).astype(np.uint8) * rng.integers(1, 256, m).astype(np.uint8) if kind != "node" else None
    nr = (rng.random(n) < 0.3).astype(np.uint8) * rng.integers(1, 256, n).astype(np.uint8) if kind != "edge" else None
    if nr is not None:
        nr[n - 1] = 0
    sources = np.unique(np.array([0, n - 1], np.int32))
    g, og = hs.hsaw_graph_from_edges(n, src, dst, w), oracle.Graph(n, src, dst, w)
    walks = hs.hsaw_sample(g, hs.Query(sources=sources, seed=5), 0, 500, edge_removed=er, node_removed=nr)
    ost = oracle.Stream(oracle.Query(og, sources, edge_removed=er, node_removed=nr, seed=5)).extend(500)
    assert_same_stream(walks, ost, 500)


@pytest.fixture(scope="module")
def streams():
    """20,000 walks on the 16 K-node Chung-Lu graph from few suspects (180 K walk elements: ranges of them run on one
    CTA, at most 2^17 elements, or on the largest cluster) and from many (short walks, thousands of picks that gain)."""
    d = synth.workload_c1()
    g, og = hs.hsaw_graph_from_edges(d["n"], d["src"], d["dst"], d["w"]), oracle.Graph(d["n"], d["src"], d["dst"], d["w"])
    got = {}
    for name, sources in (("few", d["sources"]), ("many", synth.sources(d["n"], 9000, 5))):
        got[name] = (hs.hsaw_sample(g, hs.Query(sources=sources, seed=21), 0, 20_000),
                     oracle.Stream(oracle.Query(og, sources, seed=21)).extend(20_000))
    return d, g, got


@pytest.mark.parametrize("mode", [hs.HSAW_EDGE, hs.HSAW_NODE])
@pytest.mark.parametrize("who,first,count,k,share", [
    ("few", 0, 1, 3, 1.0),            # one walk, then zero-gain picks
    ("few", 5, 33, 40, 1.0),          # every gain small
    ("few", 0, 700, 1, 1.0),          # fewer elements kept per phase than there are
    ("few", 100, 3000, 32, 0.5),      # candidate mask
    ("few", 0, 20_000, 33, 1.0),      # the largest cluster
    ("few", 0, 20_000, 1000, 0.05),   # few candidates: gains end before the picks do
    ("many", 0, 20_000, 100, 1.0),    # many ties, several phases
    ("many", 0, 20_000, 4096, 1.0),   # as many picks as one block orders
    ("many", 0, 20_000, 7000, 1.0),   # more, levels down to 1, zero-gain picks in the edge mode
    ("many", 3, 2000, 16_000, 0.9),   # gains of 1 and 2, then zero-gain picks
])
def test_greedy_by_peaks(streams, mode, who, first, count, k, share):
    """Greedy by peaks: ids, gains and their order."""
    d, g, got = streams
    walks, ost = got[who]
    M = d["m"] if mode == hs.HSAW_EDGE else d["n"]
    mask = None if share == 1.0 else (np.random.default_rng(k).random(M) < share).astype(np.uint8)
    if mask is not None:
        k = min(k, int(mask.sum()))
    ids, gains = hs.hsaw_greedy(walks, g, mode, first, count, k, candidate_mask=mask)
    oids, ogains = ost.greedy(mode, first, count, M, k, cand_mask=mask, kept_gains=True)
    assert np.array_equal(gains, ogains)
    assert np.array_equal(ids, oids)


def test_greedy_conflict_chains():
    """Ties whose walks chain into each other: picks then take several rounds.  A path 0 -> 1 -> ... -> n - 1 with
    the suspect at 0 gives nested walks; a second copy with its ids interleaved gives equal gains."""
    n = 40
    even, odd = np.arange(0, 2 * n, 2, dtype=np.int32), np.arange(2 * n - 1, 0, -2, dtype=np.int32)
    src = np.concatenate([even[:-1], odd[:-1]])
    dst = np.concatenate([even[1:], odd[1:]])
    w = np.full(src.size, int(ONE * 0.9), np.uint32)
    sources = np.array([int(even[0]), int(odd[0])], np.int32)
    g, og = hs.hsaw_graph_from_edges(2 * n, src, dst, w), oracle.Graph(2 * n, src, dst, w)
    for seed in range(6):
        walks = hs.hsaw_sample(g, hs.Query(sources=sources, seed=seed), 0, 400)
        ost = oracle.Stream(oracle.Query(og, sources, seed=seed)).extend(400)
        for mode, M in ((hs.HSAW_EDGE, src.size), (hs.HSAW_NODE, 2 * n)):
            for first, count in ((0, 400), (3, 50), (100, 7)):
                ids, gains = hs.hsaw_greedy(walks, g, mode, first, count, 30)
                oids, ogains = ost.greedy(mode, first, count, M, 30)
                assert np.array_equal(gains, ogains) and np.array_equal(ids, oids)


@pytest.mark.parametrize("count", [16_000, 16_384, 16_385, 20_000, 60_000])
def test_greedy_elements_of_many_walks(count):
    """Elements in about as many walks as a thread block keeps to itself (16,384 pairs), or more."""
    n = 30
    src, dst = np.arange(n - 1, dtype=np.int32), np.arange(1, n, dtype=np.int32)
    src, dst = np.concatenate([src, [n + 1]]).astype(np.int32), np.concatenate([dst, [n - 1]]).astype(np.int32)
    w = np.full(src.size, ONE // 2 - 1, np.uint32)
    sources = np.array([0, n - 3, n + 1], np.int32)
    g, og = hs.hsaw_graph_from_edges(n + 2, src, dst, w), oracle.Graph(n + 2, src, dst, w)
    walks = hs.hsaw_sample(g, hs.Query(sources=sources, seed=3), 0, count)
    ost = oracle.Stream(oracle.Query(og, sources, seed=3)).extend(count)
    for mode, M in ((hs.HSAW_EDGE, src.size), (hs.HSAW_NODE, n + 2)):
        for k in (1, 3, 25):
            ids, gains = hs.hsaw_greedy(walks, g, mode, 0, count, k)
            oids, ogains = ost.greedy(mode, 0, count, M, k)
            assert np.array_equal(gains, ogains) and np.array_equal(ids, oids)


@pytest.mark.parametrize("count", [1, 31, 32, 33, 127, 4095, 4097, 116_735, 116_737, 233_471, 233_473, 1 << 18])
def test_static_chunks(count):
    """The allocation-free sampler's chunks of 32 to 256 attempts, and its blocks of 128 chunks."""
    d = synth.workload_c1()
    g = hs.hsaw_graph_from_edges(d["n"], d["src"], d["dst"], d["w"])
    og = oracle.Graph(d["n"], d["src"], d["dst"], d["w"])
    bits = np.zeros((d["n"] + 31) // 32, np.uint32)
    np.bitwise_or.at(bits, d["sources"] >> 5, np.uint32(1) << (d["sources"] & 31).astype(np.uint32))
    aid = torch.full((count,), -1, dtype=torch.int64, device="cuda")
    length = torch.full((count,), -1, dtype=torch.int32, device="cuda")
    first = 12_345
    n = hs.hsaw_sample_hits_static(g, torch.from_numpy(bits.view(np.int32)).cuda(), 4, first, count, aid, length)
    out, ln = oracle.Query(og, d["sources"], seed=4).classify(first, count)
    hit = np.nonzero(out == 1)[0]
    assert n == hit.size
    assert np.array_equal(aid[:n].cpu().numpy(), first + hit) and np.array_equal(length[:n].cpu().numpy(), ln[hit])
    assert bool((aid[n:] == -1).all()) and bool((length[n:] == -1).all())


@pytest.mark.parametrize("n,keep", [(40, 1.0), (700, 1.0), (3000, 1.0), (3000, 0.999)])
def test_rewalk_segments(n, keep):
    """Walks of every length up to n: on a path to the only suspect a hit started at node j has j + 1 nodes, so the
    checkpoints, none to far more than the eight kept, cut it in every way.  From the sampler and from a walk pool."""
    src, dst = np.arange(n - 1, dtype=np.int32), np.arange(1, n, dtype=np.int32)
    w = np.full(n - 1, int(ONE * keep), np.uint32)
    g, og = hs.hsaw_graph_from_edges(n, src, dst, w), oracle.Graph(n, src, dst, w)
    sources = np.array([0], np.int32)
    ost = oracle.Stream(oracle.Query(og, sources, seed=6)).extend(1500)
    for pool in (False, True):
        if pool:
            g.build_walk_pool(seed=6, attempts=1 << 14)
        assert_same_stream(hs.hsaw_sample(g, hs.Query(sources=sources, seed=6), 0, 1500), ost, 1500)


def test_stopping_rule_counts_by_sort_then_by_id():
    """A stopping rule on more than 2^24 edges with 5,000 picks: its early rounds sort the walk elements, its last has
    an eighth as many of them as there are edges and counts by id, and more picks are made than one block orders."""
    n, k, eps = 1 << 20, 5000, 0.45
    src, dst = synth.rmat_graph(20, 17)
    w, sources = synth.wc_weights(n, dst), synth.sources(n, 1000)
    M = src.size
    g = hs.hsaw_graph_from_edges(n, src, dst, w)
    ids, gains, r = hs.hsaw_solve(g, hs.Query(sources=sources, mode=hs.HSAW_EDGE, k=k, sampling=hs.HSAW_STOP_RULE,
                                              eps=eps, seed=synth.SEED_WALKS))
    og = oracle.Graph(n, src, dst, w)
    half = r["hits"] // 2
    ost = oracle.Stream(oracle.Query(og, sources, seed=synth.SEED_WALKS)).extend_threads(2 * half, threads=8)
    off = ost.export().node_off
    elements, before = (int(off[h] - off[0]) - h for h in (half, half // 2))
    assert M > 1 << 24 and M <= 8 * elements and M > 8 * before  # the two rounds count in different ways
    oids, ogains = ost.greedy(oracle.MODE_EDGE, 0, half, M, k, kept_gains=True)
    assert ogains[-1] > 0
    assert np.array_equal(gains, ogains) and np.array_equal(ids, oids)
    assert r["cov_Rprime"] == ost.coverage(oracle.MODE_EDGE, half, half, M, oids)


def greedy_records(err):
    """The launch records of the greedy by peaks, as dicts."""
    return [dict((k, float(v)) for k, v in re.findall(r"(\w+)=([\d.]+)", line))
            for line in err.splitlines() if line.startswith("hsaw: k_greedy_peaks ")]


@pytest.mark.parametrize("count", [300, 20_000])
def test_greedy_record_names_its_kernel(streams, capfd, monkeypatch, count):
    """The launch record says which greedy ran: the one by peaks unless the environment asks for another."""
    d, g, got = streams
    monkeypatch.setenv("HSAW_LOG_LAUNCHES", "1")
    for force in (None, "cluster", "grid"):
        monkeypatch.setenv("HSAW_GREEDY", force) if force else monkeypatch.delenv("HSAW_GREEDY", raising=False)
        capfd.readouterr()
        hs.hsaw_greedy(got["many"][0], g, hs.HSAW_EDGE, 0, count, 20)
        err = capfd.readouterr().err
        runs = greedy_records(err)
        assert len(runs) == (0 if force else 1)
        if runs:
            assert runs[0]["walks"] == count and runs[0]["picks"] == 20 and runs[0]["owned"] <= runs[0]["phases"]
        else:
            assert ("hsaw: k_greedy_cluster " in err) == (force == "cluster")


def concentrated(name):
    """(n, src, dst, w, sources, mode) of streams in which few elements are in many walks."""
    if name.startswith("path"):  # nested walks
        n = int(name[4:])
        src, dst = np.arange(n - 1, dtype=np.int32), np.arange(1, n, dtype=np.int32)
        return n, src, dst, np.full(n - 1, ONE, np.uint32), np.array([0], np.int32), hs.HSAW_NODE
    if name == "chung-lu":
        d = synth.workload_c1()
        return d["n"], d["src"], d["dst"], d["w"], d["sources"], hs.HSAW_EDGE
    src, dst = synth.rmat_graph(13, 5)
    return 1 << 13, src, dst, synth.wc_weights(1 << 13, dst), synth.sources(1 << 13, 1000), hs.HSAW_NODE


# Pairs of each list against those that the thread blocks hold and those with which the greedy by peaks goes on, from
# the oracle's counts: 932 K (262 K, 276 K), 177 K (262 K, 253 K; an element in more walks than a block holds),
# 131 K (131 K, 124 K; elements of up to 2,700 do not share out evenly), 376 K (262 K, 321 K), 344 K (262 K, 451 K;
# 60 picks in 27 rounds).
@pytest.mark.parametrize("name,count,k,route", [
    ("path30", 60_000, 1, "not begun"),
    ("chung-lu", 100_000, 10, "kept"),
    ("path100", 2_700, 10, "left at once"),
    ("rmat", 120_000, 300, "left at once"),
    ("rmat", 80_000, 1000, "left later"),
])
def test_greedy_leaves_long_lists(capfd, monkeypatch, name, count, k, route):
    """Lists of many walks go to the greedy that takes one pick at a time: before the first round, or when the rounds
    take longer than their picks are worth.  The picks are the same either way."""
    n, src, dst, w, sources, mode = concentrated(name)
    M = src.size if mode == hs.HSAW_EDGE else n
    g, og = hs.hsaw_graph_from_edges(n, src, dst, w), oracle.Graph(n, src, dst, w)
    ost = oracle.Stream(oracle.Query(og, sources, seed=4)).extend_threads(count, threads=8)
    walks = hs.hsaw_sample(g, hs.Query(sources=sources, seed=4), 0, count)
    monkeypatch.setenv("HSAW_LOG_LAUNCHES", "1")
    capfd.readouterr()
    ids, gains = hs.hsaw_greedy(walks, g, mode, 0, count, k)
    err = capfd.readouterr().err
    peaks = [line for line in err.splitlines() if line.startswith("hsaw: k_greedy_peaks ")]
    one_pick = "hsaw: k_greedy_cluster " in err or "hsaw: k_greedy_onchip " in err
    assert len(peaks) == (0 if route == "not begun" else 1)
    assert one_pick == (route != "kept") and any(" left " in line for line in peaks) == route.startswith("left")
    if route.startswith("left"):
        rounds = int(re.search(r"rounds=(\d+)", peaks[0])[1])
        assert rounds <= 1 if route == "left at once" else rounds > 2
    oids, ogains = ost.greedy(mode, 0, count, M, k, kept_gains=True)
    assert np.array_equal(gains, ogains) and np.array_equal(ids, oids)


def greedy_of_one_list(capfd, monkeypatch, walks, ost, g, mode, M, count, k, mask):
    """The greedy's launch record; its picks are the oracle's."""
    monkeypatch.setenv("HSAW_LOG_LAUNCHES", "1")
    capfd.readouterr()
    ids, gains = hs.hsaw_greedy(walks, g, mode, 0, count, k, candidate_mask=mask)
    run, = greedy_records(capfd.readouterr().err)
    oids, ogains = ost.greedy(mode, 0, count, M, k, cand_mask=mask, kept_gains=True)
    assert np.array_equal(gains, ogains) and np.array_equal(ids, oids)
    return run


# 512 threads a block up to 2^14 walks, 1,024 beyond; 16 pairs a thread
@pytest.mark.parametrize("node,pairs,whole", [(0, 8191, True), (0, 8192, True), (0, 8193, False), (0, 16_383, False),
                                              (1, 16_383, True), (1, 16_384, True), (1, 16_385, False)])
def test_greedy_element_of_a_block(capfd, monkeypatch, node, pairs, whole):
    """One element in as many walks as a thread block keeps, or one more or less: the suspect, on every walk of a path,
    or the node before it."""
    n = 10
    src, dst = np.arange(n - 1, dtype=np.int32), np.arange(1, n, dtype=np.int32)
    w = np.full(n - 1, ONE, np.uint32)
    sources = np.array([0], np.int32)
    g, og = hs.hsaw_graph_from_edges(n, src, dst, w), oracle.Graph(n, src, dst, w)
    ost = oracle.Stream(oracle.Query(og, sources, seed=3)).extend(20_000)
    length = np.diff(ost.export().node_off)
    count = int(np.nonzero(np.cumsum(length > node) == pairs)[0][0]) + 1  # a walk of l nodes starts at node l - 1
    assert node == 0 or count > 1 << 14
    walks = hs.hsaw_sample(g, hs.Query(sources=sources, seed=3), 0, count)
    mask = np.zeros(n, np.uint8)
    mask[node] = 1
    run = greedy_of_one_list(capfd, monkeypatch, walks, ost, g, hs.HSAW_NODE, n, count, 1, mask)
    assert run["pairs"] == pairs and run["phases"] == 1 and run["owned"] == int(whole)


@pytest.mark.parametrize("elements,whole", [(16 * 3072 - 1, True), (16 * 3072, True), (16 * 3072 + 1, False)])
def test_greedy_elements_of_a_block(capfd, monkeypatch, elements, whole):
    """As many elements of one walk each as the thread blocks keep, 3,072 a block, or one more or less."""
    n, count = 200_000, 70_000
    src, dst, w = np.array([0], np.int32), np.array([1], np.int32), np.array([1], np.uint32)
    sources = np.arange(n, dtype=np.int32)
    g, og = hs.hsaw_graph_from_edges(n, src, dst, w), oracle.Graph(n, src, dst, w)
    ost = oracle.Stream(oracle.Query(og, sources, seed=3)).extend(count)
    walks = hs.hsaw_sample(g, hs.Query(sources=sources, seed=3), 0, count)
    once = np.nonzero(np.bincount(ost.export().nodes[:count], minlength=n) == 1)[0]
    mask = np.zeros(n, np.uint8)
    mask[once[:elements]] = 1
    assert once.size >= elements
    run = greedy_of_one_list(capfd, monkeypatch, walks, ost, g, hs.HSAW_NODE, n, count, 3200, mask)
    assert run["pairs"] == elements and run["phases"] == 1 and run["owned"] == int(whole)


def small_table_graph(kind):
    """Graphs beyond the sizes that are walked through records (128 MB of L2): tails (152 MB of records), or edges and
    guide (45 MB, random weights)."""
    n, m = (400_003, 9_500_001) if kind == "tails" else (60_003, 700_001)
    src, dst = synth.chung_lu_graph(n, m, 2.1, 6)
    return n, src, dst, synth.wc_weights(n, dst) if kind == "tails" else synth.random_lt_weights(n, dst, 7)


@pytest.fixture(scope="module", params=["tails", "edges"])
def small_tables(request):
    n, src, dst, w = small_table_graph(request.param)
    return n, src.size, hs.hsaw_graph_from_edges(n, src, dst, w), oracle.Graph(n, src, dst, w)


@pytest.mark.parametrize("kind", ["edge", "node", "both"])
def test_small_tables_removal(small_tables, kind):
    """Removed edges and nodes with the small walk tables, coins on or off."""
    n, m, g, og = small_tables
    rng = np.random.default_rng(4)
    er = (rng.random(m) < 0.2).astype(np.uint8) if kind != "node" else None
    nr = (rng.random(n) < 0.1).astype(np.uint8) if kind != "edge" else None
    sources, p = synth.sources(n, n // 50, 8), synth.probabilities(n // 50, 9)
    for coins in (None, p):
        ost = oracle.Stream(oracle.Query(og, sources, p_fixed=coins, edge_removed=er, node_removed=nr, seed=2)).extend(3000)
        walks = hs.hsaw_sample(g, hs.Query(sources=sources, p_fixed=coins, seed=2), 0, 3000, edge_removed=er, node_removed=nr)
        assert_same_stream(walks, ost, 3000)


@pytest.mark.parametrize("coins", [False, True])
def test_small_tables_pool(small_tables, coins):
    """Walk pools with the small walk tables: hits, lengths and walks, and the stream past the pool's end."""
    n, m, g, og = small_tables
    sources = synth.sources(n, n // 200, 8)
    p = synth.probabilities(n // 200, 9) if coins else None
    ost = oracle.Stream(oracle.Query(og, sources, p_fixed=p, seed=2)).extend_threads(6000, threads=8)
    inside = int(ost.export().aid[3000])  # half of the hits lie in the pool
    try:
        g.build_walk_pool(2, inside)
        assert_same_stream(hs.hsaw_sample(g, hs.Query(sources=sources, p_fixed=p, seed=2), 0, 6000), ost, 6000)
    finally:
        g.drop_walk_pool()
