"""The GPU kernels at the sizes where their tiles, words and dispatch rules change, against the oracle.

Everything compared is a whole number, so equality is exact.
"""
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
