"""The sizes of bidirectional search: CTAs of 128, 512 and 1,024 threads with their state in
shared memory, and the tables in global memory, against the oracle where a search passes from
one to the next, and against the global-memory search over graphs of every kind."""
import numpy as np
import pytest

import oracle as O
from paper_2306_03651_gb300 import inputs as I

pytestmark = pytest.mark.gpu
P = pytest.importorskip("paper_2306_03651_gb300")


def hubs(directed):
    """40 hubs beside 700 nodes, all arcs between the two sets (in one direction or one third of them when
    directed): pairs of hubs have 700 or so common neighbours, so a walk step picks among them by digits of the id."""
    a, b = np.meshgrid(np.arange(40), 40 + np.arange(700), indexing="ij")
    src, dst = a.ravel(), b.ravel()
    if directed:
        back = np.random.default_rng(1).random(src.size) < 1 / 3
        src, dst = np.concatenate([src, dst[back]]), np.concatenate([dst, src[back]])
    return I.from_edges(740, src, dst, directed)


def stars():
    """Two joined hubs with 70,000 leaves each: a level of more than 65,536 arcs is a wide CTA's."""
    leaves = 2 + np.arange(140_000)
    return I.from_edges(140_002, np.concatenate([[0], leaves % 2]), np.concatenate([[1], leaves]), False)


def layers(width, depth):
    """Complete arcs between consecutive layers: width^(d-1) shortest paths between nodes d layers apart."""
    a, b = np.meshgrid(np.arange(width), np.arange(width), indexing="ij")
    src = np.concatenate([a.ravel() + width * i for i in range(depth - 1)])
    dst = np.concatenate([b.ravel() + width * (i + 1) for i in range(depth - 1)])
    return I.from_edges(width * depth, src, dst, False)


def cycle(n):
    return I.from_edges(n, np.arange(n), (np.arange(n) + 1) % n, False)


CASES = {
    "hubs": (hubs(False), 3000), "hubs_directed": (hubs(True), 3000), "stars": (stars(), 200),
    "counts_beyond_32_bits": (layers(10, 14), 1200), "31_levels": (cycle(125), 400), "deeper": (cycle(140), 400),
    "grid": (I.grid_rewired(300, 300, 0.01, 3), 500), "two_nodes": (I.from_edges(2, [0], [1], False), 5),
    "one_arc": (I.from_edges(3, [0], [1], True), 50),
}


def same(a, b):
    for key in ("hoff", "s", "t", "d", "hmem"):
        assert np.array_equal(a[key], b[key]), key


@pytest.mark.parametrize("name", list(CASES))
def test_samples_are_the_oracles(name):
    g, m = CASES[name]
    ojob = O.Job(O.Graph.of(g), 5, 3)
    ojob.sample(m)
    job = P.Job(P.Graph.of(g), 5, 3)
    job.sample(m // 2)  # the second call starts from what the first recorded on the graph
    job.sample(m - m // 2)
    ref = ojob.hypergraph()
    same(job.samples(), dict(ref, hmem=ref["hmem"][:ref["hoff"][-1]]))
    assert job.sampler_info()["deferred_search"] == job.sampler_info()["deferred_walk"] == 0


@pytest.mark.parametrize("g", [I.rmat(14, 16, seed=2), I.rmat(15, 8, seed=4, directed=True, keep_lcc=False),
                               I.ba(30000, 6, 3), I.grid_rewired(700, 500, 0.01, 2), I.rmat(18, 16, seed=1)],
                         ids=["rmat14", "rmat15_directed", "ba30000", "grid", "rmat18"])
@pytest.mark.parametrize("warps", [-1, 1])
def test_samples_equal_the_global_memory_searchs(g, warps):
    graph, m = P.Graph.of(g), 20000 if g.name.startswith("grid") else 60000
    ref = P.Job(graph, 8, 3)
    ref.tune(bidir_table=0, bidir_warps=0)
    ref.sample(m)
    job = P.Job(graph, 8, 3)
    job.tune(bidir_warps=warps)
    job.sample(m)
    same(job.samples(), ref.samples())
    assert (job.sampler_info()["escalated"] > 0) == (warps == 1)
