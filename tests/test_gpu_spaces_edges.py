"""The kappa-path and triangle samplers where their lane groups and runs end: walks around 8 and 32
nodes, walks that use a whole component up, rows of more common neighbours than one pass holds."""
import numpy as np
import pytest

import oracle as O
from paper_2306_03651_gb300 import inputs as I

pytestmark = pytest.mark.gpu
P = pytest.importorskip("paper_2306_03651_gb300")


def complete(n, directed=False):
    a, b = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    keep = (a != b) if directed else (a < b)
    return I.from_edges(n, a[keep], b[keep], directed)


def sinks():
    """A directed path into a node without out-arcs, beside isolated nodes."""
    return I.from_edges(30, [0, 1, 2, 3, 3], [1, 2, 3, 4, 5], True)


@pytest.mark.parametrize("kappa", [7, 8, 9, 31, 32, 33, 70, 1024])
@pytest.mark.parametrize("g", [complete(34), complete(9, True), sinks(), I.ba(400, 6, 2)],
                         ids=["complete34", "complete9_directed", "sinks", "ba400"])
def test_walks_of_every_group_size(g, kappa):
    job = P.Job(P.Graph.of(g), 4, 2, space=P.SPACE_KPATH, kappa=kappa)
    ojob = O.Job(O.Graph.of(g), 4, 2, space=O.SPACE_KPATH, kappa=kappa)
    for m in (1, 300):
        job.sample(m)
        ojob.sample(m)
    a, b = job.samples(), ojob.hypergraph()
    for key in ("hoff", "s", "t", "d", "hmem"):
        assert np.array_equal(a[key], b[key]), key


@pytest.mark.parametrize("g", [complete(3), complete(34), complete(131), I.rmat(11, 24, seed=5)],
                         ids=["one_triangle", "complete34", "complete131", "rmat11"])
def test_triangles_of_long_rows(g):
    job = P.Job(P.Graph.of(g), 6, 2, space=P.SPACE_TRIANGLE)
    ojob = O.Job(O.Graph.of(g), 6, 2, space=O.SPACE_TRIANGLE)
    for m in (1, 900):
        job.sample(m)
        ojob.sample(m)
    a, b = job.samples(), ojob.hypergraph()
    for key in ("hoff", "s", "t", "d", "hmem"):
        assert np.array_equal(a[key], b[key]), key
