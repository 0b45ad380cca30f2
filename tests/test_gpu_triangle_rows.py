"""Triangle counts where a lane's arcs meet a warp's: shorter rows of about 32 entries, runs of 8 and of 32 arcs."""
import numpy as np
import pytest

import oracle as O
from paper_2306_03651_gb300 import inputs as I

pytestmark = pytest.mark.gpu
P = pytest.importorskip("paper_2306_03651_gb300")


def cliques(sizes):
    """Complete graphs side by side, and a node joined to every node of all of them."""
    src, dst, at = [], [], 1
    for n in sizes:
        a, b = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
        src.append(at + a[a < b])
        dst.append(at + b[a < b])
        at += n
    src.append(np.zeros(at - 1, np.int64))
    dst.append(np.arange(1, at))
    return I.from_edges(at, np.concatenate(src), np.concatenate(dst), False)


def lattice(n, near):
    src = np.repeat(np.arange(n), near)
    return I.from_edges(n, src, (src + np.tile(np.arange(1, near + 1), n)) % n, False)


@pytest.mark.parametrize("g", [cliques([2, 3, 31, 32, 33, 34, 60]), lattice(30000, 9), lattice(9000, 40)],
                         ids=["cliques", "short_rows", "long_rows"])
def test_triangles_match_the_oracle(g):
    m = 3000
    job = P.Job(P.Graph.of(g), 6, 2, space=P.SPACE_TRIANGLE)
    ojob = O.Job(O.Graph.of(g), 6, 2, space=O.SPACE_TRIANGLE)
    job.sample(m)
    ojob.sample(m)
    h, ref = job.samples(), ojob.hypergraph()
    for key in ("s", "t", "d"):
        assert np.array_equal(h[key], ref[key]), key
    assert np.array_equal(h["hmem"], ref["hmem"][:ref["hoff"][-1]])
