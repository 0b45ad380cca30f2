"""The largest searches of a call, a few of them: CTAs of 1,024 threads with their state in shared memory, and
with the tables in global memory what outgrows that."""
import numpy as np
import pytest

import oracle as O
from paper_2306_03651_gb300 import inputs as I

pytestmark = pytest.mark.gpu
P = pytest.importorskip("paper_2306_03651_gb300")


def layered(width, layers, arcs, seed):
    """Layers of `width` nodes, each node joined to `arcs` random nodes of the next layer."""
    r = np.random.default_rng(seed)
    src = np.concatenate([np.repeat(np.arange(width) + width * i, arcs) for i in range(layers - 1)])
    dst = np.concatenate([r.integers(0, width, width * arcs) + width * (i + 1) for i in range(layers - 1)])
    return I.from_edges(width * layers, src, dst, False)


def same(a, b):
    for key in ("hoff", "s", "t", "d", "hmem"):
        assert np.array_equal(a[key], b[key]), key


def test_layers_match_the_oracle():
    """A replay of 150 such searches on the CPU: 114 fit the small CTAs, 27 the wide ones, 5 need 6,400 to 12,288
    nodes or 10,000 to 18,432 logged arcs, so that only the 1,024-thread CTAs hold them, and 4 more than that."""
    g, m = layered(1000, 20, 2, 1), 1500
    job, ojob = P.Job(P.Graph.of(g), 6, 3), O.Job(O.Graph.of(g), 6, 3)
    job.sample(m)
    ojob.sample(m)
    assert job.stats()["bidir"]["launches"] == 4  # small, wide, 1,024 threads, and those with tables in global memory
    ref = ojob.hypergraph()
    same(job.samples(), dict(ref, hmem=ref["hmem"][:ref["hoff"][-1]]))


@pytest.mark.parametrize("side, m, seed", [(700, 700, 3), (1200, 600, 4)])
def test_grids_equal_the_global_memory_searchs(side, m, seed):
    g = I.grid_rewired(side, side, 0.01, 2)
    job, ref = P.Job(P.Graph.of(g), seed, 3), P.Job(P.Graph.of(g), seed, 3)
    ref.tune(bidir_table=0, bidir_warps=0)
    for part in (m, m // 2):  # the second call starts with the wide CTAs
        job.sample(part)
        ref.sample(part)
    assert job.stats()["bidir"]["launches"] == 4 + 3 and ref.stats()["bidir"]["launches"] == 2
    same(job.samples(), ref.samples())
