"""Sample offsets and the node -> sample rows against the samples themselves: members at the edges of
a block's share (1,024 and 4,096), nodes that find no slot in a block's table, one node in every
sample, short and long samples, and scans of one tile, of two, and of more than 2,048 (with a pass
over the tiles' sums)."""
import numpy as np
import pytest

from paper_2306_03651_gb300 import inputs as I

pytestmark = pytest.mark.gpu
P = pytest.importorskip("paper_2306_03651_gb300")


def ring(n):
    src = np.arange(n)
    return I.from_edges(n, src, (src + 1) % n, False)


def star(n):
    return I.from_edges(n, np.zeros(n - 1, np.int64), np.arange(1, n), False)


def few_edges(n):
    return I.from_edges(n, np.array([0, 1, n - 2, n - 3]), np.array([1, 2, n - 1, n - 2]), False)


CASES = {  # graph, kappa, sizes of the job's cen_sample calls
    "one": (ring(5), 1, (1,)),
    "tile_edges": (ring(4096), 1, (1023, 1, 1)),
    "tile_edges_and_a_tile_of_nodes": (ring(4097), 1, (4095, 1, 1, 4095)),
    "wide": (star(3000), 2, (400000, 3)),
    "narrow_to_wide": (ring(300000), 6, (140000, 20000)),
    "long": (ring(8193), 60, (3000, 1200)),
    "many_tiles": (few_edges(4096 * 2048 + 1), 3, (5000,)),
    "samples_beyond_a_tile": (star(200), 1, (8193, 4096, 4097)),
}


@pytest.mark.parametrize("name", list(CASES))
def test_rows_hold_each_sample_once_per_member(name):
    g, kappa, parts = CASES[name]
    job = P.Job(P.Graph.of(g), 11, 2, space=P.SPACE_KPATH, kappa=kappa)
    for part in parts:
        job.sample(part)
        sample = job.samples()
        hoff, hmem, d = sample["hoff"], sample["hmem"], sample["d"]
        assert hoff[0] == 0 and np.array_equal(np.diff(hoff), d) and hoff[-1] == len(hmem)
        job.greedy_cover(1)
        noff, nsamp = job.incidence()
        c = np.bincount(hmem, minlength=g.n)
        assert noff[0] == 0 and np.array_equal(np.diff(noff), c)
        j = np.repeat(np.arange(len(d)), d)
        want = np.lexsort((j, hmem))  # by node, then sample
        row = np.repeat(np.arange(g.n), c)
        got = np.lexsort((nsamp, row))
        assert np.array_equal(nsamp[got], j[want])
    job.close()
