"""Graph building at the ends of its tiles, passes and runs: raw arc lists of every remainder made
canonical (against a plain sort of unique keys), ids around powers of two of the sort's digits, long
runs of empty rows, and the in-arc CSR of directed graphs (through samples the oracle draws)."""
import numpy as np
import pytest

import oracle as O
from paper_2306_03651_gb300 import inputs as I

pytestmark = pytest.mark.gpu
P = pytest.importorskip("paper_2306_03651_gb300")


def raw(n, arcs, seed, low=0):
    """Arcs between ids low .. n - 1, skewed to the low ones, rows in draw order with repeats and loops."""
    rng = np.random.default_rng(seed)
    src = np.sort(low + (rng.random(arcs) ** 3 * (n - low)).astype(np.int64))
    dst = low + (rng.random(arcs) ** 2 * (n - low)).astype(np.int64)
    off = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(src, minlength=n), out=off[1:])
    return off, dst.astype(np.int32), src


def canonical(n, src, dst, symmetric):
    key = src * n + dst
    if symmetric:
        key = np.concatenate([key, dst * n + src])
    key = np.unique(key)
    key = key[key // n != key % n]
    off = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(key // n, minlength=n), out=off[1:])
    return off, (key % n).astype(np.int32)


SIZES = [(2, 1), (2, 3), (3, 255), (700, 256), (700, 257), (1024, 2047), (1025, 2048), (1025, 2049), (5000, 8191),
         (5000, 8192), (5000, 8193), (70000, 40000), (1 << 20, 30000), ((1 << 20) + 1, 30000), (3000, 300000)]


@pytest.mark.parametrize("symmetric", [False, True])
@pytest.mark.parametrize("n,arcs", SIZES)
def test_canonical_form(n, arcs, symmetric):
    off, col, src = raw(n, arcs, n + arcs)
    flags = P.GRAPH_CANONICALIZE | (P.GRAPH_SYMMETRIZE if symmetric else 0)
    got = P.Graph(n, off, col, directed=not symmetric, flags=flags).csr()
    want = canonical(n, src, col.astype(np.int64), symmetric)
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])


@pytest.mark.parametrize("n,low,arcs", [(300, 0, 900), (3000, 2500, 4000), (40000, 39000, 3000), (40000, 0, 9000)])
def test_in_arcs_of_a_directed_graph(n, low, arcs):
    """Empty rows before, between and (the heads being skewed) after the others."""
    off, col, src = raw(n, arcs, 5, low)
    g = I.from_edges(n, src, col, True)
    job = P.Job(P.Graph(n, off, col, directed=True, flags=P.GRAPH_CANONICALIZE), 2, 2)
    job.sample(400)
    ojob = O.Job(O.Graph.of(g), 2, 2)
    ojob.sample(400)
    a, b = job.samples(), ojob.hypergraph()
    for key in ("hoff", "s", "t", "d"):
        assert np.array_equal(a[key], b[key]), key
    assert np.array_equal(a["hmem"], b["hmem"][: b["hoff"][-1]])
