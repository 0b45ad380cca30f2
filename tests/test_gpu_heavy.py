"""greedyCover and the AMCERA over the heavy nodes (at most 16,384 of the largest c_u), and over all
nodes where those do not decide: against the oracle, with rows of one and of many chunks, sign rows
of every alignment, and k beyond what the heavy nodes hold."""
import numpy as np
import pytest

import oracle as O
from paper_2306_03651_gb300 import inputs as I

pytestmark = pytest.mark.gpu
P = pytest.importorskip("paper_2306_03651_gb300")


def ring(n, steps):
    src = np.repeat(np.arange(n), len(steps))
    return I.from_edges(n, src, (src + np.tile(steps, n)) % n, False)


def star(n):
    """A centre in every other walk or so: a row of some thousands of incidences beside n - 1 short ones."""
    return I.from_edges(n, np.zeros(n - 1, np.int64), np.arange(1, n), False)


CASES = {  # graph, m, kappa, t, values of k
    "all_listed": (ring(16384, [1, 5]), 3000, 6, 10, (1, 20)),
    "few_touched": (ring(60000, [1, 7]), 500, 10, 33, (1, 40, 3000)),
    "heavy_decide": (ring(60000, [1, 7]), 40000, 12, 64, (1, 10)),
    "all_needed": (ring(60000, [1, 7]), 40000, 12, 31, (10, 6000, 10)),
    "one_bucket": (ring(40000, [1]), 300000, 1, 4, (3,)),
    "many_chunks": (star(20001), 30000, 3, 130, (1, 5)),
    "chunk_edges": (star(300), 4097, 1, 128, (2,)),
    "no_samples": (ring(20000, [1]), 0, 2, 5, (3,)),
}


@pytest.mark.parametrize("name", list(CASES))
def test_cover_and_mcera_match_the_oracle(name):
    g, m, kappa, t, ks = CASES[name]
    job = P.Job(P.Graph.of(g), 3, t, space=P.SPACE_KPATH, kappa=kappa)
    ojob = O.Job(O.Graph.of(g), 3, t, space=P.SPACE_KPATH, kappa=kappa)
    for part in (m // 3, m - m // 3):  # lists and rows of a grown sample
        if part:
            job.sample(part)
            ojob.sample(part)
        for k in ks:
            S, covered, Rnum, Wnum, b = job.cover_and_mcera(k)
            oS, ocovered = ojob.greedy_cover(k)
            oR, oW, ob = ojob.mcera(k)
            assert S.tolist() == oS.tolist() and covered == ocovered, k
            assert np.array_equal(Rnum, oR) and Wnum == oW and b == ob, k
            S2, covered2 = job.greedy_cover(k)
            R2, W2, b2 = job.mcera(k)
            assert S2.tolist() == S.tolist() and covered2 == covered
            assert np.array_equal(R2, Rnum) and (W2, b2) == (Wnum, b)
    if m:
        R, c = job.rade()
        oR, oc = ojob.rade_matrix()
        assert np.array_equal(R, oR.T) and np.array_equal(c, oc)
