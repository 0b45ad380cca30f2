"""cen_job_copy_rade gives R and c of the sample that the last AMCERA read: at once, after the job has
grown, and whether the AMCERA went over the heavy nodes or over all; in several chunks of rows too."""
import numpy as np
import pytest

import oracle as O
from paper_2306_03651_gb300 import inputs as I

pytestmark = pytest.mark.gpu
P = pytest.importorskip("paper_2306_03651_gb300")


def ring(n, steps):
    src = np.repeat(np.arange(n), len(steps))
    return I.from_edges(n, src, (src + np.tile(steps, n)) % n, False)


# t rows of n entries; the third needs two chunks (256 MB hold 33 rows of two million entries)
CASES = {"small": (I.ba(400, 4, 2), 900, 33, 5), "heavy_decide": (ring(60000, [1, 7]), 9000, 64, 10),
         "all_needed": (ring(60000, [1, 7]), 9000, 31, 6000), "two_chunks": (ring(2_000_000, [1]), 3000, 40, 5)}


@pytest.mark.parametrize("name", list(CASES))
def test_rade_is_of_the_sample_the_amcera_read(name):
    g, m, t, k = CASES[name]
    space = dict() if name == "small" else dict(space=P.SPACE_KPATH, kappa=12)
    job, ojob = P.Job(P.Graph.of(g), 3, t, **space), O.Job(O.Graph.of(g), 3, t, **space)
    job.sample(m)
    ojob.sample(m)
    job.mcera(k)
    oR, oc = ojob.rade_matrix()
    R, c = job.rade()
    assert np.array_equal(R, oR.T) and np.array_equal(c, oc)
    job.sample(m // 2)
    with pytest.raises(P.CenError):  # the incidence is of the shorter sample
        job.rade()
    job.greedy_cover(k)
    for _ in range(2):  # reading changes nothing
        R, c = job.rade()
        assert np.array_equal(R, oR.T) and np.array_equal(c, oc)
    job.mcera(k)
    ojob.sample(m // 2)
    oR, oc = ojob.rade_matrix()
    R, c = job.rade()
    assert np.array_equal(R, oR.T) and np.array_equal(c, oc)
