"""Where the heavy nodes do not decide every pick, greedyCover goes on from the picks that they did decide:
in a cluster (of 16 and of 8 CTAs) and, on a graph whose gains no cluster holds, in the grid form.  The picks
are those of the grid form over all nodes from the first pick on; a later call of few picks goes over the
heavy nodes again."""
import numpy as np
import pytest

from paper_2306_03651_gb300 import inputs as I

pytestmark = pytest.mark.gpu
P = pytest.importorskip("paper_2306_03651_gb300")


def ring(n):
    src = np.repeat(np.arange(n), 2)
    return I.from_edges(n, src, (src + np.tile([1, 7], n)) % n, False)


# (n, samples, nodes a sample, k); the samples of the last two are moved by 32 and by 4 lanes each
CASES = {"cluster": (60000, 40000, 12, 6000), "long_samples": (60000, 20000, 24, 9000),
         "grid": (1_000_000, 60000, 12, 20000)}


def launches(job, kernel):
    return job.stats()[kernel]["launches"]


@pytest.mark.parametrize("name", list(CASES))
def test_the_picks_go_on_over_all_nodes(name, monkeypatch):
    n, m, kappa, k = CASES[name]
    graph = P.Graph.of(ring(n))

    def sampled():
        job = P.Job(graph, 3, 4, space=P.SPACE_KPATH, kappa=kappa)
        job.sample(m)
        return job

    monkeypatch.setenv("CEN_GREEDY_GRID", "1")
    job = sampled()
    ref, few = job.greedy_cover(k), job.greedy_cover(10)
    monkeypatch.delenv("CEN_GREEDY_GRID")
    for size in ("16", "8"):
        monkeypatch.setenv("CEN_GREEDY_CLUSTER", size)
        job = sampled()
        # the heavy nodes, the gains that are left (two), the rest; then the heavy nodes alone
        for picks, want, kernels in ((k, ref, 4), (10, few, 5)):
            S, covered = job.greedy_cover(picks)
            assert S.tolist() == want[0].tolist() and covered == want[1]
            assert launches(job, "greedy") == kernels
        S, covered = job.greedy_cover(k)
        assert S.tolist() == ref[0].tolist() and covered == ref[1]


def test_a_large_k_leaves_the_amcera_of_a_small_one_to_the_heavy_nodes():
    job, fresh = (P.Job(P.Graph.of(ring(60000)), 3, 4, space=P.SPACE_KPATH, kappa=12) for _ in range(2))
    for j in (job, fresh):
        j.sample(40000)
    job.mcera(6000)
    before = launches(job, "select")
    a, b = job.mcera(10), fresh.mcera(10)
    assert np.array_equal(a[0], b[0]) and a[1:] == b[1:]
    assert launches(job, "select") - before == launches(fresh, "select") == 1
