"""What calls record on a graph about the sizes of bidirectional search: which launches a later call makes.
A call that starts with the small shared-memory CTAs makes two (small, wide) or four (and two for the
few left), one that starts with the wide ones one or three, one with the tables in global memory one."""
import numpy as np
import pytest

import oracle as O
from paper_2306_03651_gb300 import inputs as I

pytestmark = pytest.mark.gpu
P = pytest.importorskip("paper_2306_03651_gb300")


def launches(graph, m, seed=1, **params):
    job = P.Job(graph, seed, 1)
    job.tune(**params)
    job.sample(m)
    return job.stats()["bidir"]["launches"]


def test_warp_searches_leave_no_record_for_cta_searches():
    """On this grid some 43% of all searches outgrow the small CTAs, but more than half of those that the
    warps hand on do; a later job without warp searches still starts small."""
    g = I.grid_rewired(120, 120, 0.01, 1)
    fresh, after = P.Graph.of(g), P.Graph.of(g)
    launches(after, 3000, bidir_warps=1)
    assert launches(fresh, 3000) == 2
    assert launches(after, 3000) == 2


def test_searches_that_outgrow_a_wide_cta_are_counted_once():
    """Nearly all of these outgrow the wide CTAs, and most of those the 1,024-thread ones too."""
    job = P.Job(P.Graph.of(I.grid_rewired(2048, 2048, 0.01, 1)), 1, 1)
    job.sample(400)
    assert job.stats()["bidir"]["launches"] == 4 and 200 < job.sampler_info()["migrated"] <= 400


def test_short_calls_settle_on_the_wide_ctas():
    """Most of this grid's searches outgrow the small CTAs and none the wide ones: calls of 300 learn it together."""
    graph = P.Graph.of(I.grid_rewired(200, 200, 0.01, 1))
    assert [launches(graph, 300, seed) for seed in range(4)] == [2, 2, 1, 1]


def test_many_deep_searches_start_in_global_memory_and_few_do_not():
    """Here the wide CTAs leave 10%.  The first call of 8,000 finds that out on the way (small, wide, and the rest
    with the tables in global memory), later ones start there; a call of 500 stays in shared memory."""
    graph = P.Graph.of(I.grid_rewired(500, 500, 0.01, 1))
    assert [launches(graph, m, 1) for m in (8000, 8000, 500, 8000)] == [3, 1, 3, 1]


def test_a_first_call_of_long_samples_is_searched_once():
    """Some 21 members a sample, more than eight and the arena's spare million hold: a short arena would have the
    samples searched twice, in twice as many launches (small, wide, and in global memory the many that are left)."""
    job = P.Job(P.Graph.of(I.grid_rewired(200, 200, 0.01, 1)), 1, 1)
    job.sample(80000)
    assert job.size()[1] > 8 * 80000 + (1 << 20) and job.stats()["bidir"]["launches"] == 3


def test_searches_left_untried_do_not_count_as_left_by_the_wide_ctas():
    """The first call hands nearly all on untried; the wide CTAs would leave 10%, so a call of 950 still starts there."""
    graph = P.Graph.of(I.grid_rewired(500, 500, 0.01, 1))
    assert [launches(graph, m, 1) for m in (8000, 950)] == [3, 3]


@pytest.mark.parametrize("nodes, kernels", [(150, 2), (220, 2), (222, 2), (244, 2), (246, 3), (700, 3)])
def test_long_thin_searches(nodes, kernels):
    """Pairs of a cycle are up to half its length apart, and the sides grow in turn, up to LV - 1 and LV - 2 levels:
    110 arcs fit the small CTAs' 56 levels, 122 the wide ones' 62, and more go to the 128-thread CTAs with tables in
    global memory, not by way of the 1,024-thread ones."""
    g = I.from_edges(nodes, np.arange(nodes), (np.arange(nodes) + 1) % nodes, False)
    job, ojob = P.Job(P.Graph.of(g), 1, 1), O.Job(O.Graph.of(g), 1, 1)
    job.sample(2000)
    ojob.sample(2000)
    assert job.stats()["bidir"]["launches"] == kernels
    h, ref = job.samples(), ojob.hypergraph()
    assert h["d"].max() >= nodes // 2 - 1
    for key in ("hoff", "s", "t", "d"):
        assert np.array_equal(h[key], ref[key]), key
    assert np.array_equal(h["hmem"], ref["hmem"][:ref["hoff"][-1]])


def test_deep_searches_that_small_ctas_leave_skip_the_wide_ones_where_they_are_many():
    """Some 43% of this grid's searches outgrow the small CTAs, 3,400 of 8,000: from the second call on those go
    straight to the tables in global memory; 1,290 of 3,000 do not."""
    graph = P.Graph.of(I.grid_rewired(120, 120, 0.01, 1))
    job = P.Job(graph, 2, 1)
    job.tune(bidir_table=0, bidir_warps=0)
    job.sample(8000)
    for m in (8000, 8000, 3000):
        other = P.Job(graph, 2, 1)
        other.sample(m)
        h, ref = other.samples(), job.samples()
        members = int(h["hoff"][-1])
        assert all(np.array_equal(h[key], ref[key][:len(h[key])]) for key in ("hoff", "s", "t", "d"))
        assert np.array_equal(h["hmem"], ref["hmem"][:members])
    assert other.sampler_info()["migrated"] == 0
    last = P.Job(graph, 2, 1)
    last.sample(8000)
    assert last.stats()["bidir"]["launches"] == 2 and last.sampler_info()["migrated"] > 3000
