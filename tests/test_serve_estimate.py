"""The serving loop's memory estimate covers the arrays that a job holds for each sample and each node."""
from paper_2306_03651_gb300 import serve


def est(n, t, m, **kw):
    return serve.estimate_job_bytes(n, 8 * n, t, m, **kw)


def test_every_array_of_a_sample_is_counted():
    t, members = 40, 6
    # offset, pair and distance, sign words; members, their incidence and places; five lists of a call's samples
    each = 8 + 12 + 4 * 2 + 3 * 4 * members + 5 * 8
    assert est(2000, t, 2 << 20, avg_hyperedge=members) - est(2000, t, 1 << 20, avg_hyperedge=members) >= each << 20


def test_every_array_of_a_node_is_counted():
    t, n = 10, 2_000_000
    waves = 24 * 2 * 32  # a node's share of the wave workspace without its levels
    # R of all nodes and c; counts, offsets, gains and those left, list entries; all nodes' list, counts and chunks
    each = 4 * (t + 1) + 4 + 8 + 4 + 4 + 4 + 4 + 4 + 8
    assert est(n + 1000, t, 1000, levels=-6) - est(n, t, 1000, levels=-6) >= 1000 * (waves + each)


def test_the_first_arena_is_counted():
    """64 members a sample up to 2^24 entries, whatever the mean."""
    few, many = (est(2000, 10, m, avg_hyperedge=0.0) for m in (0, 1 << 18))
    assert many - few >= 4 * (1 << 24)
