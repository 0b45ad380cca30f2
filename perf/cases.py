"""Workloads of the library as a user's program runs them, for timing and for comparing results.

A case is a plain dict.  ``kind`` says which calls a pass makes:

  round     one round of Algorithm 1 on a resident graph: a new job, cen_sample, greedyCover beside the AMCERA, bounds
  load      the same on a graph that the pass uploads from pinned host memory first
  certify   Algorithm 1 to its certificate (cen_run_ex) on a resident graph
  batch     several certified runs of uneven size side by side (cen_run_batch)
  canon     a raw arc list on the device made into the canonical CSR (cen_graph_load_ex), read back on the device
  walks     kappa-path hyper-edges drawn and read back

``keep``: the program also reads the round's hyper-edges back, into pinned buffers that it owns, to judge other node
sets on the same sample later.

Graphs are made on the GPU from the seed alone, with the shapes of the paper's networks: Barabasi-Albert ("ba"),
R-MAT with (.57, .19, .19, .05) undirected with its largest component kept ("rmat") or directed ("rmatd"), and a
4-neighbour grid with 1% of its edges rewired ("grid").  Each state has its own graph and its own job seed.
"""
import math

import numpy as np
import torch

import paper_2306_03651_gb300 as P
from paper_2306_03651_gb300 import inputs

SPACES = {"paths": P.SPACE_BETWEENNESS, "kpath": P.SPACE_KPATH, "triangle": P.SPACE_TRIANGLE}


def listed():
    return [
        # The smallest call: the first round on a graph of 2,000 nodes.  Launches, synchronisations and host work.
        {"name": "round-ba2k", "kind": "round", "graph": "ba", "n": 2000, "d": 4, "space": "paths", "m": 1000,
         "k": 10, "t": 10, "keep": False},
        # The same graph to its certificate from 1,000 pairs, doubling: a whole small problem, nine or so rounds.
        {"name": "certify-ba2k", "kind": "certify", "graph": "ba", "n": 2000, "d": 4, "k": 10, "t": 10, "eps": 0.05,
         "delta": 0.1, "plan": "doubling"},
        # An ordinary round: a social network of com-dblp's size, hubs, the default number of sign vectors.
        {"name": "round-rmat18", "kind": "round", "graph": "rmat", "scale": 18, "ef": 16, "space": "paths",
         "m": 65536, "k": 50, "t": 10, "keep": True},
        # The same network to its certificate in the fewest rounds: millions of samples, the store growing.
        {"name": "certify-rmat18", "kind": "certify", "graph": "rmat", "scale": 18, "ef": 16, "k": 50, "t": 10,
         "eps": 0.02, "delta": 0.1, "plan": "predicting"},
        # A large directed network (soc-LiveJournal1's size), many sign vectors over 4.2 million nodes.
        {"name": "round-rmat22d", "kind": "round", "graph": "rmatd", "scale": 22, "ef": 16, "space": "paths",
         "m": 65536, "k": 100, "t": 100, "keep": True},
        # High diameter: deep searches of tens of levels, long hyper-edges, 4.2 million nodes.
        {"name": "round-grid2048", "kind": "round", "graph": "grid", "w": 2048, "h": 2048, "space": "paths",
         "m": 16384, "k": 100, "t": 100, "keep": True},
        # A program that is handed a directed graph and wants one estimate: the upload and the in-arc CSR count.
        {"name": "load-rmat20d", "kind": "load", "graph": "rmatd", "scale": 20, "ef": 16, "space": "paths",
         "m": 16384, "k": 50, "t": 10, "keep": False},
        # Raw arcs with repeats and self-loops, as a data set comes, made canonical and undirected.
        {"name": "canon-rmat20", "kind": "canon", "scale": 20, "ef": 8, "symmetrize": True},
        # The kappa-path walks of the network, read back for use outside the library.
        {"name": "walks-rmat18", "kind": "walks", "graph": "rmat", "scale": 18, "ef": 16, "m": 65536, "kappa": 8},
        # Triangle centrality, one round (a graph's triangle ranks are kept on it after its first such job).
        {"name": "triangle-rmat16", "kind": "round", "graph": "rmat", "scale": 16, "ef": 16, "space": "triangle",
         "m": 65536, "k": 50, "t": 10, "keep": True},
        # Several users' graphs of uneven size at once, each to its certificate.
        {"name": "batch-ba8", "kind": "batch", "jobs": 8, "n_low": 10000, "n_high": 100000, "t": 32, "eps": 0.05,
         "delta": 0.1, "workers": 8},
        # Many sign vectors over a large sample (the study of the bound's dependence on t).
        {"name": "round-rmat16-t256", "kind": "round", "graph": "rmat", "scale": 16, "ef": 16, "space": "paths",
         "m": 262144, "k": 100, "t": 256, "keep": True},
    ]


def _log_int(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def _draw_graph(rng, kinds):
    g = rng.choice(kinds)
    if g == "ba":
        return {"graph": g, "n": _log_int(rng, 300, 200000), "d": rng.randint(2, 8)}
    if g == "grid":
        return {"graph": g, "w": _log_int(rng, 40, 1500), "h": _log_int(rng, 40, 1500)}
    return {"graph": g, "scale": rng.randint(11, 18 if g == "rmat" else 21), "ef": rng.randint(6, 16)}


def draw(rng):
    kind = rng.choice(["round", "round", "round", "round", "load", "certify", "canon", "walks", "triangle", "batch"])
    k, t = rng.randint(5, 200), rng.choice([1, 10, 32, 100, rng.randint(1, 128)])
    if kind in ("round", "load"):
        g = _draw_graph(rng, ["ba", "rmat", "rmatd", "grid"])
        m = _log_int(rng, 300, 8192 if g["graph"] == "grid" else 65536)
        return {"kind": kind, **g, "space": "paths", "m": m, "k": k, "t": t, "keep": rng.random() < 0.5}
    if kind == "triangle":
        g = _draw_graph(rng, ["ba", "rmat"])
        if g["graph"] == "rmat":
            g["scale"] = min(g["scale"], 16)
        return {"kind": "round", **g, "space": "triangle", "m": _log_int(rng, 300, 65536), "k": k, "t": t,
                "keep": rng.random() < 0.5}
    if kind == "walks":
        return {"kind": kind, **_draw_graph(rng, ["ba", "rmat", "rmatd", "grid"]), "m": _log_int(rng, 300, 65536),
                "kappa": rng.randint(2, 16)}
    if kind == "certify":
        g = _draw_graph(rng, ["ba", "rmat"])
        return {"kind": kind, **g, "k": rng.randint(5, 100), "t": t, "eps": round(rng.uniform(0.05, 0.2), 3),
                "delta": 0.1, "plan": rng.choice(["doubling", "predicting"])}
    if kind == "canon":
        return {"kind": kind, "scale": rng.randint(11, 20), "ef": rng.randint(2, 8),
                "symmetrize": rng.random() < 0.5}
    return {"kind": "batch", "jobs": rng.randint(2, 8), "n_low": 2000, "n_high": _log_int(rng, 10000, 100000), "t": 32,
            "eps": round(rng.uniform(0.06, 0.2), 3), "delta": 0.1, "workers": rng.randint(2, 8)}


# ------------------------------------------------------------------ graphs
def _rmat_arcs(scale, ef, gen):
    """ef * 2^scale R-MAT draws as (tail, head), repeats and self-loops included."""
    a, b, c = 0.57, 0.19, 0.19
    ne = ef << scale
    src = torch.zeros(ne, dtype=torch.int64, device="cuda")
    dst = torch.zeros(ne, dtype=torch.int64, device="cuda")
    for _ in range(scale):
        u = torch.rand(ne, generator=gen, device="cuda")
        low = u >= a + b  # the lower half of the adjacency matrix
        src = 2 * src + low
        dst = 2 * dst + (((u >= a) & ~low) | (u >= a + b + c))
    return src, dst


def _csr(n, src, dst, symmetric):
    """Canonical CSR of an arc list: rows ascending, no repeats, no self-loops."""
    key = src * n + dst
    if symmetric:
        key = torch.cat([key, dst * n + src])
    key = torch.unique(key)
    src, dst = key // n, key % n
    keep = src != dst
    src, dst = src[keep], dst[keep]
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(torch.bincount(src, minlength=n), 0)
    return off, dst.to(torch.int32), src


def _largest_component(n, off, col, src):
    """The component of the node of most neighbours, relabelled in id order (for R-MAT graphs, the largest)."""
    label = torch.zeros(n, dtype=torch.bool, device="cuda")
    label[torch.argmax(off[1:] - off[:-1])] = True
    count = 0
    while int(label.sum()) != count:
        count = int(label.sum())
        label[col[label[src]].long()] = True
    new = torch.cumsum(label, 0) - 1
    keep = label[src]
    src, dst = new[src[keep]], new[col[keep].long()]
    off = torch.zeros(count + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(torch.bincount(src, minlength=count), 0)
    return count, off, dst.to(torch.int32)


def _graph(case, seed):
    """(n, off, col, directed): device tensors, or host arrays for "ba"."""
    if case["graph"] == "ba":
        g = inputs.ba(max(case["n"], case["d"] + 2), case["d"], 1 + seed)
        return g.n, g.off, g.col, False
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if case["graph"] == "grid":
        w, h = case["w"], case["h"]
        ids = torch.arange(w * h, device="cuda").view(h, w)
        src = torch.cat([ids[:, :-1].reshape(-1), ids[:-1].reshape(-1)])
        dst = torch.cat([ids[:, 1:].reshape(-1), ids[1:].reshape(-1)])
        moved = torch.rand(src.numel(), generator=gen, device="cuda") < 0.01
        dst = torch.where(moved, torch.randint(0, w * h, dst.shape, generator=gen, device="cuda"), dst)
        off, col, _ = _csr(w * h, src, dst, True)
        return w * h, off, col, False
    n, directed = 1 << case["scale"], case["graph"] == "rmatd"
    src, dst = _rmat_arcs(case["scale"], case["ef"], gen)
    off, col, src = _csr(n, src, dst, not directed)
    if directed:
        return n, off, col, True
    n, off, col = _largest_component(n, off, col, src)
    return n, off, col, False


def _batch_params(case):
    """Sizes and k of the jobs of a batch: spread evenly over the logarithm of the range, k cycling 10, 50, 100."""
    low, high, jobs = math.log(case["n_low"]), math.log(case["n_high"]), case["jobs"]
    return [(int(round(math.exp(low + (high - low) * (i + 0.5) / jobs))), 2 + i % 7, (10, 50, 100)[i % 3])
            for i in range(jobs)]


# ------------------------------------------------------------------ a user's program
def _buffers(case):
    """The program's pinned buffers for the hyper-edges of m samples, with room for the longest that the case draws."""
    m, room = case["m"], case.get("kappa") or (256 if case["graph"] == "grid" else 32)
    rows = {key: torch.zeros(m, dtype=torch.int32).pin_memory() for key in ("s", "t", "d")}
    return {"hoff": torch.zeros(m + 1, dtype=torch.int64).pin_memory(),
            "hmem": torch.zeros(m * room, dtype=torch.int32).pin_memory(), **rows}


def prepare(case, seed):
    state = {"case": case, "seed": 1 + 7919 * seed}
    kind = case["kind"]
    if kind == "batch":
        state["jobs"] = []
        for i, (n, d, k) in enumerate(_batch_params(case)):
            g = P.Graph.of(inputs.ba(n, d, 1 + 64 * seed + i))
            state["jobs"].append(dict(graph=g, k=k, eps=case["eps"], delta=case["delta"], t=case["t"],
                                      seed=state["seed"] + i, m0=1000, schedule=P.SCHEDULE_DOUBLING))
    elif kind == "canon":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        src, dst = _rmat_arcs(case["scale"], case["ef"], gen)
        src, order = torch.sort(src, stable=True)  # rows of an unsorted CSR, heads in draw order
        n = 1 << case["scale"]
        state["n"] = n
        state["off"] = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
        state["off"][1:] = torch.cumsum(torch.bincount(src, minlength=n), 0)
        state["col"] = dst[order].to(torch.int32)
        state["off_out"] = torch.zeros_like(state["off"])
        state["col_out"] = torch.zeros(_most_arcs(case), dtype=torch.int32, device="cuda")
    else:
        n, off, col, directed = _graph(case, seed)
        if kind == "load":  # what the program holds is in pinned host memory
            off, col = (torch.as_tensor(x).cpu().pin_memory() for x in (off, col))
            state.update(n=n, off=off, col=col, directed=directed)
        else:
            state["graph"] = P.Graph(n, off, col, directed)
        if kind == "walks" or case.get("keep"):
            state["buffers"] = _buffers(case)
    torch.cuda.synchronize()
    return state


def _most_arcs(case):
    return (case["ef"] << case["scale"]) * (2 if case["symmetrize"] else 1)


def _padded(values, size):
    out = np.full(size, -1, np.int32)
    out[: len(values)] = values
    return out


def _read_back(job, buffers):
    if job.size()[1] > buffers["hmem"].numel():
        raise RuntimeError("hyper-edges longer than the program's buffer")
    rc = P.cen_job_copy_samples(job.h, *(buffers[key].data_ptr() for key in ("hoff", "hmem", "s", "t", "d")))
    if rc != P.OK:
        raise RuntimeError(P.last_error())
    return buffers


def _round(graph, state):
    case = state["case"]
    job = P.Job(graph, state["seed"], case["t"], space=SPACES[case["space"]])
    job.sample(case["m"])
    S, covered, Rnum, Wnum, b = job.cover_and_mcera(case["k"])
    stop, bounds = P.bounds(covered, case["m"], int(Rnum.sum()), case["t"], Wnum, b, 0.01, 0.1, 1)
    out = {"S": _padded(S, case["k"]), "covered": covered, "Rnum": Rnum, "Wnum": Wnum, "b": b, "stop": stop,
           "bounds": bounds}
    if case["keep"]:
        out["sample"] = _read_back(job, state["buffers"])
    job.close()
    return out


def _certified(r, k):
    log = np.zeros((64, r["log"].shape[1]))
    log[: len(r["log"])] = r["log"]
    return {"S": _padded(r["S"], k), "log": log, **{key: r[key] for key in ("status", "covered", "m_final", "rounds")}}


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "round":
        return _round(state["graph"], state)
    if kind == "load":
        graph = P.Graph(state["n"], state["off"].numpy(), state["col"].numpy(), state["directed"])
        out = _round(graph, state)
        graph.close()
        return out
    if kind == "certify":
        plan = P.SCHEDULE_DOUBLING if case["plan"] == "doubling" else P.SCHEDULE_EXTRAPOLATE
        return _certified(P.run(state["graph"], case["k"], case["eps"], case["delta"], case["t"], state["seed"],
                                m0=1000, schedule=plan), case["k"])
    if kind == "batch":
        jobs = state["jobs"]
        return [_certified(r, j["k"]) for j, r in zip(jobs, P.run_batch(jobs, nworkers=case["workers"]))]
    if kind == "canon":
        flags = P.GRAPH_CANONICALIZE | (P.GRAPH_SYMMETRIZE if case["symmetrize"] else 0)
        graph = P.Graph(state["n"], state["off"], state["col"], directed=not case["symmetrize"], flags=flags)
        rc = P.cen_graph_copy(graph.h, state["off_out"].data_ptr(), state["col_out"].data_ptr())
        nnz = graph.nnz
        graph.close()
        if rc != P.OK:
            raise RuntimeError(P.last_error())
        return {"off": state["off_out"], "col": state["col_out"], "nnz": nnz}
    job = P.Job(state["graph"], state["seed"], 1, space=P.SPACE_KPATH, kappa=case["kappa"])
    job.sample(case["m"])
    out = _read_back(job, state["buffers"])
    job.close()
    return out


def exact(case, seed):
    """The canonical CSR by sorting 64-bit arc keys.  The other kinds return whole numbers and FP64 functions of them
    that follow from a full run of the method, which takes longer than a check may in plain numpy or torch."""
    if case["kind"] != "canon":
        return None
    state = prepare(case, seed)
    n, off = state["n"], state["off"]
    src = torch.repeat_interleave(torch.arange(n, device="cuda"), off[1:] - off[:-1])
    off, col, _ = _csr(n, src, state["col"].long(), case["symmetrize"])
    out = torch.zeros_like(state["col_out"])
    out[: col.numel()] = col
    return {"off": off, "col": out, "nnz": col.numel()}


# ------------------------------------------------------------------ what a pass cannot do without
def _graph_size(case):
    """(nodes, arcs) of a case's graph, near enough: R-MAT draws lose some 7% to repeats."""
    if case["graph"] == "ba":
        return case["n"], 2 * case["n"] * case["d"]
    if case["graph"] == "grid":
        return case["w"] * case["h"], 4 * case["w"] * case["h"]
    n, arcs = 1 << case["scale"], int(0.93 * (case["ef"] << case["scale"]))
    return n, 2 * arcs if case["graph"] == "rmat" else arcs


def work(case):
    """The graph (or the arcs) read once and the results written once: hyper-edges (28 bytes of offset, pair, distance
    and sign words each, and four bytes a member) for the kinds that draw them.  All arithmetic is on whole numbers."""
    kind = case["kind"]
    if kind == "canon":
        raw, n = case["ef"] << case["scale"], 1 << case["scale"]
        return {"bytes": 4 * raw + 8 * n + 8 * n + 4 * raw * (2 if case["symmetrize"] else 1), "flops": 0}
    if kind == "batch":
        sizes = [(n, 2 * n * d) for n, d, _ in _batch_params(case)]
        return {"bytes": sum(8 * n + 4 * a + 28 * 20000 for n, a in sizes), "flops": 0}
    n, arcs = _graph_size(case)
    members = 30 if case["graph"] == "grid" else 3
    m = case.get("m", 20000)
    return {"bytes": 8 * n + 4 * arcs + m * (28 + 4 * members), "flops": 0}
