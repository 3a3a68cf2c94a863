"""Performance cases of the G-ES-MC library: what a user's program does with
it, through its public entry points, from a graph of a few thousand edges to
one of 1.3e8.

A program that samples graphs with a prescribed degree sequence keeps a chain
(or a pool of chains, or a server) on the GPU, advances it by some global
switches or ES-MC switches, and reads the edge list: one pass here.  A pass
can be repeated; the chain then moves on, as in a program that takes every
k-th state of a chain as a sample.  Every output is a list of packed edge ids
(whole numbers), so every case is compared exactly and no case has a 64-bit
reference.

Kinds of cases:
  chain    Chain.run(rounds, seed), Chain.edges(out on the GPU)
  noalloc  gesmc_run_noalloc in place on a list on the GPU
  sample   a whole request of a program that has a graph in host memory:
           Chain(edges), run, edges (back to host memory), close
  pool     Pool.run(rounds), Pool.edges of every chain
  es       Chain.es_run(switches, seed), Chain.edges
  es_pool  Pool.es_run(switches), Pool.edges of every chain
  serve    Server.submit of a batch of requests, steps until idle
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2111_03005_gb300 import gesmc, inputs, serve

LAZY_HALF = 1 << 63  # P_L = 1/2


def listed():
    return [
        # the smallest graph of the benchmark, ten global switches a sample, the
        # chain in one SM's shared memory: launches and latency are what count
        {"name": "chain_gnp_1k_resident", "kind": "chain", "graph": "gnp", "n": 1000, "degree": 9.99, "rounds": 10,
         "launch": "resident", "lazy": "none"},
        # the same graph with the options as they come (a graph of kernels per round)
        {"name": "chain_gnp_1k", "kind": "chain", "graph": "gnp", "n": 1000, "degree": 9.99, "rounds": 10,
         "launch": "kernels", "lazy": "none"},
        # a small network with hubs, every switch lazy with probability 1/2 (the
        # chain as the paper's Def. 2 states it), one cooperative launch a round
        {"name": "chain_pld_10k_lazy", "kind": "chain", "graph": "pld", "n": 7301, "gamma": 2.2, "rounds": 20,
         "launch": "one", "lazy": "switch"},
        # a caller that owns all device memory, a graph of about 2e4 edges
        {"name": "noalloc_gnp_5k", "kind": "noalloc", "graph": "gnp", "n": 5003, "degree": 8.0, "rounds": 5},
        # the power-law graph of the benchmark (10^6 nodes, degrees up to 1000):
        # hubs, several waves a round
        {"name": "chain_pld_1m", "kind": "chain", "graph": "pld", "n": 1_000_000, "gamma": 2.5, "dmax": 1000,
         "rounds": 20, "launch": "kernels", "lazy": "none"},
        # the benchmark's large graph, 1.34e8 edges: bandwidth and L2 operations
        {"name": "chain_gnp_2p24", "kind": "chain", "graph": "gnp", "n": 1 << 24, "degree": 16.0, "rounds": 5,
         "launch": "kernels", "lazy": "none"},
        # one sample of a graph in host memory, from the list to the list
        {"name": "sample_pld_1m", "kind": "sample", "graph": "pld", "n": 600_011, "gamma": 2.3, "rounds": 20},
        # a null-model ensemble of graphs of uneven size, half G(n, p), half power
        # law, 50 global switches a sample as in the benchmark
        {"name": "pool_mixed_256", "kind": "pool", "chains": 256, "n_lo": 100, "n_hi": 100_000, "rounds": 50,
         "launch": "kernels"},
        # an ensemble of small graphs, one CTA per chain
        {"name": "pool_small_1024", "kind": "pool", "chains": 1024, "n_lo": 100, "n_hi": 2400, "rounds": 50,
         "launch": "resident"},
        # ES-MC (single edge switches in order) on one chain of about 1e6 edges
        {"name": "es_gnp_1m", "kind": "es", "graph": "gnp", "n": 1 << 17, "degree": 16.0, "switches": 1 << 19},
        # ES-MC on an ensemble, the same number of switches per chain
        {"name": "es_pool_512", "kind": "es_pool", "chains": 512, "n_lo": 100, "n_hi": 30_000, "switches": 1 << 14},
        # sampling requests of all sizes that arrive together, in three size classes
        {"name": "serve_24", "kind": "serve", "requests": 24, "m_lo": 1000, "m_hi": 1_000_000, "rounds_hi": 40},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["chain", "chain", "chain", "noalloc", "sample", "pool", "pool", "es", "es_pool", "serve"])
    if kind in ("pool", "es_pool"):
        small = rng.random() < 0.5
        n_hi = _log_uniform(rng, 200, 2400) if small else _log_uniform(rng, 3000, 100_000)
        # chains x n_hi bounds the edges of the pool (about those of 256 chains up to 1e5)
        chains = min(1024, max(2, _log_uniform(rng, 2, min(1024, 25_600_000 // n_hi))))
        case = {"kind": kind, "chains": chains, "n_lo": 100, "n_hi": n_hi}
        if kind == "pool":
            return {**case, "rounds": rng.randint(1, 50), "launch": "resident" if small else "kernels"}
        return {**case, "switches": _log_uniform(rng, 1 << 8, 1 << 14)}
    if kind == "serve":
        return {"kind": kind, "requests": rng.randint(2, 24), "m_lo": 1000, "m_hi": _log_uniform(rng, 10_000, 1_000_000),
                "rounds_hi": rng.randint(10, 40)}
    graph = rng.choice(["gnp", "pld"])
    case = {"kind": kind, "graph": graph}
    if graph == "gnp":
        degree = round(rng.uniform(4.0, 24.0), 2)
        per_node = degree / 2
        case["degree"] = degree
    else:
        gamma = round(rng.uniform(2.2, 3.0), 2)
        per_node = 1.0  # about 0.7 to 1.6 edges per node
        case["gamma"] = gamma
    if kind == "noalloc":
        return {**case, "n": int(_log_uniform(rng, 500, 32_000) / per_node), "rounds": rng.randint(1, 10)}
    if kind == "sample":
        return {**case, "n": int(_log_uniform(rng, 1000, 1_000_000) / per_node), "rounds": rng.randint(10, 20)}
    if kind == "es":
        return {**case, "n": int(_log_uniform(rng, 1000, 2_000_000) / per_node),
                "switches": _log_uniform(rng, 1 << 10, 1 << 19)}
    m = _log_uniform(rng, 1000, 6_000 if rng.random() < 0.3 else (100_000_000 if graph == "gnp" else 1_500_000))
    launch = "resident" if m <= 6000 and rng.random() < 0.5 else "one" if m <= 50_000 and rng.random() < 0.5 else "kernels"
    return {**case, "n": max(50, int(m / per_node)), "rounds": rng.randint(1, max(1, min(20, 600_000_000 // m))),
            "launch": launch, "lazy": rng.choice(["none", "none", "switch", "exact"])}


# ---------------------------------------------------------------- graphs
def _dmax(case):
    """Largest degree of a power-law graph: as given, else n^(1 / (gamma - 1)) (the paper's choice)."""
    n = case["n"]
    return case.get("dmax") or max(1, min(n - 1, int(n ** (1.0 / (case["gamma"] - 1.0)))))


def _edges_of(case):
    """Expected number of edges of a case's graph."""
    if case["graph"] == "gnp":
        return case["n"] * case["degree"] / 2
    return case["n"] * inputs.pld_mean_degree(case["gamma"], 1, _dmax(case)) / 2


def _relabelled(edges, n, seed):
    """The same graph with its nodes renamed and its edges listed in another
    order: the list of another user with the same degrees."""
    rng = np.random.default_rng(seed)
    name = rng.permutation(n).astype(np.uint64)
    a, b = name[edges >> np.uint64(32)], name[edges & np.uint64(0xFFFFFFFF)]
    return rng.permutation((np.minimum(a, b) << np.uint64(32)) | np.maximum(a, b))


def _gnp_extra(case):
    """(edges m of the case's random graph, p of a G(n, p) that has more than m)."""
    m = int(_edges_of(case))
    return m, (m + 8 * math.sqrt(m) + 32) / (case["n"] * (case["n"] - 1) / 2)


def _host_graph(case, seed):
    """A uniform random graph of a fixed number of edges (G(n, p) without its
    excess edges), or a power-law degree sequence that the case fixes,
    realised, with nodes and list order from the seed."""
    if case["graph"] == "gnp":
        m, p = _gnp_extra(case)
        edges = inputs.gnp(case["n"], p, seed)
        return np.random.default_rng(seed).permutation(edges)[:m]
    return _relabelled(inputs.graphical_pld_graph(case["n"], case["gamma"], _dmax(case), 2), case["n"], seed)


def _gpu_graph(case, seed):
    if case["graph"] == "gnp":
        m, p = _gnp_extra(case)
        edges = gesmc.generate_gnp(case["n"], p, seed)
        keep = torch.ones(edges.numel(), dtype=torch.bool, device="cuda")
        drop = np.random.default_rng(seed).choice(edges.numel(), edges.numel() - m, replace=False, shuffle=False)
        keep[torch.from_numpy(drop).cuda()] = False
        return edges[keep]
    return torch.from_numpy(_host_graph(case, seed).view(np.int64)).cuda()


def _ensemble(case):
    """The graphs of a pool: n spread over [n_lo, n_hi] on a logarithmic scale
    in mixed order, even ones G(n, 8 / (n - 1)), odd ones power law with
    exponents from 2.2 to 3.0."""
    out, count = [], case["chains"]
    for t in range(count):
        u = (t * 0.6180339887498949 + 0.5) % 1.0
        n = int(round(case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** u))
        if t % 2 == 0:
            out.append({"graph": "gnp", "n": n, "degree": 8.0})
        else:
            out.append({"graph": "pld", "n": n, "gamma": 2.2 + 0.8 * ((t * 0.7548776662466927) % 1.0)})
    return out


def _requests(case):
    """Sizes and rounds of the requests of a batch, both spread over their ranges in mixed order."""
    out = []
    for t in range(case["requests"]):
        u = (t * 0.6180339887498949 + 0.5) % 1.0
        v = (t * 0.7548776662466927 + 0.5) % 1.0
        out.append((int(case["m_lo"] * (case["m_hi"] / case["m_lo"]) ** u), 10 + int(v * (case["rounds_hi"] - 9))))
    return out


# ---------------------------------------------------------------- prepare
def _lazy_options(case):
    if case["lazy"] == "none":
        return {}
    return {"lazy_threshold": LAZY_HALF, "exact_ell": case["lazy"] == "exact"}


_LAUNCH = {"kernels": 0, "one": 32, "resident": gesmc.ROUND_RESIDENT}


def prepare(case, seed):
    kind = case["kind"]
    state = {"case": case, "seed": seed}
    if kind in ("chain", "es"):
        edges = _gpu_graph(case, seed)
        options = _lazy_options(case) if kind == "chain" else {}
        state["chain"] = gesmc.Chain(edges, n=case["n"], **options)
        if kind == "chain" and case["launch"] != "kernels":
            state["chain"].set_round_launch(_LAUNCH[case["launch"]])
        state["out"] = torch.empty_like(edges)
    elif kind == "noalloc":
        state["edges"] = _gpu_graph(case, seed)
        state["round"] = 0
    elif kind == "sample":
        state["edges"] = _host_graph(case, seed)
    elif kind in ("pool", "es_pool"):
        graphs = [(_host_graph(g, seed + 7919 * t), g["n"]) for t, g in enumerate(_ensemble(case))]
        total = sum(len(e) for e, _ in graphs)
        pool = gesmc.Pool(max_edges=total, max_chains=len(graphs))
        out = torch.empty(total, dtype=torch.int64, device="cuda")
        at, chains = 0, []
        for t, (e, n) in enumerate(graphs):
            chains.append((pool.add(e, n=n, seed=seed * 1000003 + t), out[at:at + len(e)]))
            at += len(e)
        if case.get("launch", "kernels") != "kernels":
            pool.set_round_launch(_LAUNCH[case["launch"]])
        state.update(pool=pool, chains=chains, out=out)
    else:
        requests = []
        for t, (m, rounds) in enumerate(_requests(case)):
            edges, n = inputs.request_graph(m, 7919 * t + 1)
            requests.append((_relabelled(edges, n, seed + t), n, seed * 1000003 + t, rounds))
        state["requests"] = requests
        total = sum(len(r[0]) for r in requests)
        state["server"] = serve.Server(max_edges=total, max_chains=len(requests), size_classes=(10_240, 131_072),
                                       small_round_ctas=gesmc.ROUND_RESIDENT)
    return state


# ---------------------------------------------------------------- run
def run(state):
    case, seed = state["case"], state["seed"]
    kind = case["kind"]
    if kind == "chain":
        return state["chain"].run(case["rounds"], seed).edges(state["out"])
    if kind == "es":
        return state["chain"].es_run(case["switches"], seed).edges(state["out"])
    if kind == "noalloc":
        gesmc.gesmc_run_noalloc(state["edges"], case["n"], case["rounds"], seed, start_round=state["round"])
        state["round"] += case["rounds"]
        return state["edges"]
    if kind == "sample":
        with gesmc.Chain(state["edges"], n=case["n"]) as chain:
            return chain.run(case["rounds"], seed).edges()
    if kind in ("pool", "es_pool"):
        pool = state["pool"]
        if kind == "pool":
            pool.run(case["rounds"])
        else:
            pool.es_run(case["switches"])
        for chain, out in state["chains"]:
            pool.edges(chain, out)
        return state["out"]
    server = state["server"]
    requests = [serve.Request(rid=t, edges=e, n=n, seed=s, rounds=r)
                for t, (e, n, s, r) in enumerate(state["requests"])]
    for request in requests:
        server.submit(request)
    while not server.idle():
        server.step()
    return [request.result for request in requests]


# ---------------------------------------------------------------- work and tolerance
def work(case):
    """A round reads the list and writes it (8 bytes an edge each); an ES-MC
    switch reads two edges and writes two; the list is read and written once
    more to give it to the caller (from and to host memory it is read and
    written once more on the way in)."""
    kind = case["kind"]
    if kind in ("pool", "es_pool"):
        m = sum(_edges_of(g) for g in _ensemble(case))
        moved = 16 * m * case["rounds"] if kind == "pool" else 32 * case["switches"] * case["chains"]
        return {"bytes": moved + 16 * m, "flops": 0}
    if kind == "serve":
        return {"bytes": sum(16 * m * (rounds + 2) for m, rounds in _requests(case)), "flops": 0}
    m = _edges_of(case)
    if kind == "es":
        return {"bytes": 32 * case["switches"] + 16 * m, "flops": 0}
    extra = {"chain": 1, "noalloc": 0, "sample": 2}[kind]
    return {"bytes": 16 * m * (case["rounds"] + extra), "flops": 0}


def tolerance(case):
    # lists of edge ids: whole numbers, the same for every correct implementation
    return "exact"
