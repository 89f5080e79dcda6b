"""Performance cases: what users of this framework run, over the sizes they run it at.

A case is a plain dict.  ``prepare`` builds what a program holds before the call (graph handle, input
tensors, caches, search handles), ``run`` is one pass through the public entry points.  All inputs are
synthetic and seeded; every quantity on these paths is an integer, so results are compared exactly.

Kinds
  eval       Graph.eval_batch: candidate sequences scored on the device (the inner call of any search)
  host       Graph.eval_batch_host / _host16: the same for sequences that a host program produced
  profile    Graph.mem_profile: memory profile and free steps of one sequence, for a report or a plot
  search     Search.run: generations of the device-resident local search, then the chains' state
  edits      EditCache.build / eval_edits: single edits of evaluated sequences (large neighbourhood steps)
  intervals  Graph.check_intervals: solutions of a constraint solver checked in interval form
"""
from __future__ import annotations

import math
import zlib

import numpy as np
import torch

from paper_2304_14463_b200 import binding, workloads

BUDGET_PCT = 80


def _case(name, kind, graph, n, B, **more):
    c = dict(kind=kind, graph=graph, n=n, edges=0, layers=0, C=2, p=0.2, B=B, mu=6.0, sigma=1.5, scale=1, damaged=0.0)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a toy or unit-sized graph in a driver loop: the call itself is what counts
        _case("eval_n20_b1024", "eval", "layered", 20, 1024, edges=40, layers=4, p=0.5, mu=4.0, sigma=0.5),
        # small published random-layered graph, large population
        _case("eval_n100_b65536", "eval", "layered", 100, 65536, edges=236, layers=10, mu=4.0, sigma=1.0),
        # the benchmark configuration: real-world training graph
        _case("eval_n442_b16384", "eval", "training", 442, 16384),
        # a convolutional network with its backward pass, three copies per node
        _case("eval_n1000_c3_b4096", "eval", "resnet", 1000, 4096, C=3, p=0.3, mu=7.0),
        # the largest configuration
        _case("eval_n5000_c3_b1024", "eval", "layered", 5000, 1024, edges=15000, layers=50, C=3, p=0.3, mu=8.0, sigma=2.0),
        # sizes in bytes (64-bit sums), an odd number of candidates, some of which a search step broke
        _case("eval_n353_bytes_b1501", "eval", "layered", 353, 1501, edges=751, layers=19, scale=4096, damaged=0.0625),
        # sequences from a host program, node ids as 16-bit words in pinned memory
        _case("host16_n442_b16384", "host", "training", 442, 16384, bits=16),
        # one sequence in full detail
        _case("profile_n442", "profile", "training", 442, 1),
        # local search, one proposal per chain and generation, a population of moderate size
        _case("search_n442_p4096", "search", "training", 442, 4096, samples=1, generations=20),
        # local search, many proposals per chain scored from the cached evaluation, a large population
        _case("search_n442_p32768_e32", "search", "training", 442, 32768, samples=32, generations=10),
        # parents evaluated and cached, then 16 edits of each
        _case("edits_n442_p16384", "edits", "training", 442, 16384, per_parent=16, build=True),
        # solver output checked against the model, plain event domain
        _case("intervals_n442_b16384", "intervals", "training", 442, 16384, staged=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eval"] * 6 + ["host", "profile", "search", "search", "edits", "intervals"])
    n = _log_int(rng, 20, 5000 if kind in ("eval", "host", "profile") else 1000)
    graph = rng.choice(["layered", "training", "resnet"]) if n >= 40 else "layered"
    C = rng.choice([2, 2, 2, 2, 2, 2, 3, 3, 3, 4]) if kind in ("eval", "host", "profile") else 2
    p = round(rng.uniform(0.05, 0.4), 3)
    more = dict(C=C, p=p, mu=round(rng.uniform(4.0, 8.0), 2), sigma=round(rng.uniform(0.5, 2.0), 2))
    if graph == "layered":
        more.update(edges=int(n * rng.uniform(2.0, 4.0)), layers=max(4, min(50, int(math.sqrt(n)))))
    else:
        n -= n % 2
    if rng.random() < 0.25:
        more["scale"] = 4096
    steps = n * (1 + (C - 1) * p)

    def batch(most_steps, most):
        """Number of sequences: total steps spread over a logarithmic scale."""
        return max(1, min(most, int(_log_int(rng, 20000, most_steps) / steps)))

    if kind == "eval":
        B = batch(7_500_000, 65536)
        more["damaged"] = rng.choice([0.0, 0.0, 0.0625])
    elif kind == "host":
        B = batch(7_500_000, 65536)
        more["bits"] = rng.choice([16, 32])
    elif kind == "profile":
        B = 1
    elif kind == "search":
        B = batch(8_000_000, 32768)
        more["samples"] = rng.choice([1, 1, 8, 32])
        more["generations"] = rng.choice([5, 10, 20]) if more["samples"] == 1 else rng.choice([5, 10])
    elif kind == "edits":
        B = batch(7_500_000, 16384)
        more.update(per_parent=rng.choice([2, 4, 8, 16]), build=rng.random() < 0.5)
    else:
        B = batch(7_500_000, 16384)
        more["staged"] = rng.random() < 0.5
    return _case(None, kind, graph, n, B, **more)


# ---------------------------------------------------------------------------------- inputs

def _steps(case):
    """Steps of a typical sequence."""
    return min(case["n"] * (1 + (case["C"] - 1) * case["p"]), case["n"] * 2)


def _graph(case, seed):
    n = case["n"]
    if case["graph"] == "layered":
        edges = workloads.layered_dag(n, case["edges"], case["layers"], seed)
    elif case["graph"] == "training":
        F = n // 2
        edges = workloads.training_dag(F, int(round(F * 293 / 221)), 2, 8, seed)
    else:
        edges = workloads.resnet_dag(n // 2)
    w = workloads.weights_uniform(n, 1, 50, seed, 1)
    m = workloads.weights_lognormal(n, case["mu"], case["sigma"], seed, 2) * case["scale"]
    return edges, w, m


def _sequences(case, edges, seed):
    n, C, p = case["n"], case["C"], case["p"]
    if case["kind"] == "profile":  # first ops recomputed until the sequence has its usual length
        return workloads.schedules(n, edges, C, 1.0, 1, seed, t_cap=int(_steps(case)))
    seqs, lens = workloads.schedules(n, edges, C, p, case["B"], seed, t_cap=n * min(C, 2) if C > 2 else None)
    hurt = int(round(case["B"] * case["damaged"]))
    if hurt:  # two steps of the row exchanged: mostly a consumer in front of its producer
        r = np.random.default_rng(seed)
        rows = r.choice(case["B"], hurt, replace=False)
        offs = np.concatenate([[0], np.cumsum(lens, dtype=np.int64)])[rows]
        i = offs + r.integers(0, 1 << 30, hurt) % lens[rows]
        j = offs + r.integers(0, 1 << 30, hurt) % lens[rows]
        seqs[i], seqs[j] = seqs[j].copy(), seqs[i].copy()
    return seqs, lens


def _ends(starts, active, edges, D):
    """End of every active interval: the latest start of a consumer before the node's next active
    interval, else its own start (a sink's last interval lasts to the last step)."""
    B, n, C = starts.shape
    big = D + 1
    at = torch.where(active, starts, big)
    after = torch.cat([at[:, :, 1:], torch.full_like(at[:, :, :1], big)], 2)
    ends = torch.where(active, starts, 0)
    u, v = (torch.from_numpy(np.ascontiguousarray(edges[:, k])).to(starts.device).long() for k in (0, 1))
    for i in range(C):
        for j in range(C):
            t = at[:, v, j]
            t = torch.where((t > at[:, u, i]) & (t < after[:, u, i]) & (t < big), t, 0)
            ends[:, :, i].scatter_reduce_(1, u.expand(B, -1), t, "amax")
    sink = torch.ones(n, dtype=torch.bool, device=starts.device)
    sink[u] = False
    last_step = torch.where(active, starts, 0).amax((1, 2))[:, None, None]
    last = active & (after == big) & sink[None, :, None]
    return torch.where(last, last_step, ends)


def _intervals(case, edges, seed):
    """(s, e, a, D, topo_index) of valid solutions."""
    n, C, B, dev = case["n"], case["C"], case["B"], "cuda"
    g = torch.Generator(dev).manual_seed(seed)
    if case["staged"]:
        # node k first in stage k; with probability p once more in a later stage
        D = n * (n + 1) // 2
        k = torch.arange(1, n + 1, device=dev).expand(B, n)
        stage = k + 1 + (torch.rand((B, n), generator=g, device=dev) * (n - k)).long()
        again = (torch.rand((B, n), generator=g, device=dev) < case["p"]) & (stage <= n)
        s = torch.full((B, n, C), D, device=dev, dtype=torch.int64)
        s[:, :, 0] = k * (k + 1) // 2
        s[:, :, 1] = torch.where(again, stage * (stage - 1) // 2 + k, D)
        active = torch.stack([torch.ones_like(again), again], 2)
        e = torch.where(active, _ends(s, active, edges, D), D)
        topo = torch.arange(1, n + 1, dtype=torch.int32, device=dev)
    else:
        # event t = step t of a sequence; unused slots on the events behind its last step
        D, topo = C * n, None
        seqs, lens = (torch.from_numpy(x).to(dev).long() for x in _sequences(case, edges, seed))
        row = torch.repeat_interleave(torch.arange(B, device=dev), lens)
        offs = torch.cumsum(lens, 0) - lens
        t = torch.arange(len(seqs), device=dev) - offs[row] + 1
        key, order = torch.sort((row * n + seqs) * (D + 1) + t)
        node = key // (D + 1)
        first = torch.searchsorted(node, node)
        slot = torch.arange(len(seqs), device=dev) - first
        s = torch.zeros((B, n, C), device=dev, dtype=torch.int64)
        active = torch.zeros((B, n, C), device=dev, dtype=torch.bool)
        s.view(-1)[node * C + slot] = t[order]
        active.view(-1)[node * C + slot] = True
        spare = torch.cumsum((~active).view(B, -1), 1).view(B, n, C) + lens[:, None, None]
        s = torch.where(active, s, spare)
        e = torch.where(active, _ends(s, active, edges, D), s)
    return s.to(torch.int32).contiguous(), e.to(torch.int32).contiguous(), active.to(torch.int32).contiguous(), D, topo


def prepare(case, seed):
    seed = zlib.crc32(f"{case['kind']} {case['n']} {seed}".encode()) >> 1
    n, C, B = case["n"], case["C"], case["B"]
    edges, w, m = _graph(case, seed)
    G = binding.Graph(n, edges, w, m, C)
    st = dict(case=case, graph=G, M=workloads.budget_from_peak(G.no_remat_peak(), BUDGET_PCT))
    kind = case["kind"]
    if kind == "intervals":
        st["s"], st["e"], st["a"], st["D"], st["topo"] = _intervals(case, edges, seed)
        return st
    seqs, lens = _sequences(case, edges, seed)
    if kind == "host":
        st["seqs"] = torch.from_numpy(seqs.astype(np.uint16) if case["bits"] == 16 else seqs).pin_memory()
        st["lens"] = torch.from_numpy(lens).pin_memory()
        st["out"] = tuple(torch.zeros(B, dtype=d).pin_memory() for d in (torch.int64, torch.int64, torch.int32))
        return st
    st["seqs"], st["lens"] = torch.from_numpy(seqs).cuda(), torch.from_numpy(lens).cuda()
    if kind == "search":
        st["search"] = binding.Search(G, st["seqs"], st["lens"], st["M"], seed=seed)
        if case["samples"] > 1:
            st["search"].set_samples(case["samples"], True)
    elif kind == "edits":
        st["cache"] = binding.EditCache(G, B)
        st["cache"].build(st["seqs"], st["lens"], st["M"])
        g, count = torch.Generator("cuda").manual_seed(seed), B * case["per_parent"]

        def below(k):
            return (torch.rand(count, generator=g, device="cuda", dtype=torch.float64) * k).long()

        parent = torch.randperm(count, generator=g, device="cuda") % B
        T = st["lens"][parent].long()
        op = below(3)
        q = below(T)
        j = below(torch.where(op == 0, T + 1, T))
        st["edits"] = tuple(x.to(torch.int32) for x in (parent, op, q, j))
    return st


def run(state):
    case, G, M = state["case"], state["graph"], state["M"]
    kind = case["kind"]
    if kind == "eval":
        return G.eval_batch(state["seqs"], state["lens"], M)
    if kind == "host":
        call = G.eval_batch_host16 if case["bits"] == 16 else G.eval_batch_host
        return call(state["seqs"], state["lens"], M, *state["out"])
    if kind == "profile":
        return G.mem_profile(state["seqs"])
    if kind == "search":
        state["search"].run(case["generations"])
        return state["search"].state()
    if kind == "edits":
        parents = state["cache"].build(state["seqs"], state["lens"], M) if case["build"] else ()
        return (*parents, *state["cache"].eval_edits(*state["edits"], M))
    return G.check_intervals(state["s"], state["e"], state["a"], M, state["D"], state["topo"])


# ---------------------------------------------------------------------------------- what a pass needs

def work(case):
    """Inputs read once and outputs written once; operations: integer additions and comparisons."""
    n, C, B, kind = case["n"], case["C"], case["B"], case["kind"]
    T = _steps(case)
    edges = {"layered": case["edges"], "training": 2.83 * n, "resnet": 3.0 * n}[case["graph"]]
    one = 4 * T + edges  # an addition and a maximum per step, a copy's two ends, a comparison per edge
    if kind == "eval":
        return {"bytes": B * (4 * T + 24), "flops": B * one}
    if kind == "host":
        return {"bytes": B * (T * case["bits"] / 8 + 24), "flops": B * one}
    if kind == "profile":
        return {"bytes": 4 * T + 12 * T + 4, "flops": one}
    if kind == "search":
        # every chain's state read and written once per pass; a proposal recomputes about a third of
        # the steps of the valid fifth when it is scored from its chain's evaluation
        k = case["generations"] * case["samples"]
        return {"bytes": B * (12 * T + 56), "flops": B * k * (2 * T / 15 + 30)}
    if kind == "edits":
        count = B * case["per_parent"]
        return {"bytes": (B * (4 * T + 24) if case["build"] else 0) + count * 36 + count * 4 * T / 15,
                "flops": (B * one if case["build"] else 0) + count * (2 * T / 15 + 30)}
    return {"bytes": B * (12 * n * C + 20 + 4 * T + 4), "flops": B * (one + 6 * n * C)}


def tolerance(case):
    return "exact"
