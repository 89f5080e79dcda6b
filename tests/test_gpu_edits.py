"""Parity of the incremental evaluation (moc_cache_build + moc_eval_edits, through the C ABI) with the
oracle: every edited sequence is built on the CPU (the oracle's edit, pinned in test_search_oracle.py)
and evaluated from scratch by the oracle's evaluator; peak, duration and status must be identical."""
import numpy as np
import pytest
import torch

import oracle
from oracle import OracleGraph
from paper_2304_14463_b200 import workloads as W

pytestmark = pytest.mark.gpu
BIG = 1 << 60


@pytest.fixture(scope="module")
def B():
    from paper_2304_14463_b200 import build
    build.build()
    from paper_2304_14463_b200 import binding
    return binding


def dev(a, dtype=torch.int32):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype).cuda()


def reference(O, seqs, lens, parent, op, q, j, M, parent_status):
    offs = np.concatenate([[0], np.cumsum(np.clip(lens, 0, None))])
    out = np.zeros((len(parent), 3), np.int64)
    for b in range(len(parent)):
        c = parent[b]
        if c < 0 or c >= len(lens):
            out[b] = (-1, -1, -2)
            continue
        if parent_status[c] < 0:
            out[b] = (-1, -1, -3)
            continue
        row = seqs[offs[c]:offs[c + 1]]
        T = len(row)
        ok = 0 <= op[b] <= 2 and 0 <= q[b] < T and (op[b] == 1 or 0 <= j[b] <= (T if op[b] == 0 else T - 1))
        if not ok:
            out[b] = (-1, -1, -2)
            continue
        child = oracle.mutate(row, int(op[b]), int(q[b]), int(j[b]))
        r = O.eval(child, M)
        out[b] = (r["peak"], r["dur"], r["status"])
    return out


def run_case(B, wl, seqs, lens, M, parent, op, q, j, caps=None, what=""):
    O = OracleGraph(wl.n, wl.edges, wl.w, wl.m, wl.C)
    G = B.Graph(wl.n, wl.edges, wl.w, wl.m, wl.C)
    if caps is not None:
        O.set_caps(caps)
        G.set_caps(caps)
    cache = B.EditCache(G, len(lens))
    pk, du, st = cache.build(dev(seqs), dev(lens), M)
    torch.cuda.synchronize()
    rp, rd, rs, _ = O.eval_batch(seqs, lens, M)
    assert (pk.cpu().numpy() == rp).all() and (du.cpu().numpy() == rd).all() and (st.cpu().numpy() == rs).all(), what
    window = torch.full((len(parent),), -7, dtype=torch.int32, device="cuda")
    got = cache.eval_edits(dev(parent), dev(op), dev(q), dev(j), M, window=window)
    torch.cuda.synchronize()
    got = np.stack([got[0].cpu().numpy(), got[1].cpu().numpy(), got[2].cpu().numpy().astype(np.int64)], 1)
    # steps whose usage was recomputed: none for a refused edit, at most the child's length for a scored one
    win = window.cpu().numpy()
    scored = got[:, 2] >= 0
    child_len = lens[np.clip(parent, 0, len(lens) - 1)] + (op == 0) - (op == 1)
    assert (win[~scored] == 0).all() and (win[scored] >= 0).all() and (win[scored] <= child_len[scored]).all(), what
    assert not scored.any() or win[scored].max() > 0, what
    want = reference(O, seqs, lens, parent, op, q, j, M, rs)
    bad = np.nonzero((got != want).any(1))[0]
    assert len(bad) == 0, f"{what}: {len(bad)} of {len(parent)} edits differ; first: edit {bad[0]} parent {parent[bad[0]]} " \
                          f"op {op[bad[0]]} q {q[bad[0]]} j {j[bad[0]]}: gpu {got[bad[0]]} oracle {want[bad[0]]}"
    return want


def random_edits(rng, lens, nE):
    parent = rng.integers(0, len(lens), nE).astype(np.int32)
    op = rng.integers(0, 3, nE).astype(np.int32)
    T = lens[parent]
    q = (rng.integers(0, 1 << 30, nE) % np.maximum(T, 1)).astype(np.int32)
    j = (rng.integers(0, 1 << 30, nE) % np.where(op == 0, T + 1, np.maximum(T, 1))).astype(np.int32)
    return parent, op, q, j


def test_edits_tiny_exhaustive(B):
    """Every edit of several sequences on small graphs (all q, all j, all three kinds)."""
    rng = np.random.default_rng(0)
    for n, edges in [(4, [(0, 1), (1, 2), (2, 3), (0, 3)]), (5, [(0, 1), (0, 2), (1, 3), (2, 3), (3, 4)]),
                     (5, [(0, 2), (1, 2), (2, 3), (2, 4)]), (3, [])]:
        class WL:
            pass
        wl = WL()
        wl.n, wl.edges, wl.C = n, np.array(edges, np.int32).reshape(-1, 2), 2
        wl.w = rng.integers(1, 9, n).astype(np.int64)
        wl.m = rng.integers(1, 20, n).astype(np.int64)
        rows = [list(range(n))]
        for _ in range(6):                       # valid sequences with extra copies
            r = list(range(n))
            for v in range(n):
                if rng.random() < 0.5:
                    r.insert(int(rng.integers(r.index(v) + 1, len(r) + 1)), v)
            rows.append(r)
        rows.append(list(range(n))[::-1] if edges else list(range(n)))     # an invalid parent (when there are edges)
        seqs = np.array([x for r in rows for x in r], np.int32)
        lens = np.array([len(r) for r in rows], np.int32)
        parent, op, q, j = [], [], [], []
        for c, r in enumerate(rows):
            for o in range(3):
                for qq in range(len(r)):
                    for jj in range(len(r) + 1 if o == 0 else (1 if o == 1 else len(r))):
                        parent.append(c); op.append(o); q.append(qq); j.append(jj)
        M = int(wl.m.sum()) * 2 // 3
        run_case(B, wl, seqs, lens, M, np.array(parent, np.int32), np.array(op, np.int32), np.array(q, np.int32),
                 np.array(j, np.int32), what=f"tiny n={n}")


@pytest.mark.parametrize("idx,P,nE", [(0, 256, 20000), (1, 128, 20000), (2, 64, 12000)])
def test_edits_random(B, idx, P, nE):
    """Random edits of workload sequences (1/16 of the parents damaged), plus malformed edit records."""
    wl = W.make(idx, seed=2, B=P)
    rng = np.random.default_rng(10 + idx)
    seqs, lens = W.mutate(wl.seqs, wl.lens, wl.n, wl.C, seed=6, frac=1 / 16)
    O0 = OracleGraph(wl.n, wl.edges, wl.w, wl.m, wl.C)
    M = O0.eval(np.arange(wl.n), BIG)["peak"] * 80 // 100
    parent, op, q, j = random_edits(rng, np.clip(lens, 0, None), nE)
    # malformed records
    parent[:4] = [-1, P, 0, 0]
    op[4:6] = [3, -1]
    q[6] = lens[parent[6]]
    j[7] = lens[parent[7]] + 5
    want = run_case(B, wl, seqs, lens, M, parent, op, q, j, what=f"config {idx}")
    seen = set(want[:, 2].tolist())
    assert {1, -1, -2, -3} <= seen or {0, -1, -2, -3} <= seen


def test_edits_node_caps_and_wide(B):
    wl = W.make(1, seed=3, B=64)
    rng = np.random.default_rng(5)
    caps = np.where(rng.random(wl.n) < 0.5, 1, 2).astype(np.int32)
    O0 = OracleGraph(wl.n, wl.edges, wl.w, wl.m, wl.C)
    M = O0.eval(np.arange(wl.n), BIG)["peak"] * 80 // 100
    # parents that respect the caps: the identity order and orders with copies of uncapped nodes only
    rows = []
    for _ in range(64):
        r = list(range(wl.n))
        for v in np.nonzero(caps == 2)[0]:
            if rng.random() < 0.3:
                r.insert(int(rng.integers(r.index(v) + 1, len(r) + 1)), int(v))
        rows.append(r)
    seqs = np.array([x for r in rows for x in r], np.int32)
    lens = np.array([len(r) for r in rows], np.int32)
    run_case(B, wl, seqs, lens, M, *random_edits(rng, lens, 8000), caps=caps, what="caps")
    # 64-bit sums
    wl.m = wl.m * (1 << 33)
    run_case(B, wl, seqs, lens, M * (1 << 33), *random_edits(rng, lens, 4000), what="wide")


def test_edits_of_a_star_graph(B):
    """In-degree 1199: the correction lists of the lane-per-edit kernel (4 + 2 * in-degree entries per edit) do not
    fit eight warps of an SM, so the warp-per-edit kernel scores; same results."""
    class WL:
        pass
    wl = WL()
    n = 1200
    rng = np.random.default_rng(21)
    wl.n, wl.C = n, 2
    wl.edges = np.array([(i, n - 1) for i in range(n - 1)], np.int32)
    wl.w = rng.integers(1, 9, n).astype(np.int64)
    wl.m = rng.integers(1, 99, n).astype(np.int64)
    rows = []
    for _ in range(8):
        r = list(rng.permutation(n - 1)) + [n - 1]
        for v in rng.integers(0, n - 1, 40):                       # a second copy of some sources, in front of the sink
            if r.count(int(v)) == 1:
                r.insert(int(rng.integers(r.index(int(v)) + 1, len(r))), int(v))
        rows.append(r)
    seqs = np.array([x for r in rows for x in r], np.int32)
    lens = np.array([len(r) for r in rows], np.int32)
    M = int(wl.m.sum()) * 9 // 10
    want = run_case(B, wl, seqs, lens, M, *random_edits(rng, lens, 3000), what="star")
    assert {0, -1, -2} <= set(want[:, 2].tolist()) or {1, -1, -2} <= set(want[:, 2].tolist())


def test_stale_cache_is_refused(B):
    """Caps or C changed after the build: the cache's copy is stale, edits are refused until a rebuild,
    and after the rebuild they follow the new caps."""
    wl = W.make(1, seed=4, B=32)
    rng = np.random.default_rng(8)
    O = OracleGraph(wl.n, wl.edges, wl.w, wl.m, wl.C)
    G = B.Graph(wl.n, wl.edges, wl.w, wl.m, wl.C)
    M = O.eval(np.arange(wl.n), BIG)["peak"] * 80 // 100
    rows = [list(range(wl.n)) for _ in range(32)]
    seqs = np.array([x for r in rows for x in r], np.int32)
    lens = np.array([len(r) for r in rows], np.int32)
    parent, op, q, j = random_edits(rng, lens, 3000)
    cache = B.EditCache(G, len(lens))
    cache.build(dev(seqs), dev(lens), M)
    cache.eval_edits(dev(parent), dev(op), dev(q), dev(j), M)
    caps = np.where(rng.random(wl.n) < 0.5, 1, 2).astype(np.int32)
    for change in (lambda: G.set_caps(caps), lambda: G.set_caps(None), lambda: G.set_max_copies(2)):
        change()
        with pytest.raises(B.MocError, match="rebuild"):
            cache.eval_edits(dev(parent), dev(op), dev(q), dev(j), M)
        cache.build(dev(seqs), dev(lens), M)
        cache.eval_edits(dev(parent), dev(op), dev(q), dev(j), M)
    # with the caps in force after a rebuild the results are the oracle's for those caps
    G.set_caps(caps)
    O.set_caps(caps)
    cache.build(dev(seqs), dev(lens), M)
    window = torch.full((len(parent),), -7, dtype=torch.int32, device="cuda")
    got = cache.eval_edits(dev(parent), dev(op), dev(q), dev(j), M, window=window)
    torch.cuda.synchronize()
    got = np.stack([got[0].cpu().numpy(), got[1].cpu().numpy(), got[2].cpu().numpy().astype(np.int64)], 1)
    # steps whose usage was recomputed: none for a refused edit, at most the child's length for a scored one
    win = window.cpu().numpy()
    scored = got[:, 2] >= 0
    child_len = lens[np.clip(parent, 0, len(lens) - 1)] + (op == 0) - (op == 1)
    assert (win[~scored] == 0).all() and (win[scored] >= 0).all() and (win[scored] <= child_len[scored]).all(), what
    assert not scored.any() or win[scored].max() > 0, what
    want = reference(O, seqs, lens, parent, op, q, j, M, O.eval_batch(seqs, lens, M)[2])
    assert (got == want).all()
    torch.cuda.synchronize()


@pytest.mark.parametrize("n,shift,nE", [(21, 0, 1), (22, 33, 37), (23, 0, 1184), (99, 33, 4735), (100, 0, 4736), (101, 33, 4737), (100, 33, 160000), (1642, 33, 300)])
def test_edits_per_warp(B, n, shift, nE):
    """Batches from one edit per warp to several rounds, ends of the block's copy of the graph (odd numbers of nodes and edges), and
    state that leaves room for few warps: against the oracle, and every edit the same in batches of other sizes."""
    edges = W.layered_dag(n, 3 * n + n % 4, max(4, n // 40), n)
    wl = type("WL", (), dict(n=n, edges=edges, C=2, w=W.weights_uniform(n, 0, 30, n, 1), m=W.weights_lognormal(n, 3.0, 1.0, n, 2) << shift))
    seqs, lens = W.schedules(n, edges, 2, 0.3, 9, n)
    rng = np.random.default_rng(n)
    M = OracleGraph(n, edges, wl.w, wl.m, 2).eval(np.arange(n), BIG)["peak"] * 90 // 100
    rec = random_edits(rng, lens, nE)
    some = np.sort(rng.choice(nE, min(nE, 5000), replace=False))
    run_case(B, wl, seqs, lens, M, *(x[some] for x in rec), what=f"n {n}")
    cache = B.EditCache(B.Graph(n, edges, wl.w, wl.m, 2), len(lens))
    cache.build(dev(seqs), dev(lens), M)
    whole = cache.eval_edits(*(dev(x) for x in rec), M)
    part = cache.eval_edits(*(dev(x[some]) for x in rec), M)
    for a, b in zip(whole, part):
        assert torch.equal(a[torch.from_numpy(some).cuda()], b)


@pytest.mark.parametrize("n,shift,P", [(100, 0, 1), (100, 33, 147), (101, 0, 149), (100, 44, 149), (442, 33, 300), (101, 0, 3553), (64, 33, 8000)])
def test_build_of_few_and_many_parents(B, n, shift, P):
    """Parents by block and warp, in one round and in several, with sums in one, two and 64-bit parts; some edits of damaged and good ones."""
    edges = W.layered_dag(n, 3 * n, max(4, n // 40), n)
    m = np.minimum(W.weights_lognormal(n, 3.0, 1.0, n, 2), 255) << shift
    wl = type("WL", (), dict(n=n, edges=edges, C=2, w=W.weights_uniform(n, 0, 30, n, 1), m=m))
    seqs, lens = W.schedules(n, edges, 2, 0.3, P, n)
    seqs, lens = W.mutate(seqs, lens, n, 2, seed=5, frac=1 / 8)
    M = OracleGraph(n, edges, wl.w, wl.m, 2).eval(np.arange(n), BIG)["peak"] * 90 // 100
    run_case(B, wl, seqs, lens, M, *random_edits(np.random.default_rng(P), np.clip(lens, 0, None), 1500), what=f"n {n} P {P}")


@pytest.mark.parametrize("n,edges", [(3, []), (5, [(0, 1), (0, 2), (1, 3), (2, 3), (3, 4)]), (6, [(0, 2), (1, 2), (2, 3), (2, 4)]), (33, None), (34, None)])
def test_edits_by_pairs_of_steps(B, n, edges):
    """64-bit sums, whose windows are read by pairs of the parent's steps: every edit of sequences of even and odd length, and with one pair a
    lane and two: insertions in front of the first step and behind the last, the deleted step first or second of a pair."""
    rng = np.random.default_rng(n)
    edges = W.layered_dag(n, 2 * n, 5, n) if edges is None else np.array(edges, np.int32).reshape(-1, 2)
    wl = type("WL", (), dict(n=n, edges=edges, C=2, w=rng.integers(0, 9, n).astype(np.int64), m=rng.integers(1, 20, n).astype(np.int64) << 33))
    rows = []
    for extra in (0, 1, 2, n // 2):
        r = list(range(n))
        for v in rng.permutation(n)[:extra]:
            r.insert(int(rng.integers(r.index(v) + 1, len(r) + 1)), int(v))
        rows.append(r)
    seqs, lens = W.pack([np.array(r, np.int32) for r in rows])
    every = [(c, o, q, j) for c, r in enumerate(rows) for o in range(3) for q in range(len(r)) for j in range(len(r) + (o == 0) if o != 1 else 1)]
    if len(every) > 4000:       # the ends of the sequences and a sample of the rest
        near = [e for e in every if min(e[2], e[3]) < 2 or max(e[2], e[3]) >= len(rows[e[0]]) - 2]
        every = [near[k] for k in rng.permutation(len(near))[:2500]] + [every[k] for k in rng.permutation(len(every))[:2500]]
    parent, op, q, j = (np.array(x, np.int32) for x in zip(*every))
    want = run_case(B, wl, seqs, lens, int(wl.m.sum()) // 2, parent, op, q, j, what=f"n {n}")
    assert (want[:, 2] >= 0).any()
