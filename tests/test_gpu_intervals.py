"""Parity of moc_check_intervals (through the C ABI) with the interval-form oracle: mask, peak,
duration, and the execution sequence, solution by solution."""
import numpy as np
import pytest
import torch

import interval_pins
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


def test_interval_pins_through_the_gpu(B):
    """The oracle's own pins (worked example of the paper, one violation per constraint, random valid
    solutions) with the CUDA checker in place of the oracle."""
    class GpuGraph:
        def __init__(self, n, edges, w, m, C):
            self.n, self.C = n, C
            self.G = B.Graph(n, edges, w, m, C)
            self.O = OracleGraph(n, edges, w, m, C)     # sequence evaluator, for building inputs only

        def eval(self, seq, M):
            return self.O.eval(seq, M)

        def _call(self, s, e, a, M, D, topo_index):
            sh = (1, self.n, self.C)
            t = None if topo_index is None else dev(topo_index)
            return self.G.check_intervals(dev(np.reshape(s, sh)), dev(np.reshape(e, sh)), dev(np.reshape(a, sh)), M,
                                          D=D, topo_index=t)

        def check_intervals(self, s, e, a, M, D=None, topo_index=None):
            r = self._call(s, e, a, M, D, topo_index)
            torch.cuda.synchronize()
            ref = self.O.check_intervals(s, e, a, M, D=D, topo_index=topo_index)   # usage per event: oracle only
            return dict(mask=int(r["mask"][0]), peak=int(r["peak"][0]), dur=int(r["dur"][0]), usage=ref["usage"])

        def intervals_to_sequence(self, s, e, a, D=None, staged=False):
            topo = np.arange(1, self.n + 1, dtype=np.int32) if staged else None
            r = self._call(s, e, a, BIG, D, topo)
            torch.cuda.synchronize()
            k = int(r["lens"][0])
            return None if k < 0 else r["seqs"][0, :k].cpu().numpy()

    interval_pins.run_all(lambda n, e, w, m, C: GpuGraph(n, e, w, m, C))


def staged_sequence(rng, n, C, p):
    seq, cnt = [], np.zeros(n, np.int64)
    for j in range(n):
        again = np.nonzero((rng.random(j) < p) & (cnt[:j] < C))[0]
        seq.extend(again.tolist())
        cnt[again] += 1
        seq.append(j)
        cnt[j] += 1
    return seq


def build_batch(O, wl, rng, nB, staged):
    n, C = wl.n, wl.C
    s = np.zeros((nB, n, C), np.int32)
    e = np.zeros((nB, n, C), np.int32)
    a = np.zeros((nB, n, C), np.int32)
    topo = np.arange(1, n + 1, dtype=np.int32) if staged else None
    offs = np.concatenate([[0], np.cumsum(wl.lens)])
    for b in range(nB):
        seq = staged_sequence(rng, n, C, 0.3 / max(1, n // 20)) if staged else wl.seqs[offs[b]:offs[b + 1]].tolist()
        s[b], e[b], a[b], _ = interval_pins.intervals_from_sequence(O, n, C, seq, staged_topo=topo)
    D = n * (n + 1) // 2 if staged else C * n
    # damage three quarters of the solutions: a few entries each, of every kind
    for b in range(nB):
        if b % 4 == 0:
            continue
        for _ in range(int(rng.integers(1, 4))):
            v, i, kind = int(rng.integers(n)), int(rng.integers(C)), int(rng.integers(8))
            if kind == 0:
                e[b, v, i] = max(1, e[b, v, i] - int(rng.integers(1, 4)))
            elif kind == 1:
                e[b, v, i] = min(D, e[b, v, i] + int(rng.integers(1, 50)))
            elif kind == 2:
                s[b, v, i] = int(rng.integers(1, D + 1))
            elif kind == 3:
                a[b, v, i] ^= 1
            elif kind == 4:
                s[b, v, i] = s[b, int(rng.integers(n)), int(rng.integers(C))]
            elif kind == 5 and b % 16 == 1:
                s[b, v, i] = [0, D + 1, -5][int(rng.integers(3))]
            elif kind == 6 and b % 16 == 2:
                a[b, v, i] = 2
            else:
                s[b, v, i] = e[b, v, i] = int(rng.integers(1, D + 1))
    return s, e, a, D, topo


@pytest.mark.parametrize("idx,nB,staged", [(0, 512, False), (0, 512, True), (1, 128, False), (1, 96, True),
                                           (2, 64, False), (2, 6, True), (3, 16, False), (4, 3, False)])
def test_interval_batch_parity(B, idx, nB, staged):
    wl = W.make(idx, seed=3, B=nB)
    rng = np.random.default_rng(100 + idx)
    O = OracleGraph(wl.n, wl.edges, wl.w, wl.m, wl.C)
    G = B.Graph(wl.n, wl.edges, wl.w, wl.m, wl.C)
    s, e, a, D, topo = build_batch(O, wl, rng, nB, staged)
    M = O.eval(np.arange(wl.n), BIG)["peak"] * 80 // 100
    r = G.check_intervals(dev(s), dev(e), dev(a), M, D=D, topo_index=None if topo is None else dev(topo))
    torch.cuda.synchronize()
    mask, peak, dur = r["mask"].cpu().numpy(), r["peak"].cpu().numpy(), r["dur"].cpu().numpy()
    lens, seqs = r["lens"].cpu().numpy(), r["seqs"].cpu().numpy()
    seen = set()
    for b in range(nB):
        ref = O.check_intervals(s[b], e[b], a[b], M, D=D, topo_index=topo)
        assert (int(mask[b]), int(peak[b]), int(dur[b])) == (ref["mask"], ref["peak"], ref["dur"]), (idx, staged, b)
        seq = O.intervals_to_sequence(s[b], e[b], a[b], D=D)
        assert (seq is None) == (lens[b] < 0), (idx, staged, b)
        if seq is not None:
            assert lens[b] == len(seq) and (seqs[b, :lens[b]] == seq).all()
        seen.add(ref["mask"])
    assert 0 in seen or any(m & ~4 == 0 for m in seen)
    if nB >= 64:
        assert len(seen) >= 4        # the damage produced several kinds of violation


def test_interval_argument_errors(B):
    wl = W.make(4, seed=1, B=1)      # n = 5000: the staged domain (12.5 M events) does not fit on chip
    G = B.Graph(wl.n, wl.edges, wl.w, wl.m, wl.C)
    z = torch.ones((1, wl.n, wl.C), dtype=torch.int32, device="cuda")
    with pytest.raises(B.MocError) as err:
        G.check_intervals(z, z, z, 1, topo_index=dev(np.arange(1, wl.n + 1)))
    assert err.value.code == -1
    with pytest.raises(B.MocError):
        G.check_intervals(z, z, z, 1, D=7, topo_index=dev(np.arange(1, wl.n + 1)))   # staged needs D = n(n+1)/2
    with pytest.raises(B.MocError):
        G.check_intervals(z, z, z, 1, D=0)


def test_interval_full_size_sampled(B):
    """The benchmark's shape (headline graph, 16384 solutions, plain domain): every 37th solution is
    compared with the oracle; the rest must agree with the copy of the same solution among them."""
    nB, distinct = 16384, 128
    wl = W.make(2, seed=1, B=distinct)
    rng = np.random.default_rng(9)
    O = OracleGraph(wl.n, wl.edges, wl.w, wl.m, wl.C)
    G = B.Graph(wl.n, wl.edges, wl.w, wl.m, wl.C)
    s, e, a, D, _ = build_batch(O, wl, rng, distinct, staged=False)
    perm = rng.permutation(nB) % distinct
    M = O.eval(np.arange(wl.n), BIG)["peak"] * 80 // 100
    r = G.check_intervals(dev(s[perm]), dev(e[perm]), dev(a[perm]), M, D=D)
    torch.cuda.synchronize()
    mask, peak, dur, lens = (r[k].cpu().numpy() for k in ("mask", "peak", "dur", "lens"))
    ref = {}
    for b in range(0, nB, 37):
        k = int(perm[b])
        if k not in ref:
            x = O.check_intervals(s[k], e[k], a[k], M, D=D)
            ref[k] = (x["mask"], x["peak"], x["dur"])
        assert (int(mask[b]), int(peak[b]), int(dur[b])) == ref[k], b
    first = {}
    for b in range(nB):
        k = int(perm[b])
        got = (int(mask[b]), int(peak[b]), int(dur[b]), int(lens[b]))
        assert first.setdefault(k, got) == got, b


def check_against_oracle(G, O, s, e, a, M, D, topo=None, tensors=None):
    t = tensors or [dev(x) for x in (s, e, a)]
    r = G.check_intervals(*t, M, D=D, topo_index=None if topo is None else dev(topo))
    torch.cuda.synchronize()
    r = {k: v.cpu().numpy() for k, v in r.items()}
    seen = set()
    for b in range(len(s)):
        ref = O.check_intervals(s[b], e[b], a[b], M, D=D, topo_index=topo)
        assert (int(r["mask"][b]), int(r["peak"][b]), int(r["dur"][b])) == (ref["mask"], ref["peak"], ref["dur"]), b
        seq = O.intervals_to_sequence(s[b], e[b], a[b], D=D)
        k = -1 if seq is None else len(seq)
        assert r["lens"][b] == k and (seq is None or (r["seqs"][b, :k] == seq).all()) and (r["seqs"][b, max(k, 0):] == -1).all(), b
        seen.add(ref["mask"])
    return seen


@pytest.mark.parametrize("idx,nB,shift", [(0, 200, 20), (0, 37, 34), (2, 40, 20), (2, 13, 30), (2, 9, 41)])
def test_interval_sums_in_64_bits(B, idx, nB, shift):
    """Two slots per node in the plain domain with sums beyond 32 bits: in two 32-bit parts, and (the last)
    beyond what the parts cover, where another kernel serves them."""
    wl = W.make(idx, seed=5, B=nB)
    m = np.minimum(wl.m, 255) << shift
    O, G = OracleGraph(wl.n, wl.edges, wl.w, m, wl.C), B.Graph(wl.n, wl.edges, wl.w, m, wl.C)
    assert G.info()["wide"]
    s, e, a, D, _ = build_batch(O, wl, np.random.default_rng(idx), nB, False)
    assert len(check_against_oracle(G, O, s, e, a, O.eval(np.arange(wl.n), BIG)["peak"] * 80 // 100, D)) >= 3


@pytest.mark.parametrize("shift", [0, 20])
@pytest.mark.parametrize("D", [7102, 7103, 14205, 14206, 14207, 32766, 32767, 40001])
def test_interval_long_plain_domains(B, D, shift):
    """Few intervals spread over more and more events: from the kernel for two slots per node (whose events have to fit an SM
    four times: up to 14206, 7102 with 64-bit sums) to the general one, last events and the ones behind them included."""
    nB = 24
    wl = W.make(0, seed=6, B=nB)
    m = wl.m << shift
    O, G = OracleGraph(wl.n, wl.edges, wl.w, m, wl.C), B.Graph(wl.n, wl.edges, wl.w, m, wl.C)
    rng = np.random.default_rng(D)
    s, e, a, D0, _ = build_batch(O, wl, rng, nB, False)
    for b in range(nB):                                      # events moved apart, in order; what lies outside stays outside
        place = np.concatenate([[0], np.sort(rng.choice(np.arange(1, D + 1), D0, replace=False)), [D + 1]])
        place[D0] = D
        for x in (s, e):
            inside = (x[b] >= 0) & (x[b] <= D0 + 1)
            x[b][inside] = place[x[b][inside]]
    assert len(check_against_oracle(G, O, s, e, a, O.eval(np.arange(wl.n), BIG)["peak"], D)) >= 3


@pytest.mark.parametrize("k", [0, 1, 2])
def test_interval_arrays_off_an_eight_byte_boundary(B, k):
    """One of the three arrays starts four bytes off: the pairs of slots cannot be read as one word."""
    wl = W.make(2, seed=7, B=12)
    O, G = OracleGraph(wl.n, wl.edges, wl.w, wl.m, wl.C), B.Graph(wl.n, wl.edges, wl.w, wl.m, wl.C)
    s, e, a, D, _ = build_batch(O, wl, np.random.default_rng(k), 12, False)
    t = []
    for i, x in enumerate((s, e, a)):
        flat = torch.zeros(x.size + 1, dtype=torch.int32, device="cuda")
        t.append((flat[1:] if i == k else flat[:-1]).view(x.shape))
        t[-1].copy_(dev(x))
        assert t[-1].data_ptr() % 8 == (4 if i == k else 0)
    check_against_oracle(G, O, s, e, a, O.eval(np.arange(wl.n), BIG)["peak"] * 80 // 100, D, tensors=t)


@pytest.mark.parametrize("n,shift", [(361, 0), (361, 20), (362, 0), (600, 0), (600, 20), (1000, 0), (1200, 0)])
def test_interval_staged_around_the_rule_for_kept_solutions(B, n, shift):
    """Staged domains whose solutions stay on chip (16 bits per event up to n = 361, 32 beyond) while two fit an SM, and
    domains too large for that."""
    nB = 3
    edges = W.layered_dag(n, 3 * n, 20, n)
    w, m = W.weights_uniform(n, 1, 30, n, 1), W.weights_lognormal(n, 4.0, 1.0, n, 2) << shift
    O, G = OracleGraph(n, edges, w, m, 2), B.Graph(n, edges, w, m, 2)

    class Shape:
        pass

    wl = Shape()
    wl.n, wl.C, wl.lens = n, 2, np.zeros(nB, np.int32)
    s, e, a, D, topo = build_batch(O, wl, np.random.default_rng(n), nB, True)
    seen = check_against_oracle(G, O, s, e, a, O.eval(np.arange(n), BIG)["peak"], D, topo=topo)
    assert any(x & ~4 == 0 for x in seen) and len(seen) >= 2


@pytest.mark.parametrize("n,C,D,staged,shift,nB", [(300, 2, 0, True, 0, 9000), (420, 2, 0, True, 20, 5000), (1140, 2, 0, True, 0, 800),
                                                   (200, 3, 40001, False, 0, 9000), (700, 3, 2100, False, 20, 8500)])
def test_interval_blocks_that_take_several_solutions(B, n, C, D, staged, shift, nB):
    """A block per solution and more solutions than blocks can be resident at once, so that a block takes several in turn, valid ones,
    damaged ones and ones outside the domain (which end early) in any order: every kept form (16 and 32 bits, none), marks by bytes
    and by bits, 32- and 64-bit sums."""
    distinct = 16 if n < 1000 else 8                         # (the oracle walks the events of the domain: 3 s per solution at n = 1140)
    rng = np.random.default_rng(n)
    edges = W.layered_dag(n, 3 * n, 20, n)
    w, m = W.weights_uniform(n, 1, 30, n, 1), W.weights_lognormal(n, 4.0, 1.0, n, 2) << shift
    O, G = OracleGraph(n, edges, w, m, C), B.Graph(n, edges, w, m, C)
    assert G.info()["wide"] == (shift > 0)

    class Shape:
        pass

    wl = Shape()
    wl.n, wl.C = n, C
    wl.seqs, wl.lens = W.schedules(n, edges, C, 0.2, distinct, n)
    s, e, a, D0, topo = build_batch(O, wl, rng, distinct, staged)
    if not staged and D > D0:                                # events moved apart, in order; what lies outside stays outside
        place = np.concatenate([[0], np.sort(rng.choice(np.arange(1, D + 1), D0, replace=False)), [D + 1]])
        for x in (s, e):
            inside = (x >= 0) & (x <= D0 + 1)
            x[inside] = place[x[inside]]
    D = max(D, D0)
    s[5, n // 2, 0], e[6, n - 1, 1], a[7, 0, 0] = 0, D + 1, 2
    sms, per_solution = torch.cuda.get_device_properties(0).multi_processor_count, (D // 8) * (1 if staged else 2) + 4 * n * C
    assert nB > sms * min(32, 232448 // per_solution)        # more than the blocks (of two warps at least) that fit
    M = O.eval(np.arange(n), BIG)["peak"] * 80 // 100
    masks = check_against_oracle(G, O, s, e, a, M, D, topo=topo)
    assert 64 in masks and any(x & ~4 == 0 for x in masks) and len(masks) >= 3
    t = [dev(x) for x in (s, e, a)]
    topo = None if topo is None else dev(topo)
    few = G.check_intervals(*t, M, D=D, topo_index=topo)
    which = torch.from_numpy(rng.integers(0, distinct, nB)).cuda()
    many = G.check_intervals(*(x[which] for x in t), M, D=D, topo_index=topo)
    for k in ("mask", "peak", "dur", "lens", "seqs"):
        assert torch.equal(many[k], few[k][which]), k
