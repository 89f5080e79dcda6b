"""The host side of the library on a stand-in for the CUDA runtime (fake_cudart.cpp): which kernels are
looked up and launched, what is copied, and what an error leaves behind.  Runs without a GPU; no kernel runs."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2304_14463_b200 import build, workloads

HERE = os.path.dirname(os.path.abspath(__file__))
P, i32, i64 = ctypes.c_void_p, ctypes.c_int32, ctypes.c_int64


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    workloads.build()
    lib = str(tmp_path_factory.mktemp("fake") / "libmoc_fake.so")
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    # no machine code and no optimisation of the kernels: they are never run
    subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=compute_100a", "-Xcicc", "-O0", "-std=c++17", "-cudart", "none", "-shared",
                    "-Xcompiler", "-fPIC", "-Xlinker", "-Bsymbolic,--no-undefined", "-t", "8", "-o", lib,
                    *[os.path.join(build.CSRC, f) for f in build.SOURCES], os.path.join(HERE, "fake_cudart.cpp")], check=True)
    L = ctypes.CDLL(lib)
    L.fake_log.restype = L.fake_modules.restype = L.fake_shapes.restype = ctypes.c_char_p
    L.fake_pin.argtypes = [P, ctypes.c_size_t]
    L.moc_last_error.restype = ctypes.c_char_p
    L.moc_graph_create.argtypes = [i32, i64, P, P, P, ctypes.POINTER(P)]
    L.moc_graph_set_max_copies.argtypes = [P, i32]
    L.moc_graph_destroy.argtypes = [P]
    L.moc_graph_destroy.restype = None
    L.moc_eval_batch.argtypes = [P, P, P, i32, i64, P, P, P, P]
    L.moc_graph_set_node_caps.argtypes = [P, P]
    L.moc_search_create.argtypes = [P, P, P, i32, i64, ctypes.c_uint64, ctypes.c_uint32, P, ctypes.POINTER(P)]
    L.moc_search_set_samples.argtypes = [P, i32, i32]
    L.moc_search_run.argtypes = [P, i32, P]
    L.moc_search_destroy.argtypes = [P]
    L.moc_search_destroy.restype = None
    L.moc_mem_profile.argtypes = [P, P, i32, P, P, P, P]
    L.moc_check_intervals.argtypes = [P, P, P, P, i32, i64, P, i64, P, P, P, P, P, P]
    for f in (L.moc_eval_batch_host, L.moc_eval_batch_host16):
        f.argtypes = [P, P, i64, P, i32, i64, P, P, P, P]
    yield L
    L.fake_reset(0)


class Graph:
    def __init__(self, L, n, C=2, scale=1, star=False):
        self.L, self.n, self.h, self.star = L, n, P(), star
        assert self.create(n, scale) == 0
        assert L.moc_graph_set_max_copies(self.h, C) == 0

    def create(self, n, scale):
        edges = workloads.layered_dag(n, 2 * n, max(2, n // 10), 1) if n >= 20 else np.zeros((0, 2), np.int32)
        if self.star:              # too uneven for successor tiles
            edges = [(0, v) for v in range(1, n)]
        edges = np.ascontiguousarray(edges, np.int32)
        w, m = np.ones(n, np.int64), np.full(n, scale, np.int64)
        return self.L.moc_graph_create(n, len(edges), edges.ctypes.data, w.ctypes.data, m.ctypes.data, ctypes.byref(self.h))

    def close(self):
        self.L.moc_graph_destroy(self.h)


class HostBatch:
    """nB sequences of n ids in a buffer with `spare` more behind them."""

    def __init__(self, n, nB, bits, spare=0):
        self.nB, self.bits, self.need = nB, bits, n * nB
        page = 4096
        self.raw = np.zeros((self.need + spare) * bits // 8 + 2 * page, np.uint8)
        self.start = (-self.raw.ctypes.data) % page
        self.n_steps = self.need + spare
        self.ids = self.raw.ctypes.data + self.start
        self.lens = np.full(nB, n, np.int32)
        self.out = [np.zeros(nB, d) for d in (np.int64, np.int64, np.int32)]

    def pin(self, L, ids=True):
        L.fake_unpin_all()
        for a in [self.lens] + self.out:
            L.fake_pin(a.ctypes.data, a.nbytes)
        if ids:
            L.fake_pin(self.ids, self.n_steps * self.bits // 8)

    def run(self, G):
        call = G.L.moc_eval_batch_host16 if self.bits == 16 else G.L.moc_eval_batch_host
        return call(G.h, self.ids, self.n_steps, self.lens.ctypes.data, self.nB, 1000, *[o.ctypes.data for o in self.out], None)


def log(L):
    return L.fake_log().decode().splitlines()


def launched(L, name):
    return [x for x in log(L) if x.startswith("launch ") and name in x]


@pytest.mark.parametrize("bits", [16, 32])
def test_a_kernel_touches_host_memory_only_where_all_of_it_is_mapped(fake, bits):
    """Ids that lie in one registration, in two that meet, and in two with an unregistered page between them."""
    G, b = Graph(fake, 20), HostBatch(20, 400, bits)
    size, page = b.n_steps * bits // 8, 4096
    for cut, gap, kernel in ((size, 0, True), (page, 0, True), (page, page, False), (page + 1, 1, False)):
        b.pin(fake, ids=False)
        fake.fake_pin(b.ids, cut)
        if cut + gap < size:
            fake.fake_pin(b.ids + cut + gap, size - cut - gap)
        fake.fake_reset(0)
        assert b.run(G) == 0
        assert bool(launched(fake, "fetch_kernel")) == kernel, (cut, gap)
    b.pin(fake)
    for k in range(3):                         # the same for the results: the k-th array has a hole
        b.pin(fake)
        fake.fake_unpin_all()
        for i, a in enumerate(b.out):
            if i == k:
                fake.fake_pin(a.ctypes.data, 64)
                fake.fake_pin(a.ctypes.data + 128, a.nbytes - 128)
            else:
                fake.fake_pin(a.ctypes.data, a.nbytes)
        fake.fake_reset(0)
        assert b.run(G) == 0
        assert any(x.startswith("copy d2h") for x in log(fake)) and not launched(fake, "deliver_kernel")
    G.close()


@pytest.mark.parametrize("bits", [16, 32])
@pytest.mark.parametrize("nB", [300, 4000, 110000])
@pytest.mark.parametrize("pinned", [True, False])
def test_no_work_outlives_a_failed_call(fake, bits, nB, pinned):
    """Every call into the runtime fails in turn: the error is returned, nothing that reads or writes the caller's arrays
    is still in flight by then, and the handle goes on working.  So with lengths that exceed the buffer."""
    fake.fake_unpin_all()
    k = 0
    while True:
        G, b = Graph(fake, 20), HostBatch(20, nB, bits)
        if pinned:
            b.pin(fake)
        k += 1
        fake.fake_reset(k)
        rc = b.run(G)
        calls = fake.fake_calls()
        if rc != 0:
            assert fake.fake_in_flight() == 0, (k, log(fake))
        fake.fake_reset(0)
        assert b.run(G) == 0 and fake.fake_in_flight() == 0
        b.n_steps -= 1
        fake.fake_reset(0)
        assert b.run(G) == -1 and fake.fake_in_flight() == 0
        G.close()
        if calls < k:
            break
    assert k > 10


@pytest.mark.parametrize("bits", [16, 32])
@pytest.mark.parametrize("n,nB", [(20, 1), (20, 300), (20, 4096), (3, 8192), (20, 8000), (20, 65536), (20, 110000), (700, 4001)])
@pytest.mark.parametrize("pinned", [True, False])
def test_ids_behind_the_batch_do_not_travel(fake, bits, n, nB, pinned):
    """A buffer of four times the batch: every id of the batch crosses the link once and none behind it, the first time (staging
    grows to the batch, not to the buffer) and later; a few more ids than the batch may travel with a long batch in
    one piece.  Batches in parts go through more than one evaluation."""
    fake.fake_unpin_all()
    G, b = Graph(fake, n), HostBatch(n, nB, bits, spare=3 * n * nB)
    if pinned:
        b.pin(fake)
    for spare in (3 * n * nB, 0, 5, -1, 0, 5, 3 * n * nB):
        if spare < 0:                         # from here on there is room for twice the batch
            assert HostBatch(n, 2 * nB, bits).run(G) == 0
            continue
        b.n_steps = b.need + spare
        fake.fake_reset(0)
        assert b.run(G) == 0
        lines = [x.split() for x in log(fake)]
        moved = sum(int(x[3]) for x in lines if x[:2] == ["copy", "h2d"] and b.ids <= int(x[2]) < b.ids + b.need * bits // 8)
        fetched = bool(launched(fake, "fetch_kernel"))
        assert fetched and moved == 0 or b.need <= moved * 8 // bits <= b.need + (5 if spare == 5 else 0)
        assert not any(b.ids + b.need * bits // 8 <= int(x[2]) < b.ids + b.n_steps * bits // 8 for x in lines if x[:2] == ["copy", "h2d"])
        assert all(int(x[1]) <= max(4 * b.need + 16, 24 * nB + 16, 8 * (nB + 1)) for x in lines if x[0] == "malloc")
        assert fetched == (pinned and b.need * bits // 8 <= 256 << 10)
        assert len(launched(fake, "eval_")) == (3 if b.need >= 1 << 21 else 1)
    G.close()


def test_lengths_that_lie(fake):
    """Negative lengths count as zero; lengths beyond 16 bits and beyond the buffer are found wherever they stand."""
    for nB, n in ((300, 20), (8000, 20), (110000, 20)):
        G, b = Graph(fake, n), HostBatch(n, nB, 16, spare=100000)
        fake.fake_reset(0)
        b.lens[nB // 2] = -7
        b.lens[nB - 2] = 70000
        assert b.run(G) == 0
        for where in (0, nB // 8, nB // 2, nB - 1):
            for _ in range(2):
                lens = b.lens.copy()
                b.lens[where] = 2 ** 31 - 1
                fake.fake_reset(0)
                assert b.run(G) == -1 and fake.fake_in_flight() == 0
                assert str(int(np.maximum(b.lens.astype(np.int64), 0).sum())) in fake.moc_last_error().decode()
                b.lens[:] = lens
        # a sample of the lengths that promises much more than there is: the batch is evaluated all the same, once
        b.lens[:] = 1
        b.lens[[nB * k // 64 for k in range(64)]] = n
        for steps in (n * nB, int(b.lens.sum())):
            b.n_steps = steps
            fake.fake_reset(0)
            assert b.run(G) == 0 and fake.fake_in_flight() == 0
            assert len(launched(fake, "eval_")) == 1
        G.close()


@pytest.mark.parametrize("n,C,scale,nB,kernel", [(20, 2, 1, 64, "eval_pair"), (20, 2, 1, 60000, "eval_live"), (100, 2, 1 << 30, 64, "eval_pair"),
                                                 (100, 3, 1, 64, "eval_quad"), (100, 4, 1, 60000, "eval_live"), (100, 5, 1, 64, "eval_shared"),
                                                 (442, 2, 1, 64, "eval_pair"), (442, 2, 1, 5000, "eval_pair"), (442, 3, 1, 5000, "eval_quad")])
def test_only_kernels_that_run_are_looked_up(fake, n, C, scale, nB, kernel):
    """A first evaluation on a handle prepares the kernel it launches and no other; a later one of another size adds its own."""
    G = Graph(fake, n, C, scale)
    x = np.zeros(8, np.int64)

    def looked_up(nB):
        fake.fake_reset(0)
        assert fake.moc_eval_batch(G.h, x.ctypes.data, x.ctypes.data, nB, 0, x.ctypes.data, x.ctypes.data, x.ctypes.data, None) == 0
        names = {x.split()[1] for x in log(fake) if x.startswith("lookup ")}
        run = {x.split()[1] for x in log(fake) if x.startswith("launch ") and "offsets" not in x}
        return names, run

    names, run = looked_up(nB)
    assert len(run) == 1 and kernel in next(iter(run)) and names == run
    assert looked_up(nB) == (set(), run)
    for other in (1, 200, 3000, 65536):
        names, run = looked_up(other)
        assert names <= run
    G.close()


def test_kernel_families_do_not_share_a_module(fake):
    """The first use of a kernel loads the whole module it lies in."""
    families = ["eval_pair_kernel", "eval_quad_kernel", "eval_live_kernel", "eval_lane_kernel", "eval_shared_kernel", "check_plain_kernel",
                "check_intervals_kernelILb0E", "check_intervals_kernelILb1E", "search_score_kernel", "search_walk_kernel", "edit_prepare_kernel"]
    modules = fake.fake_modules().decode().splitlines()
    for f in families:
        assert sum(f in m for m in modules) == 1, f
    assert all(sum(f in m for f in families) <= 1 for m in modules)


@pytest.mark.parametrize("n,scale,copies", [(1, 1, 1), (20, 1, 1), (128, 1 << 30, 1), (442, 1, 1), (5000, 1, 1), (17000, 1, None)])
def test_a_handle_is_one_allocation(fake, n, scale, copies):
    """Tables for every kernel family, one allocation and one copy (one per array for graphs with more than a megabyte of
    them), all of it given back; a failing call leaves nothing."""
    fake.fake_reset(0)
    G = Graph(fake, n, 2, scale)
    lines = [x.split()[0] for x in log(fake)]
    assert lines.count("malloc") == 1 and (copies is None or lines.count("memcpy") == copies)
    calls = fake.fake_calls()
    G.close()
    assert fake.fake_allocations() == 0 and "free of a foreign pointer" not in log(fake)
    for k in range(1, calls + 1):
        fake.fake_reset(k)
        assert G.create(n, scale) in (-5, -6) and not G.h.value and fake.fake_allocations() == 0


# batches from which on the backward walk is the faster kernel, as measured: (n, C, 64-bit sums) -> sequences
WALK_FROM = {(20, 2, 0): 5000, (40, 2, 0): 9500, (64, 2, 0): 12000, (65, 2, 0): 11500, (100, 2, 0): 17000, (128, 2, 0): 24000,
             (20, 2, 1): 4000, (40, 2, 1): 6000, (64, 2, 1): 10500, (65, 2, 1): 7500, (100, 2, 1): 12500, (128, 2, 1): 16000,
             (20, 3, 0): 2300, (40, 3, 0): 3200, (64, 3, 1): 4800, (65, 4, 0): 5500, (100, 3, 0): 8000, (128, 4, 1): 8800}


@pytest.mark.parametrize("case", WALK_FROM)
def test_the_backward_walk_starts_where_it_is_faster(fake, case):
    n, C, wide = case
    G = Graph(fake, n, C, 1 << 30 if wide else 1)
    x = np.zeros(8, np.int64)
    for nB, walk in ((int(0.8 * WALK_FROM[case]), False), (int(1.25 * WALK_FROM[case]), True)):
        fake.fake_reset(0)
        assert fake.moc_eval_batch(G.h, x.ctypes.data, x.ctypes.data, nB, 0, x.ctypes.data, x.ctypes.data, x.ctypes.data, None) == 0
        assert bool(launched(fake, "eval_live")) == walk, nB
    G.close()


@pytest.mark.parametrize("n,C,scale,D,staged,off,kernel", [
    (20, 2, 1, 40, False, 0, "check_plain_kernelIi"), (20, 2, 1, 14206, False, 0, "check_plain_kernelIi"),
    (20, 2, 1, 14207, False, 0, "check_intervals_kernelILb1ELi2EiLb1Et"), (20, 2, 1, 65536, False, 0, "check_intervals_kernelILb1ELi2EiLb1Ei"),
    (20, 2, 1, 40, False, 4, "check_intervals_kernelILb1ELi2EiLb1Et"), (20, 3, 1, 40, False, 0, "check_intervals_kernelILb1ELi4EiLb1Et"),
    (20, 2, 1 << 30, 7102, False, 0, "check_plain_kernelIl"), (20, 2, 1 << 30, 7103, False, 0, "check_intervals_kernelILb1ELi2ElLb1Et"),
    (20, 2, 1 << 54, 40, False, 0, "check_intervals_kernelILb1ELi2ElLb1Et"),
    (361, 2, 1, 361 * 181, True, 0, "check_intervals_kernelILb0ELi2EiLb1Et"), (362, 2, 1, 181 * 363, True, 0, "check_intervals_kernelILb0ELi2EiLb1Ei"),
    (1000, 2, 1, 500 * 1001, True, 0, "check_intervals_kernelILb0ELi2EiLb1Ei"), (1200, 2, 1, 600 * 1201, True, 0, "check_intervals_kernelILb0ELi2EiLb0Ei")])
def test_which_kernel_checks_intervals(fake, n, C, scale, D, staged, off, kernel):
    G = Graph(fake, n, C, scale)
    x = np.zeros(n * C + 8, np.int64)
    fake.fake_reset(0)
    rc = fake.moc_check_intervals(G.h, x.ctypes.data + off, x.ctypes.data, x.ctypes.data, 1, D, x.ctypes.data if staged else None, 0,
                                  x.ctypes.data, x.ctypes.data, x.ctypes.data, x.ctypes.data, x.ctypes.data, None)
    assert rc == 0 and len(launched(fake, kernel)) == 1, log(fake)
    G.close()


@pytest.mark.parametrize("n", [199, 601, 1600])
@pytest.mark.parametrize("C", [2, 4, 5])
@pytest.mark.parametrize("scale", [1, 1 << 30])
@pytest.mark.parametrize("star", [False, True])
def test_which_kernel_makes_a_profile(fake, n, C, scale, star):
    G, x = Graph(fake, n, C, scale, star), np.zeros(8, np.int64)
    fake.fake_reset(0)
    assert fake.moc_mem_profile(G.h, x.ctypes.data, 4, x.ctypes.data, None, x.ctypes.data, None) == 0
    wide, tiles = "l" if scale > 1 else "i", 0 if star else 1
    assert len(launched(fake, f"eval_quad_kernelI{wide}Li{4 if C == 4 else 3}ELb{tiles}ELb1E" if C <= 4 else "eval_shared_kernelILi1024")) == 1, log(fake)
    G.close()


# rows of the block kernel's code: a warp per sequence, teams of warps, a block and the graph through L1; and the warp kernel's teams
@pytest.mark.parametrize("n,C,nB,kernel", [(65, 3, 3000, "eval_quad_warp_kernelIiLi3E"), (130, 4, 18944, "eval_quad_warp_kernelIiLi4E"), (442, 3, 1, "eval_quad_kernelIiLi3ELb1ELb0ELi1E"),
                                           (1000, 4, 148, "eval_quad_kernelIiLi4ELb1ELb0ELi1E"), (5000, 4, 300, "eval_quad_kernelIiLi4ELb1ELb0ELi0E"),
                                           (442, 2, 148, "eval_pair_kernelIiLi0ELb1E"), (442, 2, 149, "eval_pair_kernelIiLi0ELb1E"),
                                           (399, 2, 1, "eval_pair_kernelIiLi0ELb1E"), (600, 2, 1, "eval_pair_kernelIiLi0ELb1E"), (600, 2, 1300, "eval_pair_kernelIiLi5ELb0E")])
def test_which_variant_takes_a_batch(fake, n, C, nB, kernel):
    G, x = Graph(fake, n, C), np.zeros(8, np.int64)
    fake.fake_reset(0)
    assert fake.moc_eval_batch(G.h, x.ctypes.data, x.ctypes.data, nB, 0, x.ctypes.data, x.ctypes.data, x.ctypes.data, None) == 0
    assert len(launched(fake, kernel)) == 1, log(fake)
    G.close()


@pytest.mark.parametrize("n,scale,star", [(1, 1, False), (20, 1, False), (128, 1 << 30, False), (442, 1, False), (601, 1, True)])
def test_host_allocations_that_fail(fake, n, scale, star):
    """Every allocation on the host fails in turn: MOC_ERR_NOMEM, no exception across the C ABI, nothing left behind."""
    fake.fake_reset(0)
    G = Graph(fake, n, 2, scale, star)
    caps = np.ones(n, np.int32)
    k = 0
    while True:
        k += 1
        fake.fake_fail_new(k)
        rc = fake.moc_graph_set_node_caps(G.h, caps.ctypes.data)
        used = fake.fake_news()
        fake.fake_fail_new(0)
        assert rc == (-6 if used >= k else 0)
        if used < k:
            break
    seqs, lens, s = np.zeros(2 * n + 8, np.int32), np.full(3, n, np.int32), P()
    assert fake.moc_search_create(G.h, seqs.ctypes.data, lens.ctypes.data, 3, 0, 1, 0, None, ctypes.byref(s)) == 0
    fake.fake_fail_new(1)
    assert fake.moc_search_set_samples(s, 4, 1) == -6
    fake.fake_fail_new(0)
    fake.moc_search_destroy(s)
    G.close()
    k = 0
    while True:
        k += 1
        fake.fake_fail_new(k)
        rc = G.create(n, scale)
        used = fake.fake_news()
        fake.fake_fail_new(0)
        if used < k:
            break
        assert rc in (0, -6) and (rc == 0) == bool(G.h.value)         # 0: the sort did without its buffer
        if rc == 0:
            G.close()
        assert fake.fake_allocations() == 0
    G.close()
    assert k > (10 if n > 1 else 3)


class Search:
    def __init__(self, L, G, chains, samples=1):
        self.L, self.h, self.chains = L, P(), chains
        lens = np.full(chains, G.n, np.int32)
        assert L.moc_search_create(G.h, lens.ctypes.data, lens.ctypes.data, chains, 0, 1, 0, None, ctypes.byref(self.h)) == 0
        if samples > 1:
            assert L.moc_search_set_samples(self.h, samples, 1) == 0

    def launches(self, generations=1):
        """(kernel, warps of a block, rounds of chains, bytes of shared memory) of the launches of a run."""
        self.L.fake_reset(0)
        assert self.L.moc_search_run(self.h, generations, None) == 0
        rows = [x.split() for x in self.L.fake_shapes().decode().splitlines()]
        return [(k, int(t) // 32, -(-self.chains // (int(b) * int(t) // 32)), int(smem)) for k, b, t, smem in rows]

    def close(self):
        self.L.moc_search_destroy(self.h)


# what fits an SM beside the graph when a warp holds two sets of words, 64 bytes of scalars and the deltas
@pytest.mark.parametrize("n,scale,chains,warps,rounds", [(442, 1, 4096, 28, 1), (500, 1, 3700, 25, 1), (600, 1, 3000, 21, 1), (940, 1, 4000, 14, 2), (990, 1, 3700, 13, 2),
                                                         (390, 1 << 30, 16000, 22, 5), (450, 1 << 30, 8000, 19, 3), (780, 1 << 30, 1600, 11, 1), (930, 1 << 30, 3700, 9, 3),
                                                         (2990, 1, 592, 4, 1)])
@pytest.mark.parametrize("samples", [1, 32])
def test_rounds_of_a_search(fake, n, scale, chains, warps, rounds, samples):
    G = Graph(fake, n, 2, scale)
    S = Search(fake, G, chains, samples)
    (kernel, *shape, _), = S.launches()
    assert "search_walk_" in kernel and shape == [warps, rounds]
    S.close()
    G.close()


# the neighbours' lists fit beside the chains, but not the lists and n output sizes (and at the last three not even the lists)
@pytest.mark.parametrize("n,scale,chains,lists", [(490, 1, 3700, 1), (660, 1, 8000, 1), (770, 1, 16000, 1), (850, 1, 4000, 1), (2950, 1, 400, 1), (380, 1 << 30, 16000, 1), (440, 1 << 30, 8000, 1),
                                                  (540, 1 << 30, 16000, 1), (620, 1 << 30, 3700, 1), (870, 1 << 30, 3700, 1), (980, 1 << 30, 8000, 1),
                                                  (500, 1, 3700, 0), (390, 1 << 30, 16000, 0), (780, 1 << 30, 1600, 0)])
@pytest.mark.parametrize("samples", [1, 32])
def test_lists_of_a_search_on_chip(fake, n, scale, chains, lists, samples):
    G = Graph(fake, n, 2, scale)
    S = Search(fake, G, chains, samples)
    (kernel, *_), = S.launches()
    assert f"kernelI{'l' if scale > 1 else 'i'}Lb{lists}E" in kernel
    S.close()
    G.close()


def test_sizes_go_on_chip_for_the_variant_that_reads_them(fake):
    """32-bit sums with the bound on the new peak, where they fit behind the lists."""
    for n, scale, chains, more in ((200, 1, 4000, 4 * 200), (490, 1, 3700, 0), (200, 1 << 30, 4000, 0)):
        G = Graph(fake, n, 2, scale)
        smem = {}
        for samples in (1, 32):
            S = Search(fake, G, chains, samples)
            (kernel, _, _, smem[samples]), = S.launches()
            S.close()
        assert more - 16 < smem[32] - smem[1] <= (more + 16 if more else 0), (n, scale, smem)
        G.close()


@pytest.mark.parametrize("n,samples", [(100, 1), (100, 7), (100, 8), (300, 8)])
def test_a_search_prepares_the_variant_that_it_launches(fake, n, samples):
    """With and without the bound on the new peak lie in two modules, of which a search loads the one that it launches; another number
    of proposals prepares its own when it is set."""
    modules = fake.fake_modules().decode().splitlines()
    for f in ("search_walk_kernel", "search_walk_floor_kernel"):
        assert sum(f in m for m in modules) == 1
    assert not any("search_walk_kernel" in m and "search_walk_floor_kernel" in m for m in modules)
    G = Graph(fake, n)
    for k in (samples, 32, 1):
        fake.fake_reset(0)
        S = Search(fake, G, 300, k)
        before = {x.split()[1] for x in log(fake) if x.startswith("lookup ") and "search_walk" in x}
        (kernel, *_), = S.launches()
        assert before == ({kernel} if k > 1 else set())
        assert {x.split()[1] for x in log(fake) if x.startswith("lookup ")} == ({kernel} if k == 1 else set())
        S.launches()
        assert not [x for x in log(fake) if x.startswith("lookup ")]
        S.close()
    G.close()


@pytest.mark.parametrize("n,samples,calls", [(100, 1, [(10, "0"), (9000, "000")]), (256, 1, [(4096, "0"), (10, "0")]), (300, 1, [(9000, "011"), (10, "1")]),
                                             (300, 1, [(4095, "0"), (1, "0"), (1, "1")]), (300, 2, [(5000, "011")]), (300, 2, [(1023, "0"), (1, "0"), (1, "1")]), (300, 3, [(10, "1")]), (100, 7, [(10, "0")]), (100, 8, [(10, "1")])])
def test_when_a_search_is_tested_with_a_bound(fake, n, samples, calls):
    """A digit per launch (4096 proposals a chain).  More than 256 nodes: with one proposal a generation from generation 4096 on, with two from 1024 on;
    until then the bound costs more than it saves."""
    G = Graph(fake, n)
    S = Search(fake, G, 300, samples)
    for generations, want in calls:
        assert "".join("01"["search_walk_floor_kernel" in k] for k, *_ in S.launches(generations)) == want
    S.close()
    G.close()
