"""Order of the kernels' reads of tables that a block copies into shared memory.  A read by an asm statement that is neither
volatile nor has a memory clobber is free to move, in front of a barrier too, unless its address is not known there:
every kernel with such reads makes the base of each table opaque (MOC_STAGED) behind the wait for the copies and the barrier.
Checked on the source; runs without a GPU."""
import os
import re

import pytest

from paper_2304_14463_b200 import build

# kernel -> bases of the tables that it reads freely
FREE = {"eval_pair_kernel": {"sell0"}, "eval_live_kernel": {"pa", "ra", "ma", "own"}, "eval_lane_kernel": {"a_succ"},
        "edit_prepare_kernel": {"sell0"}, "search_walk_kernel": {"l_node"}}


def functions():
    """(name, text) of the functions of the kernel headers, which end with a brace in the first column; without comments."""
    for f in build.HEADERS:
        if f.endswith(".cuh"):
            with open(os.path.join(build.CSRC, f)) as src:
                text = re.sub(r"//[^\n]*|__launch_bounds__\(.*\)(?= \w+\()", "", src.read())
            for part in re.split(r"^\}.*$", text, flags=re.M):
                m = re.search(r"^[^\s#}].*\b(\w+)\([^;{}]*\) *\{$", part, re.M)
                if m:
                    yield m[1], part[m.start():]


def free_readers():
    names = {name for name, text in functions() if re.search(r'\basm\((\s*"[^"]*")*?\s*"[^"]*\bld\.shared', text)}
    while True:
        more = {name for name, text in functions() if any(re.search(r"\b%s(<\w+>)?\(" % h, text.split("{", 1)[1]) for h in names)}
        if more <= names:
            return names
        names |= more


def test_which_kernels_read_freely():
    assert {"lds_u32_nv", "live_lds_v2", "live_lds_v4", "live_lds_words"} <= free_readers()
    kernels = {name for name, text in functions() if "__global__" in text}
    assert len(kernels) > 12 and kernels & free_readers() == set(FREE)


@pytest.mark.parametrize("kernel", FREE)
def test_tables_are_read_behind_their_barrier(kernel):
    text, = [t for name, t in functions() if name == kernel]
    staged = list(re.finditer(r"MOC_STAGED\((\w+)\);", text))
    assert {m[1] for m in staged} == FREE[kernel]
    for m in staged:
        barrier, copies = text.rfind("__syncthreads()", 0, m.start()), text.rfind("cp.async", 0, m.start())
        assert barrier > copies, (kernel, m[1])
        # the base is the variable itself wherever it is used: not taken by value in front of the barrier, not set behind it
        assert not re.search(r"\[=", text) and not re.search(r"\b%s\s*[-+]?=[^=]" % m[1], text[m.end():]), (kernel, m[1])
