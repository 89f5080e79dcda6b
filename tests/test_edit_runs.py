"""How a warp shares an edit's window of 16-byte vectors (64-bit sums).  Runs without a GPU: the rule is compiled for the host."""
import ctypes
import os
import re
import subprocess

import pytest

from paper_2304_14463_b200 import build


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    d = tmp_path_factory.mktemp("runs")
    src, lib = str(d / "runs.cu"), str(d / "runs.so")
    with open(src, "w") as f:
        f.write('#include "moc_edit_pass.cuh"\nextern "C" int run(int nv, int shared) { return moc::edit_run(nv, shared != 0); }\n')
    subprocess.run([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-gencode", "arch=compute_100a,code=compute_100a", "-std=c++17", "-shared",
                    "-Xcompiler", "-fPIC", "-I", build.CSRC, "-o", lib, src], check=True)
    return ctypes.CDLL(lib).run


def test_lanes_of_a_window_in_shared_memory_share_no_bank(run):
    """Shared memory serves 16-byte reads by eight lanes, from 32 banks of 4 bytes: their vectors differ modulo eight."""
    for shared in (0, 1):
        for nv in range(1, 16000, 1 if shared else 7):
            per = run(nv, shared)
            assert 32 * per >= nv, nv
            if shared:
                assert len({k * per % 8 for k in range(8)}) == 8, nv
            else:
                assert 32 * (per - 1) < nv, nv


@pytest.mark.parametrize("header,shared", [("moc_search_score_kernel.cuh", "true"), ("moc_edit_lanes_kernel.cuh", "false")])
def test_who_reads_the_usage_from_shared_memory(header, shared):
    with open(os.path.join(build.CSRC, header)) as f:
        assert re.findall(r"kShared = (\w+);", f.read()) == [shared]
    with open(os.path.join(build.CSRC, "moc_edit_pass.cuh")) as f:
        assert "edit_run(nv, decltype(view)::kShared)" in f.read()
