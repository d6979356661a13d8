"""The launch counter's share of the Morton sort: the kernels of a sort are counted
by capturing it. A capture that cannot begin costs the count only, the sort runs;
and sizes that alternate (a target's and a source's, in every registration) are
captured once each, sizes between two with the same count not at all. Host build
of index.cu over a recorded CUDA runtime (CPU only)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def sort():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    d = os.path.join(HERE, "_build")   # in-tree, git-ignored
    os.makedirs(d, exist_ok=True)
    exe = os.path.join(d, "sort_launches_host")
    subprocess.run([nvcc, "-O1", "-std=c++17", "-cudart", "none", "--expt-relaxed-constexpr", "-gencode",
                    "arch=compute_103a,code=sm_103a", os.path.join(HERE, "sort_launches_host.cu"),
                    os.path.join(HERE, "fake_cuda_runtime.cpp"), "-o", exe], check=True)

    def run(*args):
        out = subprocess.run([exe, *map(str, args)], check=True, capture_output=True, text=True).stdout
        return [tuple(map(int, line.split())) for line in out.splitlines()]
    return run


SIZES = [1000, 200_000, 500, 5_000_000, 60_000]


def test_counts_are_the_launches_and_known_sizes_are_not_captured_again(sort):
    rows = sort(*SIZES, *SIZES, 777, 4_999_999, 999, 70_001)
    assert all(result == 0 and counted == launched for result, counted, launched, _ in rows)
    captures = [r[3] for r in rows]
    # 60,000 lies below both sizes with the larger count; after it every size is known
    assert captures == [1, 2, 3, 4, 5] + [5] * (len(rows) - 5)


def test_the_sort_runs_when_it_cannot_be_captured(sort):
    rows = sort("refused", *SIZES)
    assert [r[0] for r in rows] == [0] * len(SIZES)
    assert [r[2] for r in rows] == [r[2] for r in sort(*SIZES)]
    assert [r[3] for r in rows] == [0] * len(SIZES)
