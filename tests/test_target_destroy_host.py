"""fricp_target_destroy gives a target's memory back to the pool, from which the
next allocation may take it: so it waits for the device that holds the target,
whichever device is current and wherever the calling thread's work stream lives,
frees on a stream of that device, and leaves the current device as it was.
Host build of api.cu over a recorded CUDA runtime with two devices (CPU only)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def exe():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    d = os.path.join(HERE, "_build")   # in-tree, git-ignored
    os.makedirs(d, exist_ok=True)
    out = os.path.join(d, "target_destroy_host")
    subprocess.run([nvcc, "-O1", "-std=c++17", "-cudart", "none", "--expt-relaxed-constexpr", "-Xcompiler", "-pthread",
                    os.path.join(HERE, "target_destroy_host.cu"), os.path.join(HERE, "fake_cuda_runtime.cpp"), "-o", out],
                   check=True)
    return out


@pytest.mark.parametrize("target", [0, 1])
@pytest.mark.parametrize("stream", [-1, 0, 1])
@pytest.mark.parametrize("current", [0, 1])
def test_destroy_waits_for_the_targets_own_device(exe, target, stream, current):
    out = subprocess.run([exe, str(target), str(stream), str(current)], check=True, capture_output=True,
                         text=True).stdout.splitlines()
    assert out == [f"wait {target}", f"free {target}", f"current {current}",
                   f"work stream {current if stream < 0 else stream}"]
