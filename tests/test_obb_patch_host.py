"""The oriented boxes of the patches above the buckets (128, 1,024 and 8,192 points
and ragged rests), built for the host from the kernel's own source (obb.cuh) and held
to the bound the search relies on, as the buckets' boxes are: the box's float distance
is at most (1 + 8e-6) times the squared distance to the patch's nearest point, and
zero for the patch's own points (CPU only)."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest
from scipy.spatial import cKDTree
from scipy.spatial.transform import Rotation

HERE = os.path.dirname(os.path.abspath(__file__))
BOUND = 1.0 + 8e-6
FP = ctypes.POINTER(ctypes.c_float)


@pytest.fixture(scope="module")
def H():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    d = os.path.join(HERE, "_build")   # in-tree, git-ignored
    os.makedirs(d, exist_ok=True)
    so = os.path.join(d, "libobb_patch_host.so")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-x", "cu",
                    os.path.join(HERE, "obb_patch_host.cu"), "-o", so], check=True)
    L = ctypes.CDLL(so)
    L.h_obb_fit_patch.argtypes = [FP, ctypes.c_int, FP]
    L.h_obb_d2.argtypes = [FP, FP, FP, ctypes.c_int, FP]
    return L


def _p(a):
    return a.ctypes.data_as(FP)


def _d2(H, box, xh, xl):
    out = np.empty(len(xh), np.float32)
    H.h_obb_d2(_p(box), _p(xh), _p(xl), len(xh), _p(out))
    return out


def _patches(g, n):
    def sheet(size, origin, curved=0.0, thick=0.0):
        uv = (g.random((n, 2)) - 0.5) * size
        z = curved * (uv ** 2).sum(1) + thick * g.standard_normal(n)
        return np.column_stack([uv, z]) @ Rotation.random(random_state=g.integers(1 << 30)).as_matrix().T + origin

    base = g.random(3)
    yield "tilted plane", sheet(0.05, base)
    yield "curved sheet", sheet(0.2, base, curved=2.0)
    yield "thick sheet", sheet(0.1, base, thick=0.005)
    yield "blob", base + 0.02 * g.standard_normal((n, 3))
    yield "identical points", np.repeat(base[None], n, 0)
    yield "line", base + np.linspace(-0.1, 0.1, n)[:, None] * g.standard_normal(3)
    yield "two ends of a gap", np.concatenate([sheet(0.01, base)[: n // 2], sheet(0.01, base + 0.7)[: n - n // 2]])
    yield "far from the origin", sheet(2.0, 1e4 * np.array([1.0, -0.3, 0.07]))
    yield "small, far from the origin", sheet(1e-2, 100.0 * np.ones(3))


@pytest.mark.parametrize("n", [1, 2, 77, 128, 1000, 1024, 8191, 8192])
def test_patch_boxes_bound_the_distance_to_their_points(H, n):
    g = np.random.default_rng(n)
    zero = np.zeros((n, 3), np.float32)
    for name, P in _patches(g, n):
        P = np.ascontiguousarray(P, dtype=np.float32)
        p4, box = np.zeros((n, 4), np.float32), np.zeros(16, np.float32)
        p4[:, :3] = P
        H.h_obb_fit_patch(_p(p4), n, _p(box))
        assert not _d2(H, box, P, zero).any(), name
        Pd = P.astype(float)
        span = max(float(np.ptp(Pd, axis=0).max()), 1e-3)
        u = g.standard_normal((3000, 3))
        u /= np.linalg.norm(u, axis=1)[:, None]
        off = span * 10.0 ** g.uniform(-7, 2, 3000)
        x = Pd[g.integers(n, size=3000)] + off[:, None] * u
        xh = x.astype(np.float32)
        xl = (x - xh).astype(np.float32)
        x = xh.astype(float) + xl
        true = ((x - Pd[cKDTree(Pd).query(x)[1]]) ** 2).sum(1)
        got = _d2(H, box, xh, xl)
        assert (got <= BOUND * true).all(), (name, float((got / np.maximum(true, 1e-300)).max()))
        far = off > 20 * span
        assert (got[far] >= 0.5 * true[far]).all(), name
