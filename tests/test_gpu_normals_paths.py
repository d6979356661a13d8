"""The two ways a neighbourhood is found (by float distance, and again in FP64
where the K-th and the next distance are within float rounding) and the two ways
its axis is computed (Rayleigh quotient steps, and Jacobi where the smaller
eigenvalues are close), each against FP64 numpy on the same points."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fr():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2007_07627_gb300 import build
    build.build()
    import paper_2007_07627_gb300 as fr
    fr.lib()
    return fr


def _reference(Q, k, rows):
    """Covariances of the k nearest by (FP64 distance, index), and their eigen systems."""
    Q = Q.astype(np.float64)
    C = np.empty((len(rows), 3, 3))
    for a, i in enumerate(rows):
        d = ((Q - Q[i]) ** 2).sum(1)
        nb = Q[np.lexsort((np.arange(len(Q)), d))[:k]]
        e = nb - nb.mean(0)
        C[a] = e.T @ e / k
    return C, *np.linalg.eigh(C)


def _check(fr, Q, k):
    Q = np.ascontiguousarray(Q, dtype=np.float32)
    got = fr.estimate_normals(Q, k).astype(np.float64)
    rows = np.unique(np.linspace(0, len(Q) - 1, 400).astype(int))
    C, w, V = _reference(Q, min(k, len(Q)), rows)
    g = got[rows]
    assert np.abs(np.linalg.norm(g, axis=1) - 1.0).max() < 1e-6
    # the axis minimises the Rayleigh quotient, whose error is of second order in the float rounding of the normal
    # (3 x 2^-48 of the largest eigenvalue), and it is the eigenvector itself where the eigenvalue is simple
    g = g / np.linalg.norm(g, axis=1, keepdims=True)
    rq = np.einsum("nd,nde,ne->n", g, C, g)
    assert (rq - w[:, 0] <= 1e-12 * np.maximum(w[:, 2], 1e-300)).all()
    apart = w[:, 1] - w[:, 0] > 1e-6 * w[:, 2]
    sin = np.linalg.norm(np.cross(g, V[:, :, 0]), axis=1)
    assert (sin[apart] < 2e-7).all()
    return int(apart.sum())


@pytest.mark.parametrize("k", [3, 8, 30, 31, 32])
def test_ties_at_the_last_neighbour(fr, k):
    """A lattice (every distance repeated) and points given twice: float distances
    cannot order the last neighbours, the index does."""
    g = np.random.default_rng(k)
    h = np.stack(np.meshgrid(np.arange(40.0), np.arange(40.0)), -1).reshape(-1, 2)
    L = np.column_stack([h, np.sin(0.3 * h[:, 0])])
    _check(fr, L[g.permutation(len(L))], k)
    R = g.random((700, 3))
    _check(fr, np.concatenate([R, R])[g.permutation(1400)], k)


@pytest.mark.parametrize("thin", [1.0, 1e-2, 1e-4, 0.0])
def test_close_small_eigenvalues(fr, thin):
    """Points along lines: the two smaller eigenvalues are close or equal."""
    g = np.random.default_rng(3)
    t = np.arange(3000) * 0.01
    Q = np.column_stack([t, 1e-3 * thin * g.standard_normal(3000), 1.0001e-3 * thin * g.standard_normal(3000)])
    _check(fr, Q, 16)


@pytest.mark.parametrize("n", [3, 16, 33, 9728, 9729, 40000, 77825, 1217, 4864])
def test_points_per_warp(fr, n):
    """Sizes on both sides of the rule for the points per block; few points, ragged ends."""
    g = np.random.default_rng(n)
    u = g.random((n, 2))
    Q = np.column_stack([u, 0.2 * np.sin(6 * u[:, 0]) * np.cos(5 * u[:, 1])]) + 3.0
    assert _check(fr, Q, 30) > 0 or n < 4


def test_coordinates_beyond_float_distances(fr):
    """Squared distances that overflow float fall back to FP64 distances."""
    g = np.random.default_rng(9)
    _check(fr, g.random((500, 3)) * 1e25, 12)
