"""nu_min (six nearest neighbours of every target point) on targets that take each
path of its kernels: tiles by float distance, ties (FP64 tiles), tiles scattered
over a gap of the Morton order (searched point by point), point-by-point ties,
and sizes around a tile and around the smallest tree; exact FP64 values."""
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


def _reference(Q, N):
    Q, N = Q.astype(np.float64), N.astype(np.float64)
    d6, h6 = np.empty((len(Q), 6)), np.empty((len(Q), 6))
    for i in range(len(Q)):
        e = Q - Q[i]
        d2 = (e ** 2).sum(1)
        d2[i] = np.inf
        k = np.lexsort((np.arange(len(Q)), d2))[:6]
        d6[i] = np.sqrt(d2[k])
        h6[i] = np.sort(np.abs(e[k] @ N[i]))
    d6.sort(1)
    return np.median(0.5 * (d6[:, 2] + d6[:, 3])) / (3 * np.sqrt(3)), np.median(0.5 * (h6[:, 2] + h6[:, 3])) / 6


def _check(fr, Q):
    g = np.random.default_rng(len(Q))
    Q = np.ascontiguousarray(Q[g.permutation(len(Q))], dtype=np.float32)
    N = g.standard_normal(Q.shape)
    N = (N / np.linalg.norm(N, axis=1, keepdims=True)).astype(np.float32)
    t = fr.target_create(Q, N)
    ref = _reference(Q, N)
    for v, r in zip(("p2p_welsch", "p2pl_welsch"), ref):
        assert abs(fr.target_nu_min(t, v) - r) <= 1e-13 * max(r, 1e-3)
    t.destroy()


@pytest.mark.parametrize("n", [7, 33, 64, 65, 96, 257, 1000, 3001])
def test_random_surfaces(fr, n):
    g = np.random.default_rng(n)
    u = g.random((n, 2))
    _check(fr, np.column_stack([u, 0.1 * np.sin(6 * u[:, 0])]))


def test_ties_and_duplicates(fr):
    L = np.stack(np.meshgrid(*[np.arange(12.0)] * 3), -1).reshape(-1, 3)
    _check(fr, L)
    g = np.random.default_rng(1)
    R = g.random((400, 3))
    _check(fr, np.concatenate([R, R, R[:100]]))


def test_scattered_tiles(fr):
    """Dense clusters far apart, of sizes that put the boundary of two clusters inside
    many tiles: those tiles reach everything between."""
    g = np.random.default_rng(2)
    parts = [g.random((int(k), 3)) * 1e-3 + c for k, c in zip(g.integers(5, 60, 150), g.random((150, 3)) * 10)]
    _check(fr, np.concatenate(parts + [g.random((1500, 3)) * 10]))
    # two tight clusters and a filled box between them: lattice points, so ties as well
    L = np.stack(np.meshgrid(*[np.arange(11.0)] * 3), -1).reshape(-1, 3)
    _check(fr, np.concatenate([L, g.random((23, 3)) * 1e-3 - 90.0, g.random((23, 3)) * 1e-3 + 90.0]))
