"""The group search (eight lanes per query, the box tree walked three levels at
a time) against exhaustive FP64 distances: target sizes around every depth of
the tree modulo three (the first round has 1, 2, 4 or 8 nodes) and around the
levels whose oriented boxes are fitted differently (128, 1,024, 8,192 points and
above), ragged query counts, exact ties (several equally near points, some of
them seen by the same lane), duplicates, and far-from-origin coordinates."""
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


def _dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).cuda()


def _brute(P, Q):
    """Lowest index among the smallest FP64 squared distances, and that distance."""
    P, Q = P.astype(np.float64), Q.astype(np.float64)
    idx = np.empty(len(P), np.int64)
    d2 = np.empty(len(P))
    for i in range(0, len(P), 64):
        e = ((P[i:i + 64, None] - Q[None]) ** 2).sum(-1)
        idx[i:i + 64] = e.argmin(1)
        d2[i:i + 64] = e.min(1)
    return idx, d2


def _check(fr, P, Q):
    t = fr.target_create(_dev(Q))
    idx, d2 = fr.closest_points(t, _dev(P))
    io, do = _brute(P, Q)
    assert np.array_equal(idx.cpu().numpy(), io)
    assert np.abs(d2.cpu().numpy() - do).max() <= 1e-12 * max(1.0, np.abs(P).max() ** 2)
    t.destroy()


@pytest.mark.parametrize("n", [1, 15, 16, 17, 31, 33, 64, 65, 127, 129, 255, 257, 512, 513, 1023, 1025, 2049, 4097,
                               8191, 8193, 16385, 65537, 131073, 300001])
def test_tree_depths_and_ragged_queries(fr, n):
    g = np.random.default_rng(n)
    u = g.random((n, 2))
    Q = np.stack([u[:, 0], u[:, 1], 0.1 * np.sin(7 * u[:, 0]) * np.cos(5 * u[:, 1])], 1).astype(np.float32)
    m = 37 if n > 20000 else 131
    P = np.concatenate([Q[g.integers(n, size=m // 2)] + 0.01 * g.standard_normal((m // 2, 3)),
                        1.4 * g.random((m - m // 2, 3)) - 0.2]).astype(np.float32)
    _check(fr, P, Q)


@pytest.mark.parametrize("side", [2, 3, 8, 20])
def test_exact_ties_go_to_the_lowest_index(fr, side):
    """Queries at lattice points, edge, face and cell centres: up to eight equally
    near targets, in one bucket or several; and every target present twice."""
    g = np.random.default_rng(side)
    L = np.stack(np.meshgrid(*[np.arange(side)] * 3, indexing="ij"), -1).reshape(-1, 3).astype(np.float32)
    P = np.concatenate([L[:50] + np.asarray(o, np.float32) for o in
                        [(0, 0, 0), (.5, 0, 0), (.5, .5, 0), (.5, .5, .5), (-.5, .5, 0)]])
    _check(fr, P, L[g.permutation(len(L))])
    D = np.concatenate([L, L])
    _check(fr, P, D[g.permutation(len(D))])


def test_far_from_the_origin_and_degenerate_patches(fr):
    g = np.random.default_rng(5)
    line = np.stack([np.linspace(0, 1, 3000), np.zeros(3000), np.zeros(3000)], 1)
    same = np.repeat(g.random((7, 3)), 300, 0)
    Q = (np.concatenate([line, same, g.random((4000, 3))]) + 4096.0).astype(np.float32)
    P = (Q[g.integers(len(Q), size=200)] + 0.05 * g.standard_normal((200, 3))).astype(np.float32)
    _check(fr, P, Q[g.permutation(len(Q))])


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("n", [1, 40, 130, 1030, 9000])
def test_both_search_layouts_agree(fr, n, precision):
    """Whole registrations through this search and through query tiles, bit for bit."""
    g = np.random.default_rng(n)
    Q = g.random((n, 3)).astype(np.float32)
    P = (g.random((333, 3)) * 0.9 + 0.05).astype(np.float32)
    t = fr.target_create(_dev(Q))
    a, b = (fr.register(t, _dev(P), params=fr.params_default("p2p_welsch" if n > 40 else "p2p", search=s, max_iters=20,
                                                             precision=precision), trace_capacity=500) for s in (0, 1))
    assert a["status"] == b["status"] and a["iterations"] == b["iterations"]
    assert np.array_equal(a["R"], b["R"]) and np.array_equal(a["t"], b["t"]) and np.array_equal(a["trace"], b["trace"])
    t.destroy()


@pytest.mark.parametrize("m", [(1 << 17) - 1, 1 << 17, (1 << 17) + 37])
def test_queries_dealt_by_cell(fr, m):
    """From 2^17 queries on the search deals them by cell first: points inside and
    far outside the target's box, duplicates and non-finite ones land at their own
    place, with the index and distance of a small call on the same points."""
    import torch
    g = np.random.default_rng(m)
    Q = np.concatenate([g.random((5000, 3)), np.repeat(g.random((1, 3)), 50, 0)]).astype(np.float32)
    P = np.concatenate([g.random((m - 4000, 3)), 40.0 * g.standard_normal((2000, 3)),
                        np.repeat(g.random((1, 3)), 1990, 0), np.full((10, 3), np.nan)]).astype(np.float32)
    P = P[g.permutation(m)]
    t, p = fr.target_create(_dev(Q)), _dev(P)
    T = np.eye(4)
    T[:3, 3] = (0.01, -0.02, 0.03)
    idx, d2 = fr.closest_points(t, p, T)
    for lo in (0, m // 2, m - 3001):
        i1, e1 = fr.closest_points(t, p[lo:lo + 3001], T)
        assert torch.equal(idx[lo:lo + 3001], i1) and torch.equal(d2[lo:lo + 3001].nan_to_num(-1.0), e1.nan_to_num(-1.0))
    near = np.flatnonzero(np.isfinite(P).all(1))[:200]
    io, _ = _brute(P[near].astype(np.float64) + T[:3, 3], Q)
    assert np.array_equal(idx.cpu().numpy()[near], io)
    t.destroy()
