"""The closest-point search in the FP32 and FP16-storage modes against exhaustive
FP64 distances, pass by pass of a registration: the energy of a recorded pass is
that of the nearest points (of FP16 storage: of the points as it decodes them) at
the recorded transform. A pruned nearest point shows as a larger energy.

Bounds, u = 2^-24. x = R p + t is formed in float from R and t rounded to float:
four roundings of terms no larger than |p| + |t| in each coordinate, so x is off by
at most d = 7 u (|p| + |t|); the nearest distance D then by at most d (for decoded
points, which this file rounds once more, d + u |q|). The squared distance, its
scale and their product take less than sixteen roundings. Before the first step
(T = I) x = p exactly, and d = 0."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U = 2.0 ** -24
SIZES = [1, 16, 17, 129, 1025, 8193, 70_000]   # every first level of the walk, every kind of patch box


@pytest.fixture(scope="module")
def fr():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2007_07627_gb300 import build
    build.build()
    import paper_2007_07627_gb300 as fr
    fr.lib()
    return fr


def _spread(v):
    """Bits 0..9 of v to bits 0, 3, ..., 27."""
    out = np.zeros_like(v)
    for b in range(10):
        out |= ((v >> b) & 1) << (3 * b)
    return out


def _decoded(Q):
    """Q as FP16 storage holds it: buckets of 16 in the order of 30-bit Morton keys
    (equal keys keep their order), half-precision offsets in each bucket's box."""
    f = np.float32
    lo, hi = Q.min(0), Q.max(0)
    ext = hi - lo
    inv = np.where(ext > 0, f(1) / np.where(ext > 0, ext, f(1)), f(0)).astype(f)
    k = np.clip((Q - lo) * inv * f(1024), 0, 1023).astype(np.int64)
    key = (_spread(k[:, 0]) << 2) | (_spread(k[:, 1]) << 1) | _spread(k[:, 2])
    S = Q[np.argsort(key, kind="stable")]
    out = np.empty_like(S)
    for b in range(0, len(S), 16):
        B = S[b:b + 16]
        l, e = B.min(0), B.max(0) - B.min(0)
        h = np.clip((B - l) / np.where(e > 0, e, f(1)), 0, 1).astype(np.float16)
        h[:, e == 0] = 0
        out[b:b + 16] = (h.astype(float) * e.astype(float) + l.astype(float)).astype(f)
    return out


def _nearest(X, Q):
    X, Q = X.astype(float), Q.astype(float)
    D = np.empty(len(X))
    j = np.empty(len(X), np.int64)
    for i in range(0, len(X), 16):
        e = ((X[i:i + 16, None] - Q[None]) ** 2).sum(-1)
        j[i:i + 16] = e.argmin(1)
        D[i:i + 16] = np.sqrt(e.min(1))
    return D, j


def _sets(n, kind):
    g = np.random.default_rng(n)
    if kind == "surface":   # a bent sheet, tilted: boxes far from axis-aligned
        u = g.random((n, 2))
        Q = np.stack([u[:, 0], u[:, 1], 0.4 * u[:, 0] + 0.3 * np.sin(5 * u[:, 1])], 1)
    else:
        Q = g.random((n, 3))
    m = 333 if n < 20_000 else 97
    near = Q[g.integers(n, size=m // 2)] + 0.02 * g.standard_normal((m // 2, 3))
    return Q.astype(np.float32), np.concatenate([near, 1.5 * g.random((m - m // 2, 3)) - 0.25]).astype(np.float32)


@pytest.mark.parametrize("kind", ["surface", "cube"])
@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("precision", ["fp32", "fp16"])
def test_every_pass_finds_the_nearest_points(fr, precision, n, kind):
    Q, P = _sets(n, kind)
    t = fr.target_create(Q)
    res, steps = fr.register_recorded(t, P, params=fr.params_default("p2p", precision=precision, max_iters=6),
                                      steps_capacity=64)
    t.destroy()
    assert len(steps) >= 1
    K = _decoded(Q) if precision == "fp16" else Q
    s, c = res["scale"], res["center"]
    for k, st in enumerate(steps):
        R, tn = st["T"][:3, :3], st["T"][:3, 3]
        tc = tn / s + c - R @ c
        D, j = _nearest(P.astype(float) @ R.T + tc, K)
        d = np.zeros(len(P)) if k == 0 else 7 * U * (np.linalg.norm(P, axis=1) + np.linalg.norm(tc))
        if precision == "fp16":
            d = d + U * np.linalg.norm(K[j], axis=1)
        E = s * s * (D ** 2).sum()
        tol = s * s * (2 * D * d + d * d + 16 * U * (D + d) ** 2).sum()
        assert abs(st["E"] - E) <= tol, (k, st["E"], E, tol)
