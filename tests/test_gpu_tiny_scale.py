"""Neighbour lists of point sets so small that squared distances underflow in float:
scaled by a power of two, which changes no bit of the coordinates' mantissas, a set
keeps its neighbours, hence its normals and (scaled) its spacing statistics."""
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


def _sheet(n):
    g = np.random.default_rng(n)
    u = g.random((n, 2))
    return np.stack([u[:, 0], u[:, 1], 0.2 * np.sin(4 * u[:, 0])], 1).astype(np.float32)


@pytest.mark.parametrize("exponent", [-40, -58, -62, -66])
@pytest.mark.parametrize("n", [70, 2000, 20_000])
def test_neighbours_do_not_depend_on_the_scale(fr, n, exponent):
    Q = _sheet(n)
    S = np.ldexp(Q, exponent).astype(np.float32)
    assert np.array_equal(np.ldexp(S.astype(float), -exponent), Q.astype(float))
    # the same sums in FP64, scaled: only the last float bits of a normal may differ
    d = np.abs(fr.estimate_normals(S, 16) - fr.estimate_normals(Q, 16)).max(1)
    assert (d <= 1e-5).all(), int((d > 1e-5).sum())
    a, b = fr.target_create(Q), fr.target_create(S)
    nu = fr.target_nu_min(a, "p2p_welsch")
    assert abs(np.ldexp(fr.target_nu_min(b, "p2p_welsch"), -exponent) - nu) <= 1e-12 * nu
    a.destroy()
    b.destroy()
