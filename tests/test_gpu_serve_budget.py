"""The serving loop's device-memory budget: everything a request and its target hold
is counted, and a request is either refused when it is submitted or served.

The sizes below follow the layout: 28 B per source point and 224 B per 256 of them,
a state of 3 to 5 KB (STATE bounds it with the roundings to 256 B); per target 16 B
per point, 64 B per node of L buckets and 64 B per oriented box."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N, M = 20_000, 2_000
L = 2048                                  # 1,250 buckets of 16
BOXES = 8 + 32 + 256 + L                  # oriented: 4 nodes padded to 8, then every third level
REQUEST = 28 * M + 224 * ((M + 255) // 256)
STATE = 6 * 1024
INDEX = 16 * N + 64 * L + 64 * BOXES
FP16 = 8 * N + 64 * BOXES


@pytest.fixture(scope="module")
def fr():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2007_07627_gb300 import build
    build.build()
    import paper_2007_07627_gb300 as fr
    fr.lib()
    return fr


@pytest.fixture()
def pair():
    g = np.random.default_rng(3)
    Q = g.random((N, 3)).astype(np.float32)
    P = (Q[g.integers(N, size=M)] + 0.002 * g.standard_normal((M, 3))).astype(np.float32)
    return Q, P


def _prm(fr, precision="fp64"):
    return fr.params_default("p2p", precision=precision, max_iters=5)


def _serve(srv, tickets, nsteps=8, steps=400):
    """Results of the tickets; None for those that have not finished after `steps` server steps."""
    res, most = {}, 0
    for _ in range(steps):
        flying, _ = srv.step(nsteps)
        most = max(most, flying)
        for t in tickets:
            r = srv.poll(t) if t not in res else None
            if r is not None:
                res[t] = r
        if len(res) == len(tickets):
            break
    return [res.get(t) for t in tickets], most


@pytest.mark.parametrize("precision", ["fp64", "fp16"])
def test_oriented_boxes_of_every_level_and_storage_count(fr, pair, precision):
    """A request with its target is refused just below what they hold, and served with it."""
    Q, P = pair
    t = fr.target_create(Q)
    need = REQUEST + INDEX
    # what an account of the buckets' boxes alone would come to
    short = REQUEST + 16 * N + 128 * L + STATE
    if precision == "fp16":
        fr.register(t, P, params=_prm(fr, "fp16"))      # builds the storage
        need += FP16
        short += 8 * N
    assert short < need
    srv = fr.Server(hbm_budget=short, max_slots=2)
    with pytest.raises(fr.FricpError) as ei:
        srv.submit(t, P, _prm(fr, precision))
    assert "budget" in str(ei.value)
    srv.destroy()
    srv = fr.Server(hbm_budget=need + STATE, max_slots=2)
    (r,), _ = _serve(srv, [srv.submit(t, P, _prm(fr, precision))])
    assert r is not None and r["status"] == "OK"
    srv.destroy()
    t.destroy()


def test_fp16_request_over_the_budget_is_refused_at_submit(fr, pair):
    """Accepted without its storage counted, it would wait at the head of the queue for ever."""
    Q, P = pair
    t = fr.target_create(Q)
    srv = fr.Server(hbm_budget=REQUEST + INDEX + FP16 // 2, max_slots=2)
    with pytest.raises(fr.FricpError) as ei:
        srv.submit(t, P, _prm(fr, "fp16"))
    assert "budget" in str(ei.value)
    (r,), _ = _serve(srv, [srv.submit(t, P, _prm(fr))])
    assert r is not None and r["status"] == "OK"
    srv.destroy()
    t.destroy()


def test_accepted_request_is_served_although_its_target_has_grown(fr, pair):
    """FP16 storage built between submit and admission takes the target over the budget."""
    Q, P = pair
    t = fr.target_create(Q)
    srv = fr.Server(hbm_budget=REQUEST + INDEX + STATE, max_slots=2)
    tickets = [srv.submit(t, P, _prm(fr)), srv.submit(t, P, _prm(fr))]
    fr.register(t, P, params=_prm(fr, "fp16"))
    res, most = _serve(srv, tickets)
    assert most == 1
    alone = fr.register(t, P, params=_prm(fr))
    for r in res:
        assert r is not None and r["status"] == "OK" and np.array_equal(r["R"], alone["R"])
    srv.destroy()
    t.destroy()


@pytest.mark.parametrize("room,together", [(FP16 - REQUEST // 2, 1), (FP16, 2)])
def test_storage_built_for_a_target_in_flight_is_charged(fr, pair, room, together):
    """An FP16 request joins an FP64 one on the same target only when the storage fits too."""
    Q, P = pair
    t = fr.target_create(Q)
    srv = fr.Server(hbm_budget=2 * (REQUEST + STATE) + INDEX + room, max_slots=2, steps_per_sync=1)
    prms = [fr.params_default("p2p", precision=p, max_iters=100, eps=1e-14) for p in ("fp64", "fp16")]
    res, most = _serve(srv, [srv.submit(t, P, prm) for prm in prms], nsteps=1)
    assert most == together and all(r is not None and r["status"] == "OK" for r in res)
    srv.destroy()
    t.destroy()


def test_memory_the_pool_keeps_is_free_to_a_server(fr):
    """What a destroyed target held and the pool kept is the server's to use."""
    import torch
    g = np.random.default_rng(4)
    fr.target_create(g.random((2_000_000, 3)).astype(np.float32)).destroy()   # index and sort: over 100 MB
    free, total = torch.cuda.mem_get_info()
    srv = fr.Server(hbm_budget=free + (32 << 20), max_slots=2)
    srv.destroy()
    with pytest.raises(fr.FricpError) as ei:
        fr.Server(hbm_budget=total + (1 << 30), max_slots=2)
    assert "free device memory" in str(ei.value)
