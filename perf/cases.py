"""The work a user of this library has it do, as cases that can be timed and checked.

Point-set pairs follow the package's synthetic workloads (paper_2007_07627_gb300/synth.py: torus,
sum-of-bumps height field, union of ellipsoids; two parallel cuts for the overlap, Gaussian noise,
uniform outliers, a random rigid motion), sampled here on the GPU so that preparing them is quick.

Families of cases ("op"):
  closest   the correspondence step alone, fr.closest_points (Eq. 3), target kept
  pass      one fused pass at a fixed transform, fr.eval_pass: energy, alignment and reduced sums
  index     a new target: fr.target_create and its nu_min statistics (fr.target_nu_min)
  normals   fr.estimate_normals for a scan without normals (k = 30, Sec. 6)
  register  a whole registration, fr.register (Alg. 1 / Alg. 2); with "new_target" the target is built
            in the call, as for a pair seen for the first time
  batch     many registrations at once, fr.batch_register, targets kept
"""
import math
import random

import numpy as np
import torch

import paper_2007_07627_gb300 as fr

DEV = "cuda"
F64 = torch.float64


# ----------------------------------------------------------------------------
# cases
# ----------------------------------------------------------------------------

def _case(op, kind, N, M, overlap, noise, outliers, **more):
    return dict(op=op, kind=kind, N=N, M=M, overlap=overlap, noise=noise, outliers=outliers, max_angle=25.0, **more)


def listed():
    # a small scan against a small model, once: the smallest call, all latency
    torus = ("torus", 2000, 2000, 1.0, 0.002, 0.0)
    # a depth scan against another, 60% overlap and 10% outliers
    field = ("height_field", 100_000, 80_000, 0.6, 0.005, 0.10)
    # a laser scan against a large model, half overlapping
    ellipsoids = ("ellipsoids", 500_000, 200_000, 0.5, 0.003, 0.05)
    return [
        dict(_case("closest", *torus, offset_deg=3.0), name="closest_torus_2k"),
        # from the unaligned start: loose distances, no warm start
        dict(_case("closest", *field, offset_deg=-1.0), name="closest_field_80k"),
        # the largest sets served, ragged sizes
        dict(_case("closest", "ellipsoids", 1_000_003, 999_001, 0.75, 0.003, 0.05, offset_deg=1.0),
             name="closest_ellipsoids_1m"),
        dict(_case("pass", *torus, offset_deg=3.0, variant="p2p", nu=0.0), name="pass_p2p_torus_2k"),
        dict(_case("pass", *field, offset_deg=2.0, variant="p2p_welsch", nu=0.02), name="pass_welsch_field_80k"),
        dict(_case("pass", *ellipsoids, offset_deg=2.0, variant="p2pl_welsch", nu=0.01),
             name="pass_plane_ellipsoids_200k"),
        # a new model: its index and the statistics of its spacing
        dict(_case("index", *ellipsoids, variant="p2pl_welsch"), name="index_ellipsoids_500k"),
        # a scan without normals
        dict(_case("normals", "height_field", 100_000, 16, 1.0, 0.005, 0.0, k=30), name="normals_field_100k"),
        # tracking a small part against its model: many short registrations
        dict(_case("register", *torus, variant="p2p", precision="fp64", new_target=False),
             name="register_p2p_torus_2k"),
        # the lighter arithmetic a user may choose
        dict(_case("register", *field, variant="p2pl_welsch", precision="fp32", new_target=False),
             name="register_plane_fp32_field_80k"),
        # the benchmark's headline: a pair seen for the first time
        dict(_case("register", *ellipsoids, variant="p2pl_welsch", precision="fp64", new_target=True),
             name="register_plane_ellipsoids_200k"),
        # many pairs of mixed sizes, surfaces and variants
        dict(op="batch", pairs=16, lo=2000, hi=200_000, mix=4, name="batch_16_pairs"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["closest", "pass", "index", "normals", "register", "batch"])
    kind = rng.choice(["torus", "height_field", "ellipsoids"])
    if op == "batch":
        return dict(op=op, pairs=rng.randint(3, 14), lo=1000, hi=_log(rng, 5000, 100_000), mix=rng.randint(0, 1 << 20))
    overlap, noise, outliers = rng.uniform(0.5, 1.0), rng.uniform(0.001, 0.005), rng.uniform(0.0, 0.1)
    variant = rng.choice(["p2p", "p2p_welsch", "p2pl_welsch"])
    top = {"closest": 1_000_000, "pass": 500_000, "index": 1_000_000, "normals": 200_000, "register": 100_000}[op]
    N, M = _log(rng, 1000, top), _log(rng, 1000, top)
    c = _case(op, kind, N, M, overlap, noise, outliers)
    if op == "closest":
        c.update(offset_deg=rng.choice([-1.0, rng.uniform(0.0, 10.0)]))
    elif op == "pass":
        c.update(offset_deg=rng.uniform(0.0, 10.0), variant=variant, nu=math.exp(rng.uniform(math.log(1e-3), math.log(0.1))))
    elif op == "index":
        c.update(variant=rng.choice(["p2p_welsch", "p2pl_welsch"]))
    elif op == "normals":
        c.update(k=rng.choice([8, 16, 30]))
    else:
        c.update(variant=variant, precision=rng.choice(["fp64", "fp64", "fp32", "fp16"]), new_target=rng.random() < 0.5)
    return c


# ----------------------------------------------------------------------------
# surfaces, sampled uniformly by area on the GPU
# ----------------------------------------------------------------------------

def _unit(v):
    return v / v.norm(dim=-1, keepdim=True)


def _rotation(axis, angle):
    x, y, z = (float(v) for v in axis)
    K = np.array([[0.0, -z, y], [z, 0.0, -x], [-y, x, 0.0]])
    return np.eye(3) + math.sin(angle) * K + (1.0 - math.cos(angle)) * (K @ K)


class _Surface:
    def __init__(self, kind, g):
        self.kind, self.g = kind, g
        if kind == "height_field":
            self.a, self.s, self.c = 0.3 * self.u(16) - 0.15, 0.05 + 0.15 * self.u(16), self.u(16, 2)
            gx = torch.linspace(0, 1, 161, dtype=F64, device=DEV)
            _, grad = self.height(torch.cartesian_prod(gx, gx))
            self.amax = 1.1 * float((1 + (grad ** 2).sum(1)).sqrt().max())
        elif kind == "ellipsoids":
            self.c, self.ax = self.u(8, 3), 0.1 + 0.2 * self.u(8, 3)
            q, _ = np.linalg.qr(self.n(8, 3, 3).cpu().numpy())
            self.rot = torch.from_numpy(q).to(DEV)
            self.A = torch.einsum("kij,kj,klj->kil", self.rot, 1.0 / self.ax ** 2, self.rot)
            p, (a, b, c) = 1.6075, self.ax.unbind(1)
            self.w = (((a * b) ** p + (a * c) ** p + (b * c) ** p) / 3) ** (1 / p)

    def u(self, *shape):
        return torch.rand(*shape, generator=self.g, dtype=F64, device=DEV)

    def n(self, *shape):
        return torch.randn(*shape, generator=self.g, dtype=F64, device=DEV)

    def height(self, xy):
        d = xy[:, None] - self.c
        e = self.a * torch.exp(-(d ** 2).sum(-1) / (2 * self.s ** 2))
        return e.sum(1), -(e[..., None] * d / (self.s ** 2)[:, None]).sum(1)

    def draw(self, n):
        if self.kind == "torus":
            th, ph, v = 2 * math.pi * self.u(n), 2 * math.pi * self.u(n), self.u(n)
            ok = v * 1.4 <= 1.0 + 0.4 * ph.cos()
            th, ph = th[ok], ph[ok]
            nx = torch.stack([ph.cos() * th.cos(), ph.cos() * th.sin(), ph.sin()], 1)
            return torch.stack([th.cos(), th.sin(), torch.zeros_like(th)], 1) + 0.4 * nx, nx
        if self.kind == "height_field":
            xy = self.u(n, 2)
            z, grad = self.height(xy)
            ok = self.u(n) * self.amax <= (1 + (grad ** 2).sum(1)).sqrt()
            xy, z, grad = xy[ok], z[ok], grad[ok]
            return torch.cat([xy, z[:, None]], 1), _unit(torch.cat([-grad, torch.ones_like(z)[:, None]], 1))
        k = torch.multinomial(self.w.float(), n, replacement=True, generator=self.g)
        u, ax = _unit(self.n(n, 3)), self.ax[k]
        ok = self.u(n) <= (u / ax).norm(dim=1) * ax.min(1)[0]
        k, u, ax = k[ok], u[ok], ax[ok]
        x = self.c[k] + torch.einsum("nij,nj->ni", self.rot[k], ax * u)
        nx = _unit(torch.einsum("nij,nj->ni", self.A[k], x - self.c[k]))
        d = x[:, None] - self.c
        inside = torch.einsum("nki,kij,nkj->nk", d, self.A, d) < 1.0
        inside[torch.arange(k.numel(), device=DEV), k] = False
        ok = ~inside.any(1)
        return x[ok], nx[ok]

    def fill(self, n, keep):
        pts, nrm, have = [], [], 0
        while have < n:
            x, nx = self.draw(max(4096, 3 * (n - have)))
            if keep is not None:
                x, nx = x[keep(x)], nx[keep(x)]
            pts.append(x)
            nrm.append(nx)
            have += x.shape[0]
        return torch.cat(pts)[:n], torch.cat(nrm)[:n]


def _pair(case, seed):
    """Target Q and its normals, source P (float32 CUDA tensors), the motion taking P onto Q and Q's diagonal."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    s = _Surface(case["kind"], g)
    N, M = case["N"], case["M"]
    keep_t = keep_s = None
    if case["overlap"] < 1.0:
        dim = 2 if case["kind"] == "height_field" else 3
        a = _unit(s.n(dim))
        v = s.draw(100_000)[0][:, :dim] @ a
        f = 1.0 / (2.0 - case["overlap"])
        lo, hi = float(torch.quantile(v, 1.0 - f)), float(torch.quantile(v, f))
        keep_t, keep_s = (lambda x: x[:, :dim] @ a >= lo), (lambda x: x[:, :dim] @ a <= hi)
    Q, nQ = s.fill(N, keep_t)
    diag = float((Q.max(0)[0] - Q.min(0)[0]).norm())
    out = round(case["outliers"] * M)
    S, _ = s.fill(M - out, keep_s)
    S = S + case["noise"] * diag * s.n(M - out, 3)
    if out:
        lo3, hi3 = S.min(0)[0], S.max(0)[0]
        S = torch.cat([S, lo3 + (hi3 - lo3) * s.u(out, 3)])
    S = S[torch.randperm(M, generator=g, device=DEV)]
    R = _rotation(_unit(s.n(3)).cpu(), math.radians(case["max_angle"]) * float(s.u(1)))
    t = ((2.0 * s.u(3) - 1.0) * 0.1 * diag).cpu().numpy()
    P = S @ torch.from_numpy(R.T).to(DEV) + torch.from_numpy(t).to(DEV)
    T = np.eye(4)
    T[:3, :3], T[:3, 3] = R.T, -(R.T @ t)
    off = case.get("offset_deg", 0.0)
    if off > 0.0:   # a transform part of the way: turned about the target's middle
        c = Q.mean(0).cpu().numpy()
        D = np.eye(4)
        D[:3, :3] = _rotation(_unit(s.n(3)).cpu(), math.radians(off))
        D[:3, 3] = c - D[:3, :3] @ c
        T = D @ T
    elif off < 0.0:
        T = np.eye(4)
    return Q.float().contiguous(), nQ.float().contiguous(), P.float().contiguous(), T, diag


def _normalised(T, s, c):
    Tn = np.eye(4)
    Tn[:3, :3] = T[:3, :3]
    Tn[:3, 3] = s * (T[:3, :3] @ c + T[:3, 3] - c)
    return Tn


def _batch_cases(case):
    """The pairs of a batch: sizes, surfaces and variants from the mix alone."""
    r = random.Random(case["mix"])
    out = []
    for k in range(case["pairs"]):
        c = _case("register", r.choice(["torus", "height_field", "ellipsoids"]), _log(r, case["lo"], case["hi"]),
                  _log(r, case["lo"], case["hi"]), r.uniform(0.5, 1.0), 0.003, r.uniform(0.0, 0.1))
        out.append(dict(c, variant=("p2p", "p2p_welsch", "p2pl_welsch")[k % 3]))
    return out


# ----------------------------------------------------------------------------
# prepare and run
# ----------------------------------------------------------------------------

def prepare(case, seed):
    op = case["op"]
    if op == "batch":
        targets, sources, params = [], [], []
        for k, c in enumerate(_batch_cases(case)):
            Q, nQ, P, _, _ = _pair(c, seed * 1000 + k)
            targets.append(fr.target_create(Q, nQ if c["variant"] == "p2pl_welsch" else None))
            sources.append(P)
            params.append(fr.params_default(c["variant"]))
        return dict(op=op, targets=targets, sources=sources, params=params)
    Q, nQ, P, T, diag = _pair(case, seed)
    plane = case.get("variant") == "p2pl_welsch"
    st = dict(op=op)
    if op == "closest":
        st.update(target=fr.target_create(Q), P=P, T=T)
    elif op == "pass":
        c, s = Q.double().mean(0).cpu().numpy(), 1.0 / diag
        st.update(target=fr.target_create(Q, nQ if plane else None), P=P, variant=case["variant"],
                  T=_normalised(T, s, c), nu=case["nu"], scale=s, center=c)
    elif op == "index":
        st.update(Q=Q, normals=nQ if plane else None, variant=case["variant"])
    elif op == "normals":
        st.update(Q=Q, k=case["k"])
    else:
        st.update(Q=Q, normals=nQ if plane else None, P=P,
                  params=fr.params_default(case["variant"], precision=case["precision"]))
        if not case["new_target"]:
            st["target"] = fr.target_create(st.pop("Q"), st.pop("normals"))
    return st


def _results(rs):
    d = {k: np.stack([np.asarray(r[k]) for r in rs]) for k in ("R", "t")}
    for k in ("final_energy", "nu_max", "nu_min", "scale"):
        d[k] = np.array([r[k] for r in rs], np.float64)
    for k in ("iterations", "corr_passes", "stages", "reverts", "aa_accepted", "line_search_trials"):
        d[k] = np.array([r[k] for r in rs], np.int64)
    d["ok"] = np.array([r["status"] == "OK" for r in rs], np.int64)
    return d


def run(state):
    op = state["op"]
    if op == "closest":
        idx, d2 = fr.closest_points(state["target"], state["P"], state["T"])
        return {"idx": idx, "d2": d2}
    if op == "pass":
        out = fr.eval_pass(state["target"], state["P"], state["variant"], state["T"], nu=state["nu"] or 1.0,
                           scale=state["scale"], center=state["center"])
        return {"energy": out[:1], "aligned": out[1:16], "sums": out[16:]}
    if op == "index":
        target = fr.target_create(state["Q"], state["normals"])
        return {"nu_min": np.array([fr.target_nu_min(target, state["variant"])])}
    if op == "normals":
        return {"normals": fr.estimate_normals(state["Q"], state["k"])}
    if op == "register":
        target = state["target"] if "target" in state else fr.target_create(state["Q"], state["normals"])
        return _results([fr.register(target, state["P"], params=state["params"])])
    return _results(fr.batch_register(state["targets"], state["sources"], state["params"]))


# ----------------------------------------------------------------------------
# work and 64-bit values
# ----------------------------------------------------------------------------

def work(case):
    """Inputs read once, outputs written once, and the arithmetic of one pass over the source at known
    correspondences (a registration: its first pass; the search itself has no fixed count)."""
    if case["op"] == "batch":
        parts = [work(dict(c, precision="fp64", new_target=False)) for c in _batch_cases(case)]
        return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}
    N, M, op = case["N"], case["M"], case["op"]
    nrm = 12 * N if case.get("variant") == "p2pl_welsch" else 0
    per_point = {"p2p": 70, "p2p_welsch": 95, "p2pl_welsch": 165}
    if op == "closest":
        return {"bytes": 12 * N + 12 * M + 16 * M, "flops": 26 * M}
    if op == "pass":
        return {"bytes": 12 * N + nrm + 12 * M + 384, "flops": per_point[case["variant"]] * M}
    if op == "index":
        return {"bytes": 12 * N + nrm + 8, "flops": (6 * 8 + (6 * 6 if nrm else 0)) * N}
    if op == "normals":
        return {"bytes": 24 * N, "flops": (case["k"] * 20 + 200) * N}
    return {"bytes": 12 * N + nrm + 12 * M + 200, "flops": per_point[case["variant"]] * M}


def _nearest(X, Q, k, exclude_self=False):
    """Indices and squared distances of the k nearest rows of Q for each row of X, exhaustively in 64 bits."""
    idx, d2 = [], []
    step = max(1, 100_000_000 // Q.shape[0])
    for i in range(0, X.shape[0], step):
        x = X[i:i + step]
        d = (x[:, None, 0] - Q[None, :, 0]).square_()
        for a in (1, 2):
            d += (x[:, None, a] - Q[None, :, a]).square_()
        if exclude_self:
            j = torch.arange(x.shape[0], device=DEV)
            d[j, i + j] = math.inf
        if k == 1:
            v, j = d.min(1, keepdim=True)
        else:
            v, j = d.topk(k, dim=1, largest=False)
        idx.append(j)
        d2.append(v)
    return torch.cat(idx), torch.cat(d2)


def _hat(v):
    return np.array([[0.0, -v[2], v[1]], [v[2], 0.0, -v[0]], [-v[1], v[0], 0.0]])


def _se3_log(T):
    """[w; u] with exp([[w^, u], [0, 0]]) = T, for rotation angles below pi."""
    R = T[:3, :3]
    v = 0.5 * np.array([R[2, 1] - R[1, 2], R[0, 2] - R[2, 0], R[1, 0] - R[0, 1]])
    sn, cs = np.linalg.norm(v), 0.5 * (np.trace(R) - 1.0)
    th = math.atan2(sn, cs)
    w = v * (th / sn) if sn > 0.0 else v
    V, term, W = np.eye(3), np.eye(3), _hat(w)   # V = sum W^k / (k + 1)!
    for k in range(1, 40):
        term = term @ W / (k + 1)
        V = V + term
    return np.concatenate([w, np.linalg.solve(V, T[:3, 3])])


def _plane_step(xi, T, Szz, SzB):
    """xi + d of the Gauss-Newton step: B's gradient is (L J)^T z for z = [y x n; n], with J the left Jacobian of
    SE(3) at xi and L = [[I, 0], [-t^, I]] (dx = w x x + v, and x = y + t)."""
    ad = np.zeros((6, 6))
    ad[:3, :3] = ad[3:, 3:] = _hat(xi[:3])
    ad[3:, :3] = _hat(xi[3:])
    J, term = np.eye(6), np.eye(6)
    for k in range(1, 40):
        term = term @ ad / (k + 1)
        J = J + term
    L = np.eye(6)
    L[3:, :3] = -_hat(T[:3, 3])
    K = (L @ J).T
    return xi + np.linalg.solve(K @ Szz @ K.T, -K @ SzB)


def _exact_pass(case, Q, nQ, P, T, diag):
    c, s = Q.double().mean(0), 1.0 / diag
    Tn = _normalised(T, s, c.cpu().numpy())
    q64, p64 = Q.double(), P.double()
    Rt, tt = torch.from_numpy(Tn[:3, :3]).to(DEV), torch.from_numpy(Tn[:3, 3]).to(DEV)
    pc = p64 - c
    y = s * (pc @ Rt.T)
    x = (y + tt) / s + c
    j = _nearest(x, q64, 1)[0][:, 0]
    qc, e = q64[j] - c, s * (x - q64[j])
    robust, nu = case["variant"] != "p2p", case["nu"] or 1.0
    out = np.zeros(48)
    if case["variant"] == "p2pl_welsch":
        n = nQ.double()[j]
        B = (e * n).sum(1)
        g = torch.exp(-B ** 2 / (2 * nu * nu))
        z = torch.cat([torch.linalg.cross(y, n), n], 1)
        Szz, SzB = ((g[:, None] * z).T @ z).cpu().numpy(), ((g * B)[:, None] * z).sum(0).cpu().numpy()
        E = float((1 - g).sum())
        out[1:7] = _plane_step(_se3_log(Tn), Tn, Szz, SzB)
        out[16:37], out[37:43], out[43] = Szz[np.triu_indices(6)], SzB, E
    else:
        d2 = (e ** 2).sum(1)
        w = torch.exp(-d2 / (2 * nu * nu)) if robust else torch.ones_like(d2)
        E = float((1 - w).sum() if robust else d2.sum())
        W, wp, wq = float(w.sum()), (w[:, None] * pc).sum(0).cpu().numpy(), (w[:, None] * qc).sum(0).cpu().numpy()
        wpq = ((w[:, None] * pc).T @ qc).cpu().numpy()
        pb, qb = wp / W, wq / W
        U, _, Vt = np.linalg.svd(wpq - W * np.outer(pb, qb))
        R = Vt.T @ np.diag([1.0, 1.0, np.linalg.det(Vt.T @ U.T)]) @ U.T
        out[1:10], out[10:13] = R.reshape(9), s * (qb - R @ pb)
        out[16], out[17:20], out[20:23], out[23:32], out[32] = W, wp, wq, wpq.reshape(9), E
    out[0] = E
    return {"energy": out[:1], "aligned": out[1:16], "sums": out[16:]}


def exact(case, seed):
    op = case["op"]
    if op in ("register", "batch"):
        return None   # an iterative method run to a tolerance: no closed value
    pairs = case["N"] * (case["N"] if op in ("index", "normals") else case["M"])
    if pairs > (1.5e11 if op in ("closest", "pass") else 2.0e10):
        return None   # exhaustive neighbours would take too long
    Q, nQ, P, T, diag = _pair(case, seed)
    if op == "closest":
        R, t = torch.from_numpy(T[:3, :3]).to(DEV), torch.from_numpy(T[:3, 3]).to(DEV)
        idx, d2 = _nearest(P.double() @ R.T + t, Q.double(), 1)
        return {"idx": idx[:, 0], "d2": d2[:, 0]}
    if op == "pass":
        return _exact_pass(case, Q, nQ, P, T, diag)
    q64 = Q.double()
    if op == "index":
        idx, d2 = _nearest(q64, q64, 6, exclude_self=True)
        if case["variant"] == "p2pl_welsch":
            h = ((q64[idx] - q64[:, None]) * nQ.double()[:, None]).sum(-1).abs().sort(1)[0]
        else:
            h = d2.sqrt()
        v = (0.5 * (h[:, 2] + h[:, 3])).sort()[0]   # the median of six, then of all points
        med = 0.5 * float(v[(v.numel() - 1) // 2] + v[v.numel() // 2])
        return {"nu_min": np.array([med / 6.0 if case["variant"] == "p2pl_welsch" else med / (3.0 * math.sqrt(3.0))])}
    k = min(case["k"], case["N"])
    nb = q64[_nearest(q64, q64, k)[0]]
    d = nb - nb.mean(1, keepdim=True)
    _, vec = np.linalg.eigh((torch.einsum("nki,nkj->nij", d, d) / k).cpu().numpy())
    n = torch.from_numpy(np.ascontiguousarray(vec[:, :, 0])).to(DEV)
    return {"normals": torch.where(((n * -q64).sum(1) < 0)[:, None], -n, n)}
