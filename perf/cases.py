"""What is measured: passes of the indexing path and of the learned proposal,
through the public Python entry points.

A case is a dict of plain values; ``listed`` gives the named ones, ``draw``
more of the same ranges.  Inputs are synthetic polycrystals made here (white
beam, flat detectors, rotation about +y, Gaussian spot noise, outliers) from
the case and the seed alone, in 64 bits and rounded once to the arrays that a
program hands to the library.  ``exact`` computes the results in 64 bits from
the same rounded inputs with torch and none of this repository's code.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_2404_06478_gb300 import api
from paper_2404_06478_gb300 import em as em_mod
from paper_2404_06478_gb300 import proposal as pr
from paper_2404_06478_gb300.autograd import ot_weighted_cost

LOG2E = math.log2(math.e)
SIGMA_MM = 0.5         # spot noise of every workload
CUBE_MM = 5.0          # sample cube
LATTICE_A = 2.87       # bcc iron
DEV = "cuda"


# ------------------------------------------------------------------- cases
def listed():
    return [
        # an E-step of the 5-grain configuration: the smallest solve, launches and latency
        dict(name="estep_tiny", kind="estep", grains=5, hmax=4, T=10, span=180.0, outliers=0.10, geometry="flat",
             eps=1.0, n_iter=100, mode=0, harvest=True, cols=False),
        # the unbalanced E-step on two tilted detectors with the column read-out, few grains, odd sizes
        dict(name="estep_tilted_unbalanced", kind="estep", grains=23, hmax=6, T=17, span=360.0, outliers=0.30,
             geometry="tilted", eps=4.0, n_iter=100, mode=2, harvest=True, cols=True),
        # the E-step of the 100-grain configuration at the final temperature, with its read-out
        dict(name="estep_medium", kind="estep", grains=100, hmax=6, T=60, span=360.0, outliers=0.30, geometry="flat",
             eps=1.0, n_iter=200, mode=0, harvest=True, cols=False),
        # an early step of the annealed EM (half-way down from 100 eps) with per-angle dustbins: no read-out, as
        # the EM's steps take it
        dict(name="estep_warm", kind="estep", grains=317, hmax=6, T=45, span=360.0, outliers=0.60, geometry="flat",
             eps=21.0, n_iter=100, mode=1, harvest=False, cols=False),
        # the E-step of the 1000-grain configuration at the final temperature: the largest solve
        dict(name="estep_full", kind="estep", grains=1000, hmax=6, T=90, span=360.0, outliers=0.70, geometry="flat",
             eps=1.0, n_iter=200, mode=0, harvest=True, cols=False),
        # the same polycrystal through the sparse E-step (32 nearest neighbours)
        dict(name="sparse_full", kind="sparse", grains=1000, hmax=6, T=90, span=360.0, outliers=0.70,
             geometry="flat", eps=1.0, n_iter=200, mode=0, rho=32),
        # an M-step (Newton on positions, majorise-minimise on rotations) of a few hundred grains
        dict(name="mstep_large", kind="mstep", grains=300, hmax=6, T=90, span=360.0, outliers=0.70, geometry="flat",
             eps=1.0),
        # forward and backward of the differentiable OT cost, the gradient-check configuration
        dict(name="gradient_small", kind="grad", grains=50, hmax=6, T=20, span=360.0, outliers=0.30,
             geometry="flat", eps=1.0),
        # a whole annealed EM solve through the solver object: 20 steps from 100 eps down to eps
        dict(name="em_mid", kind="em", grains=60, hmax=6, T=20, span=360.0, outliers=0.30, geometry="flat", eps=1.0,
             n_em=20, n_iter=100),
        # single-grain fits: a slice of the start scan on the 100-grain configuration (40 annealed steps, the
        # visible spots listed again at each)
        dict(name="fit_medium", kind="fit", grains=100, hmax=6, T=60, span=360.0, outliers=0.30, geometry="flat",
             eps=1.0, starts=3000, k_max=40, anneal=1000.0),
        # one training step of the set encoder: sets of 64 single-grain scenes x 32 seeds, forward, backward, Adam
        dict(name="train_2048", kind="train", scenes=64, per_scene=32, hmax=6, T=90, span=360.0, outliers=0.70,
             geometry="flat"),
        # learned proposals for 2500 seed spots of the 100-grain configuration
        dict(name="propose_2500", kind="propose", grains=100, hmax=6, T=60, span=360.0, outliers=0.30,
             geometry="flat", seeds=2500),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["estep"] * 5 + ["sparse", "mstep", "grad", "em", "fit", "train", "propose"])
    hmax = rng.choice([4, 6, 6])
    c = dict(kind=kind, hmax=hmax, T=rng.randint(10, 90), span=rng.choice([180.0, 360.0]),
             outliers=round(rng.uniform(0.1, 0.7), 2), geometry=rng.choice(["flat", "flat", "tilted"]))
    if kind == "estep":
        mode = rng.choice([0, 0, 1, 2])
        c.update(grains=_log_int(rng, 5, 700), eps=round(math.exp(rng.uniform(0.0, math.log(100.0))), 2),
                 n_iter=rng.choice([50, 100, 200]), mode=mode, harvest=rng.random() < 0.5, cols=rng.random() < 0.25)
        if mode == 2:
            c["eps"] = max(c["eps"], 4.0)
        # the largest solves run near the final temperature, the hot ones stay smaller
        if c["eps"] > 3.0:
            c["grains"] = min(c["grains"], 350)
            c["n_iter"] = min(c["n_iter"], 100)
    elif kind == "sparse":
        c.update(grains=_log_int(rng, 20, 900), eps=round(math.exp(rng.uniform(0.0, math.log(10.0))), 2),
                 n_iter=rng.choice([50, 100, 200]), mode=rng.choice([0, 1]), rho=rng.choice([8, 16, 32]))
    elif kind == "mstep":
        c.update(grains=_log_int(rng, 20, 300), eps=round(math.exp(rng.uniform(0.0, math.log(20.0))), 2))
    elif kind == "grad":
        c.update(grains=_log_int(rng, 5, 200), eps=round(math.exp(rng.uniform(0.0, math.log(20.0))), 2))
    elif kind == "em":
        c.update(grains=_log_int(rng, 10, 80), T=rng.randint(10, 30), eps=1.0, n_em=rng.choice([8, 12, 20]),
                 n_iter=rng.choice([50, 100]), geometry="flat")
    elif kind == "fit":
        c.update(grains=_log_int(rng, 5, 100), T=rng.randint(10, 60), eps=1.0, starts=_log_int(rng, 100, 3000),
                 k_max=rng.choice([8, 20, 40]), anneal=rng.choice([100.0, 1000.0]))
    elif kind == "train":
        c.update(scenes=rng.randint(8, 64), per_scene=rng.choice([8, 17, 32]), geometry="flat", hmax=6)
    else:
        c.update(grains=_log_int(rng, 5, 100), T=rng.randint(10, 60), geometry="flat", seeds=_log_int(rng, 50, 2500))
    return c


# ---------------------------------------------------------- the experiment
class _Detector:
    def __init__(self, centre, normal, half, D=0.0):
        self.centre, self.normal, self.half, self.D = centre, normal, half, D

    def axes(self):
        n = np.asarray(self.normal, np.float64)
        n = n / np.linalg.norm(n)
        a1 = np.array([n[2], 0.0, -n[0]])
        a1 = a1 / np.linalg.norm(a1)
        return n, a1, np.cross(n, a1)


class _Geometry:
    """Beam, band, cost length and detectors, as api.geometry_struct reads them
    (every number rounded to 32 bits, so that both sides see the same)."""

    def __init__(self, D, detectors):
        self.beam, self.lam_min, self.lam_max, self.D, self.detectors = (0.0, 0.0, 1.0), 1.0, 4.0, D, detectors


def _geometry(name):
    f = lambda v: float(np.float32(v))
    if name == "flat":
        dets = (_Detector((0.0, 0.0, 200.0), (0.0, 0.0, 1.0), 128.0),
                _Detector((0.0, 0.0, -200.0), (0.0, 0.0, 1.0), 128.0))
        return _Geometry(200.0, dets)
    a = math.radians(8.0)
    dets = (_Detector((10.0, 0.0, 125.0), (0.0, 0.0, 1.0), 128.0, 125.0),
            _Detector((0.0, f(165.0 * math.sin(a)), f(-165.0 * math.cos(a))), (0.0, f(-math.sin(a)), f(math.cos(a))),
                      128.0, 165.0))
    return _Geometry(165.0, dets)


def _planes(hmax):
    """bcc plane table: unit directions, base spacings, harmonic counts."""
    out = []
    r = range(-hmax, hmax + 1)
    for p in itertools.product(r, r, r):
        if p <= (0, 0, 0) or math.gcd(math.gcd(p[0], p[1]), p[2]) != 1:
            continue
        m0 = 1 if sum(p) % 2 == 0 else 2
        nh = hmax // (m0 * max(abs(v) for v in p))
        if nh:
            g = np.array(p, np.float64) * m0
            out.append((g @ g, tuple(-g), g, nh))
    out.sort(key=lambda v: (v[0], v[1]))
    g = np.array([o[2] for o in out])
    n = np.linalg.norm(g, axis=1)
    w = (g / n[:, None]).astype(np.float32)
    d0 = (LATTICE_A / n).astype(np.float32)
    return w, d0, np.array([o[3] for o in out], np.int32)


def _rotations(n, rng):
    u1, u2, u3 = rng.random((3, n))
    a, b = np.sqrt(1 - u1), np.sqrt(u1)
    w, x, y, z = (a * np.sin(2 * np.pi * u2), a * np.cos(2 * np.pi * u2), b * np.sin(2 * np.pi * u3),
                  b * np.cos(2 * np.pi * u3))
    return np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y), 2 * (x * y + w * z),
                     1 - 2 * (x * x + z * z), 2 * (y * z - w * x), 2 * (x * z - w * y), 2 * (y * z + w * x),
                     1 - 2 * (x * x + y * y)], -1).reshape(n, 3, 3)


def _perturbed(R, x, rng, deg=0.1, mm=0.05):
    k = rng.normal(size=(len(R), 3)) * math.radians(deg) / math.sqrt(3)
    K = np.zeros((len(R), 3, 3))
    K[:, 0, 1], K[:, 0, 2], K[:, 1, 2] = -k[:, 2], k[:, 1], -k[:, 0]
    K = K - K.transpose(0, 2, 1)
    dR = np.eye(3) + K + 0.5 * K @ K
    dR = np.linalg.svd(dR)
    return (dR[0] @ dR[2]) @ R, x + rng.normal(size=x.shape) * mm


def _t64(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=DEV)


def _gamma(omega):
    c, s, o, i = torch.cos(omega), torch.sin(omega), torch.zeros_like(omega), torch.ones_like(omega)
    return torch.stack([c, o, s, o, i, o, -s, o, c], -1).reshape(-1, 3, 3)


def _rays(geom, Gam, R, x, w):
    """Rays and centres of rows (Gamma, R, x, w), any leading shape."""
    u = (Gam @ (R @ w[..., None]))[..., 0]
    c = (Gam @ x[..., None])[..., 0]
    e = torch.tensor(geom.beam, dtype=torch.float64, device=u.device)
    ue = (u * e).sum(-1, keepdim=True)
    return e - 2.0 * ue * u, c, ue[..., 0].abs(), u


def _visible(geom, R, x, omega, w, d0, nh, t_of=None):
    """Visible spots of every grain at every angle (or, with t_of, of grain n
    at the angles t_of[n] only): dict of t, n, m, ray, lam, centre, spot, det,
    sorted by (t, n, m)."""
    out = []
    Gam = _gamma(omega)
    N, M = R.shape[0], w.shape[0]
    ns = torch.arange(N, device=DEV).repeat_interleave(M)
    ms = torch.arange(M, device=DEV).repeat(N)
    for t in range(omega.shape[0]):
        r, c, ue, _ = _rays(geom, Gam[t], R[ns], x[ns], w[ms])
        lam0 = 2.0 * d0[ms] * ue
        lam = torch.zeros_like(lam0)
        for h in range(int(nh.max()), 0, -1):
            ln = lam0 / h
            ok = (h <= nh[ms]) & (ln >= geom.lam_min) & (ln <= geom.lam_max)
            lam = torch.where(ok, ln, lam)
        best = torch.full_like(lam0, 1e30)
        det = torch.full_like(ms, -1)
        spot = torch.zeros_like(r)
        for k, d in enumerate(geom.detectors):
            nrm, a1, a2 = (_t64(v) for v in d.axes())
            ctr = _t64(d.centre)
            tau = ((ctr - c) @ nrm) / (r @ nrm)
            s = c + tau[:, None] * r
            hit = (tau > 0) & (tau < best) & (((s - ctr) @ a1).abs() < d.half) & (((s - ctr) @ a2).abs() < d.half)
            best = torch.where(hit, tau, best)
            det = torch.where(hit, torch.full_like(det, k), det)
            spot = torch.where(hit[:, None], s, spot)
        ok = (lam > 0) & (det >= 0)
        if t_of is not None:
            ok &= t_of[ns, t]
        i = torch.nonzero(ok)[:, 0]
        out.append((torch.full_like(i, t), ns[i], ms[i], r[i], lam[i], c[i], spot[i], det[i]))
    return dict(zip(("t", "n", "m", "ray", "lam", "centre", "spot", "det"), (torch.cat(v) for v in zip(*out))))


def _observe(geom, true, T, total, rng):
    """`total` observed spots sorted by angle: noise in the detector plane,
    spots off the detector dropped, the rest outliers, unevenly over the
    angles.  Returns p (n, 3), I_off and the index of the true spot behind each
    (or -1)."""
    t, det, s = (true[k].cpu().numpy() for k in ("t", "det", "spot"))
    ax = [d.axes() for d in geom.detectors]
    z = rng.standard_normal((len(t), 2)) * SIGMA_MM
    p = np.array(s)
    keep = np.zeros(len(t), bool)
    for k, d in enumerate(geom.detectors):
        i = det == k
        p[i] += z[i, :1] * ax[k][1] + z[i, 1:] * ax[k][2]
        q = p[i] - np.asarray(d.centre)
        keep[i] = (np.abs(q @ ax[k][1]) < d.half) & (np.abs(q @ ax[k][2]) < d.half)
    surplus = int(keep.sum()) - total
    if surplus > 0:
        keep[rng.choice(np.nonzero(keep)[0], surplus, replace=False)] = False
    share = (np.bincount(t, minlength=T) + 1e-9) * rng.uniform(0.5, 2.0, T)
    t_out = np.repeat(np.arange(T), rng.multinomial(max(0, -surplus), share / share.sum()))
    d_out = rng.integers(0, len(geom.detectors), len(t_out))
    uv = rng.uniform(-1.0, 1.0, (len(t_out), 2))
    p_out = np.zeros((len(t_out), 3))
    for k, d in enumerate(geom.detectors):
        i = d_out == k
        p_out[i] = np.asarray(d.centre) + d.half * (uv[i, :1] * ax[k][1] + uv[i, 1:] * ax[k][2])
    P = np.concatenate([p[keep], p_out])
    Tt = np.concatenate([t[keep], t_out])
    src = np.concatenate([np.nonzero(keep)[0], np.full(len(t_out), -1)])
    key = rng.permutation(len(P))
    order = key[np.argsort(Tt[key], kind="stable")]
    off = np.zeros(T + 1, np.int64)
    np.cumsum(np.bincount(Tt, minlength=T), out=off[1:])
    return P[order].astype(np.float32), off.astype(np.int32), src[order]


class _Poly:
    """The inputs of a case: what a user holds, as 32-bit arrays on the GPU."""


def _poly(case, seed):
    rng = np.random.default_rng([seed, 7])
    P = _Poly()
    P.rng = rng
    P.geom = _geometry(case["geometry"])
    w, d0, nh = _planes(case["hmax"])
    P.w, P.d0 = torch.as_tensor(w, device=DEV), torch.as_tensor(d0, device=DEV)
    P.nh = torch.as_tensor(nh, device=DEV)
    T = P.T = case["T"]
    P.omega = torch.as_tensor((np.radians(case["span"]) * np.arange(T) / T).astype(np.float32), device=DEV)
    P.c_out = float(np.float32(4.0 * P.geom.D ** 2 * math.sin(1.5 * SIGMA_MM / P.geom.D) ** 2))
    if case["kind"] == "train":
        return P
    N = case["grains"]
    nI, nJ = (int(v) for v in _counts(case))
    found = 0
    while found < nJ:
        R, x = _rotations(N, rng), rng.uniform(-CUBE_MM / 2, CUBE_MM / 2, (N, 3))
        true = _visible(P.geom, _t64(R), _t64(x), P.omega.double(), P.w.double(), P.d0.double(), P.nh)
        R0, x0 = (a.astype(np.float32) for a in _perturbed(R, x, rng))
        m = _visible(P.geom, _t64(R0), _t64(x0), P.omega.double(), P.w.double(), P.d0.double(), P.nh)
        found = len(m["t"])
    p, off, _ = _observe(P.geom, true, T, nI, rng)
    P.p = torch.zeros(len(p), 4, device=DEV)
    P.p[:, :3] = torch.as_tensor(p, device=DEV)
    P.I_off = torch.as_tensor(off, device=DEV)
    if case["kind"] in ("fit", "propose"):
        return P
    # the prototypes' poses and the frozen list of their spots, less a few (so that every seed has as many)
    P.R, P.x = torch.as_tensor(R0.reshape(-1, 9), device=DEV), torch.as_tensor(x0, device=DEV)
    listed_ = torch.as_tensor(np.sort(rng.choice(found, nJ, replace=False)), device=DEV)
    m = {k: v[listed_] for k, v in m.items()}
    P.t, P.n, P.m, P.det = (m[k].int().contiguous() for k in ("t", "n", "m", "det"))
    P.ray = torch.cat([m["ray"], m["lam"][:, None]], 1).float().contiguous()
    P.centre = torch.nn.functional.pad(m["centre"], (0, 1)).float().contiguous()
    P.spot = torch.cat([m["spot"], m["det"][:, None].double()], 1).float().contiguous()
    J = np.zeros(T + 1, np.int64)
    np.cumsum(np.bincount(P.t.cpu().numpy(), minlength=T), out=J[1:])
    P.J_off = torch.as_tensor(J.astype(np.int32), device=DEV)
    if case["kind"] in ("mstep", "grad"):
        # potentials as an E-step leaves them
        L = _lists(P, P.ray[:, :3].double(), P.centre[:, :3].double(), case["eps"], 260.0)
        f, g, _ = _sinkhorn(P, L, case["eps"], 12, 0)
        P.f, P.g = f.float(), g.float()
    return P


def _library(P):
    """The same inputs as the library's objects."""
    lat = api.Lattice(torch.cat([P.w, P.d0[:, None]], 1).contiguous(), P.nh)
    obs = api.ObsSpots(P.p, P.I_off) if hasattr(P, "p") else None
    model = api.ModelSpots(P.T, int(P.t.numel()), P.J_off, P.n, P.m, P.t, P.ray, P.centre, P.spot) \
        if hasattr(P, "t") else None
    return lat, obs, model


# ------------------------------------------------------------------ passes
def prepare(case, seed):
    P = _poly(case, seed)
    S = dict(case=case, P=P, h=api.Handle(DEV))
    S["lat"], S["obs"], S["model"] = _library(P)
    kind = case["kind"]
    if kind == "em":
        cfg = em_mod.EMConfig(eps_final=case["eps"], n_em=case["n_em"], n_sinkhorn=case["n_iter"], c_out=P.c_out)
        S["solver"] = em_mod.EMSolver(S["h"], P.geom, S["lat"], S["obs"], S["model"], P.omega, cfg)
    elif kind == "grad":
        S["w"] = torch.as_tensor(P.rng.normal(size=(case["grains"], 3)).astype(np.float32) * 1e-3,
                                 device=DEV).requires_grad_()
        S["x"] = P.x.clone().requires_grad_()
    elif kind == "fit":
        S["R0"], S["x0"] = _starts(case, P)
    elif kind == "train":
        S["sets"] = _scene_sets(case, P)
        S["net"] = pr.Network(S["h"], params=_weights(seed))
        S["batch"] = pr.Batch(S["h"], case["scenes"] * case["per_scene"])
        S["axes"] = torch.empty(S["sets"]["p"].shape[0], 4, device=DEV)
    elif kind == "propose":
        S["net"] = pr.Network(S["h"], params=_weights(seed))
        S["seeds"] = _seeds(case, P)
        S["batch"] = pr.Batch(S["h"], case["seeds"])
    return S


def run(S):
    case, P, h = S["case"], S["P"], S["h"]
    kind = case["kind"]
    if kind == "estep":
        kw = dict(kappa=KAPPA, lam=LAMBDA) if case["mode"] == 2 else {}
        out = api.cost_sinkhorn(h, P.geom, S["obs"], S["model"], case["eps"], P.c_out, case["n_iter"],
                                dust_mode=case["mode"], harvest=case["harvest"], col_harvest=case["cols"], **kw)
        if case["mode"] == 2:
            out.pop("dust")  # not written in the unbalanced mode
        out.pop("marg_err", None)  # of a converged solve: the rounding of sums that are 1
        return out
    if kind == "sparse":
        out = api.cost_sinkhorn_sparse(h, P.geom, S["obs"], S["model"], case["eps"], P.c_out, case["n_iter"],
                                       rho=case["rho"], dust_mode=case["mode"])
        out.pop("marg_err")
        return out
    if kind == "mstep":
        R, x = P.R.clone(), P.x.clone()
        norms = torch.empty(case["grains"], 2, device=DEV)
        api.mstep(h, P.geom, S["lat"], S["obs"], S["model"], P.f, P.g, case["eps"], P.omega, R, x, step_norms=norms)
        return dict(R=R, x=x)
    if kind == "grad":
        E = ot_weighted_cost(S["w"], S["x"], P.R, h, P.geom, S["lat"], S["obs"], S["model"], P.f, P.g, case["eps"],
                             P.omega)
        gw, gx = torch.autograd.grad(E.sum(), (S["w"], S["x"]))
        return dict(E=E.detach(), gw=gw, gx=gx)
    if kind == "em":
        R, x = P.R.clone(), P.x.clone()
        out = S["solver"].run(R, x)
        return dict(out, R=R, x=x)
    if kind == "fit":
        R, x, keep, unm = api.single_fit(h, P.geom, S["lat"], S["obs"], P.omega, S["R0"], S["x0"], case["eps"],
                                         case["k_max"], P.c_out, anneal=case["anneal"], recut=True)
        return dict(R=R, x=x, keep=keep, unmatched=unm)
    if kind == "train":
        D, batch, net = S["sets"], S["batch"], S["net"]
        pr.make_sets(h, P.geom, D["p"], D["I_off"], D["omega"], D["seeds"], D["wlo"], D["whi"], batch, S["axes"],
                     label=D["label"], grainR=D["R"], grainX=D["x"])
        pr.train_step(h, net, batch, 1e-4)
        n = batch.n
        return dict(outputs=batch.outputs(), loss=batch.region("loss", torch.float32, (n,)), grads=_grads(net))
    R, x = pr.propose(h, S["net"], P.geom, S["obs"], P.omega, S["seeds"], batch=S["batch"])
    return dict(outputs=S["batch"].outputs(), R=R, x=x)


KAPPA, LAMBDA = 60.0, 40.0  # marginal weights of the unbalanced E-step (mm^2)


def _grads(net):
    """The gradients of the last training step, as the network's buffer holds
    them: after the parameters and the two Adam moments."""
    part = (4 * net.n_params + 255) // 256 * 256
    return net.buf[3 * part:3 * part + 4 * net.n_params].view(torch.float32)


def _starts(case, P):
    S = case["starts"]
    R = _rotations(S, P.rng).astype(np.float32).reshape(S, 9)
    x = P.rng.uniform(-0.5, 0.5, (S, 3)).astype(np.float32)
    return torch.as_tensor(R, device=DEV), torch.as_tensor(x, device=DEV)


def _seeds(case, P):
    n = int(P.p.shape[0])
    return P.rng.choice(n, case["seeds"], replace=n < case["seeds"])


def _weights(seed):
    """Weights in the network's order: He-normal layers, small biases, and an
    output layer whose eight hypotheses lie apart near proper frames, as in a
    network that has learned for a while."""
    rng = np.random.default_rng([seed, 11])
    out = []
    for o, i in ((256, 64), (256, 256), (256, 256), (256, 512), (72, 256)):
        out.append(rng.standard_normal(o * i) * math.sqrt((0.05 if o == 72 else 2.0) / i))
        out.append(rng.standard_normal(o) * 0.05)
    R = _rotations(8, rng)
    out[-1] = np.concatenate([R[:, :, 0], R[:, :, 1], rng.uniform(-1.0, 1.0, (8, 3))], 1).reshape(-1)
    return np.concatenate(out).astype(np.float32)


def _scene_sets(case, P):
    """Single-grain scenes of 10 consecutive angles each, and the seeds and
    windows of their sets."""
    S, per, W, rng = case["scenes"], case["per_scene"], 10, P.rng
    t0 = rng.integers(0, P.T - W + 1, S)
    R, x = _rotations(S, rng), rng.uniform(-CUBE_MM / 2, CUBE_MM / 2, (S, 3))
    in_window = (np.arange(P.T)[None] >= t0[:, None]) & (np.arange(P.T)[None] < t0[:, None] + W)
    true = _visible(P.geom, _t64(R), _t64(x), P.omega.double(), P.w.double(), P.d0.double(), P.nh,
                    t_of=torch.as_tensor(in_window, device=DEV))
    n = true["n"].cpu().numpy()
    true = dict(true, t=true["t"] - torch.as_tensor(t0, device=DEV)[true["n"]] + W * true["n"])
    p, off, src = _observe(P.geom, true, S * W, int(len(n) * (1.0 + case["outliers"])), rng)
    label = np.where(src >= 0, n[np.maximum(src, 0)], -1)
    seeds = np.full(S * per, -1)
    for s in range(S):
        inl = off[s * W] + np.nonzero(label[off[s * W]:off[(s + 1) * W]] >= 0)[0]
        if len(inl):
            seeds[s * per:(s + 1) * per] = rng.choice(inl, per)
    i32 = lambda a: torch.as_tensor(np.asarray(a, np.int32), device=DEV)
    p4 = np.zeros((len(p), 4), np.float32)
    p4[:, :3] = p
    lo = np.repeat(np.arange(S) * W, per)
    om = P.omega[torch.as_tensor((t0[:, None] + np.arange(W)).reshape(-1), device=DEV)].contiguous()
    return dict(p=torch.as_tensor(p4, device=DEV), I_off=i32(off), omega=om, seeds=i32(seeds), wlo=i32(lo),
                whi=i32(lo + W), label=i32(label),
                R=torch.as_tensor(R.reshape(-1, 9).astype(np.float32), device=DEV),
                x=torch.as_tensor(x.astype(np.float32), device=DEV))


# -------------------------------------------------------------------- work
PER_ANGLE = {("flat", 4): 6.25, ("flat", 6): 7.83, ("tilted", 4): 8.96, ("tilted", 6): 10.73}  # spots of a grain


def _counts(case):
    """Observed and model spots of the scan: the model spots a little fewer
    than nearly every draw of the grains shows."""
    mean = PER_ANGLE[case["geometry"], case["hmax"]] * case["grains"] * case["T"]
    return mean * (1.0 + case["outliers"]), mean * (0.99 - 0.2 / math.sqrt(case["grains"]))


def work(case):
    kind = case["kind"]
    if kind in ("train", "propose"):
        sets = case["seeds"] if kind == "propose" else case["scenes"] * case["per_scene"]
        per_spot = 256 * 64 + 2 * 256 * 256
        head = 256 * 512 + 72 * 256
        params = 4 * (per_spot + head + 4 * 256 + 72)
        flops = 2.0 * sets * (128 * per_spot + head) * (3 if kind == "train" else 1)
        return dict(bytes=sets * (128 * 16 + 72 * 4) + params * (5 if kind == "train" else 1), flops=flops)
    nI, nJ = _counts(case)
    pairs = nI * nJ / case["T"]  # same-angle pairs
    # the share of the pairs whose plan entry does not underflow: the disc of K C <= 130 on two detectors of
    # 256 x 256 mm, spots about twice as dense as uniform where they are
    share = min(1.0, 2.0 * math.pi * (130.0 / LOG2E) * case["eps"] / (2 * 256.0 ** 2))
    spots = 16 * nI + 40 * nJ
    if kind == "estep":
        return dict(bytes=spots + 12 * nI + 4 * nJ, flops=2.0 * case["n_iter"] * pairs * share * 14)
    if kind == "sparse":
        return dict(bytes=spots + 12 * nI + 4 * nJ, flops=2.0 * case["n_iter"] * nJ * case["rho"] * 3 + 13 * pairs * share)
    if kind in ("mstep", "grad"):
        return dict(bytes=spots + 4 * (nI + nJ) + 100 * case["grains"], flops=pairs * share * 14 * 2)
    if kind == "em":
        return dict(bytes=spots + 12 * nI, flops=2.0 * case["n_iter"] * case["n_em"] * pairs * min(1.0, 10 * share) * 14)
    # fits: the spots of one grain against every observed spot of their angles, each step
    return dict(bytes=16 * nI + 100 * case["starts"],
                flops=case["starts"] * case["k_max"] * nI * nJ / case["grains"] / case["T"] * 14)


# ------------------------------------------------------- 64-bit references
def _cost_lengths(P):
    D = torch.tensor([d.D if d.D > 0 else P.geom.D for d in P.geom.detectors], dtype=torch.float64, device=DEV)
    return D[P.det.long()]


def _lists(P, ray, centre, eps, cut, limit=None):
    """Same-angle pairs (i, j) with cost C log2(e) / eps <= cut, and their
    scaled costs; None when there are more than `limit`."""
    I, J = P.I_off.cpu().tolist(), P.J_off.cpu().tolist()
    p = P.p[:, :3].double()
    K = _cost_lengths(P) ** 2 * (LOG2E / eps)
    out, n = [], 0
    for t in range(P.T):
        c, r, k = centre[J[t]:J[t + 1]], ray[J[t]:J[t + 1]], K[J[t]:J[t + 1]]
        step = max(1, int(3e7 // max(1, len(c))))
        for a in range(I[t], I[t + 1], step):
            q = p[a:min(a + step, I[t + 1])]
            dx, dy, dz = (q[:, None, b] - c[None, :, b] for b in range(3))
            s = (dx * dx + dy * dy + dz * dz).rsqrt()
            kc = ((dx * s - r[None, :, 0]) ** 2 + (dy * s - r[None, :, 1]) ** 2 + (dz * s - r[None, :, 2]) ** 2) * k
            i, j = torch.nonzero(kc <= cut, as_tuple=True)
            n += len(i)
            if limit and n > limit:
                return None
            out.append((i + a, j + J[t], kc[i, j]))
    i, j, kc = (torch.cat(v) for v in zip(*out))
    return i, j, kc


def _sinkhorn(P, L, eps, n_iter, mode):
    """Potentials (f, g, dust) of the E-step on the listed pairs, in mm^2."""
    i, j, kc = L
    nI, nJ = int(P.p.shape[0]), int(P.t.numel())
    dev = dict(dtype=torch.float64, device=DEV)
    kco = P.c_out * LOG2E / eps
    F, G = torch.zeros(nI, **dev), torch.zeros(nJ, **dev)
    back = eps / LOG2E
    if mode == 2:
        tr, tc = KAPPA / (KAPPA + eps), LAMBDA / (LAMBDA + eps)
        lse = lambda like, at, v, m: m + torch.log2(torch.zeros_like(like).index_add_(0, at, torch.exp2(v - m[at])))
        top = lambda like, at, v: torch.full_like(like, -1e30).scatter_reduce_(0, at, v, "amax")
        for _ in range(n_iter):
            v = G[j] - kc
            F = -tr * lse(F, i, v, top(F, i, v))
            v = F[i] - kc
            G = -tc * lse(G, j, v, top(G, j, v))
        return F * back, G * back, None
    e = torch.exp2(-kc)  # the lists end far above the underflow of 64 bits
    rows = lambda G: torch.zeros(nI, **dev).index_add_(0, i, torch.exp2(G)[j] * e)
    cols = lambda F: torch.zeros(nJ, **dev).index_add_(0, j, torch.exp2(F)[i] * e)
    T = P.T if mode else 1
    cI, cJ = (P.I_off[1:] - P.I_off[:-1]).double(), (P.J_off[1:] - P.J_off[:-1]).double()
    if not mode:
        cI, cJ = cI.sum()[None], cJ.sum()[None]
    U = torch.ceil(0.4 * cJ - 1e-9)
    O = U + cI - cJ
    U, O = torch.where(O < 0, cJ - cI, U), torch.clamp(O, min=0.0)
    ti = torch.repeat_interleave(torch.arange(P.T, device=DEV), (P.I_off[1:] - P.I_off[:-1]).long())
    tj = P.t.long()
    if not mode:
        ti, tj = torch.zeros_like(ti), torch.zeros_like(tj)
    F0, G0 = torch.zeros(T, **dev), torch.zeros(T, **dev)
    total = lambda v, at: torch.zeros(T, **dev).index_add_(0, at, v)
    for _ in range(n_iter):
        F0 = torch.log2(U) - torch.log2(total(torch.exp2(G), tj) + torch.exp2(G0 - kco))
        F = -torch.log2(rows(G) + torch.exp2(G0 - kco)[ti])
        G0 = torch.log2(O) - torch.log2(total(torch.exp2(F - kco), ti) + torch.exp2(F0 - kco))
        G = -torch.log2(cols(F) + torch.exp2(F0)[tj])
    return F * back, G * back, torch.cat([F0, G0]) * back


def _margin(P, L, f, g, dust, eps, mode):
    """Plan read-out of the rows: top1 - top2 over the model spots and the outlier column."""
    i, j, kc = L
    s = LOG2E / eps
    nI = int(P.p.shape[0])
    v = g[j] * s - kc
    b1 = torch.full((nI,), -1e30, dtype=torch.float64, device=DEV).scatter_reduce_(0, i, v, "amax")
    first = v == b1[i]
    b2 = torch.full_like(b1, -1e30).scatter_reduce_(0, i, torch.where(first, -1e30, v), "amax")
    twice = torch.zeros_like(b1).index_add_(0, i, first.double()) > 1.5
    b2 = torch.where(twice, b1, b2)
    if mode != 2:
        nd = P.T if mode else 1
        d = dust[nd:] * s - P.c_out * s
        ti = torch.repeat_interleave(torch.arange(P.T, device=DEV), (P.I_off[1:] - P.I_off[:-1]).long())
        d = d[ti] if mode else d.expand(nI)
        b1, b2 = torch.maximum(b1, d), torch.maximum(b2, torch.minimum(b1, d))
    return torch.exp2(f * s + b1) - torch.exp2(f * s + b2)


def _mstep(P, L, ray, f, g, eps, R, x, n_newton=4, n_mm=4, tol_x=1e-6, tol_R=1e-9, hreg=1e-3):
    """Newton on positions, then majorise-minimise on rotations, per grain."""
    i, j, kc = L
    N = x.shape[0]
    s = LOG2E / eps
    Q = torch.exp2(f[i] * s + g[j] * s - kc)
    keep = Q > 1e-18
    i, j = i[keep], j[keep]
    Q = Q[keep] * (_cost_lengths(P)[j] / P.geom.D) ** 2
    n, m, Gam = P.n.long()[j], P.m.long()[j], _gamma(P.omega.double())[P.t.long()[j]]
    p, r = P.p[i, :3].double(), ray[j]
    eye = torch.eye(3, dtype=torch.float64, device=DEV)
    outer = lambda a, b: a[:, :, None] * b[:, None, :]
    x, R = x.clone(), R.clone()

    def hats(x):
        d = p - (Gam @ x[n][..., None])[..., 0]
        tau = d.norm(dim=1, keepdim=True)
        return d / tau, tau

    going = torch.ones(N, dtype=torch.bool, device=DEV)
    for _ in range(n_newton):
        h, tau = hats(x)
        rr = (h * r).sum(1, keepdim=True)
        gc = -Q[:, None] * (r - rr * h) / tau
        H = (Q[:, None] / tau ** 2)[..., None] * (rr[..., None] * (3 * outer(h, h) - eye) - outer(h, r) - outer(r, h))
        gx = torch.zeros(N, 3, dtype=torch.float64, device=DEV).index_add_(0, n, (Gam.mT @ gc[..., None])[..., 0])
        Hx = torch.zeros(N, 3, 3, dtype=torch.float64, device=DEV).index_add_(0, n, Gam.mT @ H @ Gam)
        fro = Hx.flatten(1).norm(dim=1)
        iota = torch.clamp(torch.linalg.eigvalsh(Hx)[:, 2] + hreg * fro, min=0.0)
        A = Hx - iota[:, None, None] * eye
        ok = going & (fro > 0)
        dx = torch.linalg.solve(torch.where(ok[:, None, None], A, eye), gx[..., None])[..., 0]
        x = torch.where(ok[:, None], x - dx, x)
        going = ok & (dx.norm(dim=1) >= tol_x)
    h, _ = hats(x)
    e = torch.tensor(P.geom.beam, dtype=torch.float64, device=DEV).expand_as(h)
    v = Q[:, None] * h
    M = P.w.shape[0]
    M0 = torch.zeros(N * M, 3, 3, dtype=torch.float64, device=DEV).index_add_(
        0, n * M + m, -(Gam.mT @ (outer(v, e) + outer(e, v)) @ Gam))
    at = torch.unique(n * M + m)
    M0 = M0[at]
    M0 = M0 + torch.clamp(-torch.linalg.eigvalsh(M0)[:, 0], min=0.0)[:, None, None] * eye
    ng, wm = at // M, P.w.double()[at % M]
    going = torch.ones(N, dtype=torch.bool, device=DEV)
    for _ in range(n_mm):
        a = (M0 @ (R[ng] @ wm[..., None]))[..., 0]
        B = torch.zeros(N, 3, 3, dtype=torch.float64, device=DEV).index_add_(0, ng, outer(a, wm))
        U, _, Vh = torch.linalg.svd(B)
        fix = torch.ones(N, 3, dtype=torch.float64, device=DEV)
        fix[:, 2] = torch.det(U @ Vh)
        Rn = U @ (fix[..., None] * Vh)
        ok = going & (B.flatten(1).norm(dim=1) > 0)
        dR = (Rn - R).flatten(1).norm(dim=1)
        R = torch.where(ok[:, None, None], Rn, R)
        going = ok & (dR >= tol_R)
    return R, x


def _schedule(eps, n_em, k, factor=100.0):
    K = math.ceil(0.75 * n_em)
    return eps if k >= K else eps * factor ** (1.0 - k / K)


def _read_out(P, L, f, g, dust, eps, mode, out):
    out.update(assign=None, margin=_margin(P, L, f, g, dust, eps, mode))
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "fit":
        return None  # tens of seconds: every observed spot against every start's spots, 40 steps
    P = _poly(case, seed)
    if kind in ("train", "propose"):
        return _network_exact(case, P, seed)
    eps = case["eps"]
    ray, cen = P.ray[:, :3].double(), P.centre[:, :3].double()
    cut = 1e30 if case.get("mode") == 2 else 260.0
    if kind == "estep":
        L = _lists(P, ray, cen, eps, cut, limit=2.5e8)
        if L is None or len(L[0]) * case["n_iter"] > 2e10:
            return None  # over 20 seconds
        f, g, dust = _sinkhorn(P, L, eps, case["n_iter"], case["mode"])
        s = LOG2E / eps
        out = dict(f=f, g=g)
        if case["mode"] != 2:
            out["dust"] = dust
        if case["harvest"]:
            out = _read_out(P, L, f, g, dust, eps, case["mode"], out)
        if case["cols"]:
            out["q"] = torch.zeros_like(g).index_add_(0, L[1], torch.exp2(f[L[0]] * s + g[L[1]] * s - L[2]))
        return out
    if kind == "sparse":
        I, J = P.I_off.cpu().tolist(), P.J_off.cpu().tolist()
        L = _nearest(P, ray, cen, eps, case["rho"], I, J)
        f, g, dust = _sinkhorn(P, L, eps, case["n_iter"], case["mode"])
        return _read_out(P, L, f, g, dust, eps, case["mode"], dict(f=f, g=g, dust=dust))
    R, x = P.R.double().reshape(-1, 3, 3), P.x.double()
    if kind == "mstep":
        L = _lists(P, ray, cen, eps, 260.0)
        R, x = _mstep(P, L, ray, P.f.double(), P.g.double(), eps, R, x)
        return dict(R=R.reshape(-1, 9), x=x)
    n, Gam, w = P.n.long(), _gamma(P.omega.double())[P.t.long()], P.w.double()[P.m.long()]
    if kind == "em":
        for k in range(case["n_em"] + 1):
            e = _schedule(eps, case["n_em"], k)
            ray, cen, _, _ = _rays(P.geom, Gam, R[n], x[n], w)
            L = _lists(P, ray, cen, e, 260.0)
            f, g, dust = _sinkhorn(P, L, e, case["n_iter"], 0)
            if k < case["n_em"]:
                R, x = _mstep(P, L, ray, f, g, e, R, x)
        out = _read_out(P, L, f, g, dust, eps, 0, dict(f=f, g=g, dust=dust))
        return dict(out, R=R.reshape(-1, 9), x=x)
    # the gradient of the OT-weighted cost, the plan held
    wv = torch.as_tensor(P.rng.normal(size=(case["grains"], 3)).astype(np.float32) * 1e-3, device=DEV).double()
    wv.requires_grad_()
    x = x.clone().requires_grad_()
    z = torch.zeros_like(wv[:, 0])
    K = torch.stack([z, -wv[:, 2], wv[:, 1], wv[:, 2], z, -wv[:, 0], -wv[:, 1], wv[:, 0], z], 1).reshape(-1, 3, 3)
    ray, cen, _, _ = _rays(P.geom, Gam, (torch.linalg.matrix_exp(K) @ R)[n], x[n], w)
    with torch.no_grad():
        i, j, kc = _lists(P, ray.detach(), cen.detach(), eps, 260.0)
        Q = torch.exp2(P.f.double()[i] * (LOG2E / eps) + P.g.double()[j] * (LOG2E / eps) - kc)
        keep = Q > 1e-18
        i, j, Q = i[keep], j[keep], Q[keep]
    d = P.p[i, :3].double() - cen[j]
    C = ((d / d.norm(dim=1, keepdim=True) - ray[j]) ** 2).sum(1) * _cost_lengths(P)[j] ** 2
    E = torch.zeros_like(z).index_add(0, n[j], Q * C)
    gw, gx = torch.autograd.grad(E.sum(), (wv, x))
    return dict(E=E.detach(), gw=gw, gx=gx)


def _nearest(P, ray, centre, eps, rho, I, J):
    p = P.p[:, :3].double()
    K = _cost_lengths(P) ** 2 * (LOG2E / eps)
    out = []
    for t in range(P.T):
        q = p[I[t]:I[t + 1]]
        for a in range(J[t], J[t + 1], 1024):
            b = min(a + 1024, J[t + 1])
            d = [q[None, :, k] - centre[a:b, None, k] for k in range(3)]
            s = (d[0] * d[0] + d[1] * d[1] + d[2] * d[2]).rsqrt()
            kc = sum((d[k] * s - ray[a:b, None, k]) ** 2 for k in range(3)) * K[a:b, None]
            v, i = torch.topk(kc, min(rho, len(q)), dim=1, largest=False)
            out.append(((i + I[t]).flatten(), torch.arange(a, b, device=DEV).repeat_interleave(v.shape[1]),
                        v.flatten()))
    return tuple(torch.cat(v) for v in zip(*out))


# ----- the set encoder in 64 bits
def _sets_exact(P, p, I_off, omega, seeds, lo, hi):
    """Features (B, 128, 64), valid flags and seed frames of the sets."""
    p = p[:, :3].double()
    off = I_off.long()
    t = torch.repeat_interleave(torch.arange(len(off) - 1, device=DEV), off[1:] - off[:-1])
    om = omega.double()
    e = torch.tensor(P.geom.beam, dtype=torch.float64, device=DEV)
    u = p / p.norm(dim=1, keepdim=True) - e
    u = u / u.norm(dim=1, keepdim=True)
    ax = (_gamma(om)[t].mT @ u[..., None])[..., 0]
    B = len(seeds)
    X = torch.zeros(B, 128, 64, dtype=torch.float64, device=DEV)
    live = seeds >= 0
    s0 = seeds.clamp(min=0)
    n0 = ax[s0]
    y = torch.tensor([0.0, 1.0, 0.0], dtype=torch.float64, device=DEV)
    a1 = y - n0[:, 1:2] * n0
    a1 = a1 / a1.norm(dim=1, keepdim=True)
    F = torch.stack([n0, a1, torch.linalg.cross(n0, a1)], -1)
    first, last = off[lo], off[hi]
    width = int((last - first).max())
    for a in range(0, B, 256):
        b = min(a + 256, B)
        k = first[a:b, None] + torch.arange(width, device=DEV)
        ok = (k < last[a:b, None]) & (k != s0[a:b, None])
        k = k.clamp(max=len(p) - 1)
        d = 1.0 - (ax[k] @ n0[a:b, :, None])[..., 0].abs()
        d = torch.where(ok, d, 9.0)
        v, at = torch.topk(d, min(127, width), dim=1, largest=False, sorted=True)
        sel = torch.cat([s0[a:b, None], torch.gather(k, 1, at)], 1)
        good = torch.cat([torch.ones_like(v[:, :1]), (v < 8.0).double()], 1) * live[a:b, None]
        q, m = p[sel], sel.shape[1]
        dot = (ax[sel] @ n0[a:b, :, None])[..., 0]
        x = torch.zeros(b - a, m, 64, dtype=torch.float64, device=DEV)
        x[..., 0:3] = (ax[sel] @ F[a:b]) * torch.where(dot < 0, -1.0, 1.0)[..., None]
        dw = om[t[sel]] - om[t[s0[a:b]]][:, None]
        x[..., 3], x[..., 4] = torch.sin(dw), torch.cos(dw)
        x[..., 5], x[..., 6], x[..., 7] = q[..., 2] / 200.0, q[..., 0] / 128.0, q[..., 1] / 128.0
        x[..., 8], x[..., 9], x[..., 10] = q[:, :1, 0] / 128.0, q[:, :1, 1] / 128.0, q[:, :1, 2] / 200.0
        x[:, 0, 11] = 1.0
        x[..., 12] = 1.0
        x[..., 13] = (t[sel] - t[s0[a:b]][:, None]).double() / 10.0
        X[a:b, :m] = x * good[..., None]
    return X, X[..., 12] > 0.5, F


def _encoder(W, X, valid):
    w = [v for v in W]
    Hs = X
    for k in range(3):
        Hs = torch.relu(Hs @ w[2 * k].T + w[2 * k + 1])
    nv = valid.sum(1)
    mean = (Hs * valid[..., None]).sum(1) / nv.clamp(min=1)[:, None]
    mx = torch.where(valid[..., None], Hs, -1.0).amax(1)
    pool = torch.cat([mean, torch.where(nv[:, None] > 0, mx, torch.zeros_like(mx))], 1)
    return torch.relu(pool @ w[6].T + w[7]) @ w[8].T + w[9]


def _unit(v):
    return v / v.norm(dim=-1, keepdim=True)


def _gram_schmidt(o):
    e1 = _unit(o[..., 0:3])
    b = o[..., 3:6]
    e2 = _unit(b - (e1 * b).sum(-1, keepdim=True) * e1)
    return torch.stack([e1, e2, torch.linalg.cross(e1, e2)], -1)


def _network_exact(case, P, seed):
    vec, W, o = torch.as_tensor(_weights(seed), device=DEV).double().requires_grad_(), [], 0
    for rows, cols in ((256, 64), (256, 256), (256, 256), (256, 512), (72, 256)):
        W.append(vec[o:o + rows * cols].reshape(rows, cols))
        W.append(vec[o + rows * cols:o + rows * cols + rows])
        o += rows * (cols + 1)
    if case["kind"] == "propose":
        seeds = _seeds(case, P)
        off = P.I_off.cpu().numpy().astype(np.int64)
        t = np.searchsorted(off, seeds, side="right") - 1
        lo = np.clip(t - 4, 0, P.T)
        hi = np.clip(lo + 10, 0, P.T)
        lo = np.clip(hi - 10, 0, P.T)
        i64 = lambda a: torch.as_tensor(a, device=DEV)
        with torch.no_grad():
            X, valid, F = _sets_exact(P, P.p, P.I_off, P.omega, i64(seeds), i64(lo), i64(hi))
            O = torch.cat([_encoder(W, X[a:a + 256], valid[a:a + 256]) for a in range(0, len(X), 256)])
            Oh = O.reshape(-1, 8, 9)
            R = F[:, None] @ _gram_schmidt(Oh)
        return dict(outputs=O, R=R.reshape(-1, 9), x=(2.5 * Oh[..., 6:9]).reshape(-1, 3))
    D = _scene_sets(case, P)
    seeds = D["seeds"].long()
    X, valid, F = _sets_exact(P, D["p"], D["I_off"], D["omega"], seeds, D["wlo"].long(), D["whi"].long())
    lab = D["label"].long()[seeds.clamp(min=0)].clamp(min=0)
    Rloc = F.mT @ D["R"].double().reshape(-1, 3, 3)[lab]
    xt = D["x"].double()[lab] / 2.5
    sym = []
    for perm in itertools.permutations(range(3)):
        for sgn in itertools.product([1, -1], repeat=3):
            Sm = np.zeros((3, 3))
            for a, b in enumerate(perm):
                Sm[a, b] = sgn[a]
            if np.linalg.det(Sm) > 0:
                sym.append(Sm)
    RS = Rloc[:, None] @ _t64(np.array(sym))
    ok = (seeds >= 0).double()
    O, per_set = [], []
    for a in range(0, len(X), 256):
        o_ = _encoder(W, X[a:a + 256], valid[a:a + 256])
        Oh = o_.reshape(-1, 8, 9)
        tr = torch.einsum("bhij,bsij->bhs", _gram_schmidt(Oh), RS[a:a + 256]).amax(-1)
        Lh = 6.0 - 2.0 * tr + 0.1 * ((Oh[..., 6:9] - xt[a:a + 256, None]) ** 2).sum(-1)
        ls = (Lh.amin(1) + 0.05 * Lh.mean(1)) * ok[a:a + 256]
        (ls.sum() / max(1.0, float(ok.sum()))).backward(retain_graph=True)
        O.append(o_.detach())
        per_set.append(ls.detach())
    return dict(outputs=torch.cat(O), loss=torch.cat(per_set), grads=vec.grad)
