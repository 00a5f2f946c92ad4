"""The forms of the pair passes against each other: listed slices, slices left
to the sweep for want of scratch, and every pair evaluated.

All three add the same nonzero terms in the same order, so potentials,
dustbins and read-outs are equal bit for bit; the parity with the oracle is
checked elsewhere on the default form."""
import ctypes

import numpy as np
import pytest

import synthgen as sg
from _cases import GEOM, make_case, to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_2404_06478_gb300 import api, build
    build.build()
    torch.cuda.set_device(0)
    return dict(torch=torch, api=api, dev=torch.device("cuda", 0))


def _blocks(sizes, seed, geom):
    """Observed and model spots of len(sizes) angle blocks, the first m model
    spots and about half as many noisy copies and half random ones observed."""
    rng = np.random.default_rng(seed)
    case = make_case(sg.CONFIGS["medium"], seed=seed, n_grains=60, T=4, geom=geom)
    pool = case.fw
    n = len(pool["t"])
    ob, mod = [], []
    for ni, nj in sizes:
        j = rng.choice(n, nj, replace=nj > n)
        s = pool["spot"][rng.choice(n, ni)] + rng.normal(size=(ni, 3)) * np.array([1.0, 1.0, 0.0])
        far = rng.random(ni) < 0.3
        s[far, :2] = rng.uniform(-128, 128, (int(far.sum()), 2))
        ob.append(s)
        mod.append(j)
    j = np.concatenate(mod)
    I_off = np.r_[0, np.cumsum([a for a, _ in sizes])]
    J_off = np.r_[0, np.cumsum([b for _, b in sizes])]
    return np.concatenate(ob), I_off, {k: pool[k][j] for k in ("grain", "plane", "ray", "center", "spot", "det")}, J_off


def _smallest_workspace(h, torch, call, most):
    """The fewest workspace bytes (to 4 KB) with which call() is accepted."""
    from paper_2404_06478_gb300 import _native as N
    from paper_2404_06478_gb300.api import LaueError
    ws = torch.empty(most, dtype=torch.uint8, device="cuda")

    def accepted(nbytes):
        assert h.L.laue_set_workspace(h.h, ctypes.c_void_p(ws.data_ptr()), nbytes, None) == 0
        try:
            call()
            return True
        except LaueError as e:
            assert e.code == N.LAUE_ERR_WORKSPACE
            return False

    lo, hi = 4096, most
    while hi - lo > 4096:
        mid = (lo + hi) // 2 // 256 * 256
        lo, hi = (lo, mid) if accepted(mid) else (mid, hi)
    assert accepted(hi)
    return ws


# blocks at the edges of slices (64 spots), sub-granules (16) and tiles (128); empty blocks; a block beyond the
# lists' 16-bit slots
EDGES = [(1, 1), (0, 5), (5, 0), (63, 64), (64, 63), (65, 129), (127, 15), (128, 16), (129, 17), (700, 311), (1, 700),
         (900, 1)]


@pytest.mark.parametrize("geom", [GEOM, sg.tilted_geometry()], ids=["flat", "tilted"])
@pytest.mark.parametrize("eps,mode,sizes", [(1.0, 0, EDGES), (6.0, 1, EDGES), (300.0, 0, EDGES), (2.0, 2, EDGES),
                                            (1.0, 0, [(70001, 33), (40, 20)]), (1.0, 1, [(33, 70001), (40, 20)])])
def test_lists_sweeps_and_every_pair_agree(env, geom, eps, mode, sizes):
    api, torch, dev = env["api"], env["torch"], env["dev"]
    p, I_off, m, J_off = _blocks(sizes, 21, geom)
    ob = api.ObsSpots.from_numpy(p, I_off, device=dev)
    ms = api.ModelSpots.from_numpy(J_off, m["grain"], m["plane"], m["ray"], m["center"], m["spot"], m["det"], device=dev)
    h = api.Handle(dev)

    def call():
        out = api.cost_sinkhorn(h, geom, ob, ms, eps, 2.25, 25, dust_mode=mode, harvest=True, col_harvest=True,
                                kappa=30.0, lam=20.0)
        torch.cuda.synchronize()
        h.device_status()  # an isolated spot of the unbalanced mode may be reported; the bits are compared below
        return out

    listed = call()
    h.set_pair_skipping(False)
    every = call()
    h.set_pair_skipping(True)
    size = h.ws.numel()
    h.reserve = lambda *a, **k: None
    keep = _smallest_workspace(h, torch, call, size)
    swept = call()
    for k in listed:
        assert torch.equal(listed[k].nan_to_num(9e9), every[k].nan_to_num(9e9)), ("every pair", k)
        assert torch.equal(listed[k].nan_to_num(9e9), swept[k].nan_to_num(9e9)), ("swept", k)
    del keep


@pytest.mark.parametrize("eps,sizes", [(2.0, EDGES), (8.0, EDGES), (2.0, [(9, 31), (33, 7), (8, 8), (260, 257)])])
def test_split_exact_sums_agree(env, eps, sizes):
    """The unbalanced update, few slices (several warps share a slice's exact
    sums) against the same blocks many times over (one warp each); blocks are
    independent without dustbins.  A sum merged from four parts has at most
    twelve roundings of 2^-22 more, so a potential at most 6e-6 (base 2) more
    error per update, and the rounding of an exponent at most 4 ulp of the
    largest potential; an iteration contracts by tau_row tau_col."""
    api, torch, dev = env["api"], env["torch"], env["dev"]
    p, I_off, m, J_off = _blocks(sizes, 23, GEOM)
    kappa, lam, copies = 30.0, 20.0, 120

    def solve(k):
        h = api.Handle(dev)
        off = lambda o: np.concatenate([[0]] + [o[1:] + c * o[-1] for c in range(k)])
        tile = lambda v: np.concatenate([v] * k)
        ob = api.ObsSpots.from_numpy(tile(p), off(I_off), device=dev)
        ms = api.ModelSpots.from_numpy(off(J_off), *(tile(m[n]) for n in ("grain", "plane", "ray", "center", "spot", "det")),
                                       device=dev)
        out = api.cost_sinkhorn(h, GEOM, ob, ms, eps, 2.25, 25, dust_mode=2, harvest=False, kappa=kappa, lam=lam)
        torch.cuda.synchronize()
        c = h.counters()
        return [out[n].double().cpu().numpy() for n in ("f", "g")], c

    one, c_one = solve(1)
    many, c_many = solve(copies)
    assert c_one["exact_rows"] > 0 and c_one["exact_cols"] > 0
    top = max(np.abs(v).max() for v in one) / (eps * np.log(2.0))
    assert top < 1e6
    tau = kappa / (kappa + eps) * lam / (lam + eps)
    tol = 2 * (6e-6 + 4 * 2.0 ** -23 * top) / (1.0 - tau) * eps * np.log(2.0)
    for a, b in zip(one, many):
        assert np.abs(np.tile(a, copies) - b).max() <= tol


@pytest.mark.parametrize("rho", [1, 8, 64])
@pytest.mark.parametrize("sizes", [EDGES, [(5000, 40), (3, 900), (64, 64)]], ids=["edges", "uneven"])
def test_sparse_neighbour_searches_agree(env, rho, sizes):
    """The neighbour search over the cones against the one over every pair
    (which a workspace without room for the order takes): lists, potentials
    and read-out equal bit for bit."""
    api, torch, dev = env["api"], env["torch"], env["dev"]
    p, I_off, m, J_off = _blocks(sizes, 22, GEOM)
    ob = api.ObsSpots.from_numpy(p, I_off, device=dev)
    ms = api.ModelSpots.from_numpy(J_off, m["grain"], m["plane"], m["ray"], m["center"], m["spot"], m["det"], device=dev)
    h = api.Handle(dev)

    def call():
        out = api.cost_sinkhorn_sparse(h, GEOM, ob, ms, 2.0, 2.25, 15, rho=rho, dust_mode=1, col_harvest=True,
                                       neighbours=True)
        torch.cuda.synchronize()
        return out

    cones = call()
    size = h.ws.numel()
    h.reserve_bytes = lambda *a, **k: None
    keep = _smallest_workspace(h, torch, call, size)
    pairs = call()
    for k in cones:
        assert torch.equal(cones[k].nan_to_num(9e9), pairs[k].nan_to_num(9e9)), k
    del keep
