"""Which form the pair passes take, and that the forms agree where the choice
changes: the counters tell listed from swept pairs (a listed entry counts with
its padding, a swept pair once), the results are equal bit for bit."""
import ctypes

import numpy as np
import pytest

import synthgen as sg
from _cases import GEOM
from test_gpu_lists import _blocks, _smallest_workspace, env  # noqa: F401

pytestmark = pytest.mark.gpu


def _lists(env, data):
    api, dev = env["api"], env["dev"]
    p, I_off, m, J_off = data
    ob = api.ObsSpots.from_numpy(p, I_off, device=dev)
    ms = api.ModelSpots.from_numpy(J_off, m["grain"], m["plane"], m["ray"], m["center"], m["spot"], m["det"], device=dev)
    return ob, ms


def _forms(env, call):
    """(outputs, pass pairs, M-step pairs) of call(h) with room for lists and
    with the smallest workspace, which has none."""
    api, torch, dev = env["api"], env["torch"], env["dev"]
    h = api.Handle(dev)

    def counted():
        out = call(h)
        torch.cuda.synchronize()
        h.counters()
        out = call(h)
        torch.cuda.synchronize()
        c = h.counters()
        return out, c["pass_pairs"], c["mstep_pairs"]

    roomy = counted()
    size = h.ws.numel()
    h.reserve = lambda *a, **k: None
    keep = _smallest_workspace(h, torch, lambda: call(h), size)
    tight = counted()
    del keep
    for a, b in zip(roomy[0], tight[0]):
        assert torch.equal(a, b)
    return roomy[1:], tight[1:]


@pytest.mark.parametrize("eps,n_iter,listed", [(1.0, 50, True), (30.0, 3, False), (300.0, 50, False)])
def test_lists_are_made_where_they_pay(env, eps, n_iter, listed):
    sizes = [(1500, 1200), (1400, 1300)]
    ob, ms = _lists(env, _blocks(sizes, 31, GEOM))

    def call(h):
        out = env["api"].cost_sinkhorn(h, GEOM, ob, ms, eps, 2.25, n_iter, harvest=True, col_harvest=True)
        return [out[k] for k in ("f", "g", "dust", "assign", "margin", "q")]

    (n_roomy, _), (n_tight, _) = _forms(env, call)
    # (a slice of spots with few others near them may be listed for any number of iterations)
    assert n_roomy < 0.5 * n_tight if listed else n_roomy > 0.75 * n_tight, n_roomy / n_tight


def test_lists_of_more_than_32_chunks(env):
    """Long lists: the lane's chunk numbers (8 entries a spot each) are read
    again behind the first 32."""
    eps, n_iter = 24.0, 200
    data = p, _, m, _ = _blocks([(6000, 6000)], 32, GEOM)
    ob, ms = _lists(env, data)

    def call(h):
        out = env["api"].cost_sinkhorn(h, GEOM, ob, ms, eps, 2.25, n_iter, harvest=True)
        return [out[k] for k in ("f", "g", "dust", "assign", "margin")]

    (n_roomy, _), (n_tight, _) = _forms(env, call)
    assert n_roomy < 0.8 * n_tight, n_roomy / n_tight  # many slices are listed
    # entries of a spot (K e2 <= 127): more than 32 chunks of most
    entries = []
    for c, r in zip(m["center"][::20], m["ray"][::20, :3]):
        d = p - c
        e = d / np.linalg.norm(d, axis=1, keepdims=True) - r
        entries.append(np.sum(GEOM.D ** 2 * np.log2(np.e) / eps * np.sum(e * e, axis=1) <= 127.0))
    assert np.median(entries) > 8 * 32


@pytest.mark.parametrize("eps,listed", [(1.0, True), (100.0, False)])
def test_plan_lists_of_a_single_pass(env, eps, listed):
    api, torch, dev = env["api"], env["torch"], env["dev"]
    sizes = [(1500, 1200), (1400, 1300)]
    ob, ms = _lists(env, _blocks(sizes, 33, GEOM))
    cfg = sg.CONFIGS["medium"]
    lat = api.Lattice.cubic(cfg.a, cfg.hmax, cfg.centering, device=dev)
    n = int(ms.grain.max()) + 1
    om = torch.tensor([0.1, 0.4], device=dev)
    R = torch.eye(3, device=dev).reshape(1, 9).repeat(n, 1).contiguous()
    x = torch.zeros(n, 3, device=dev)
    e = api.cost_sinkhorn(api.Handle(dev), GEOM, ob, ms, eps, 2.25, 30, harvest=False)

    def call(h):
        return api.objective_grad(h, GEOM, lat, ob, ms, e["f"], e["g"], eps, om, R, x)

    (_, n_roomy), (_, n_tight) = _forms(env, call)
    assert n_roomy != n_tight if listed else n_roomy == n_tight


@pytest.mark.parametrize("kind", ["plain", "adjoint"])
@pytest.mark.parametrize("mode,shapes,n_iter", [(0, (3, 3), 30), (1, (0, 3), 30), (0, (3, 0), 1), (1, (1, 1), 0)])
def test_mstep_keeps_the_order_of_its_estep(env, kind, mode, shapes, n_iter):
    """An M-step inside laue_em takes the order, tiles and cones of the E-step
    before it; one that is called by itself makes them anew.  Poses and
    potentials are equal bit for bit."""
    from _cases import make_case, to_device
    api, torch, dev = env["api"], env["torch"], env["dev"]
    case = make_case(sg.CONFIGS["medium"], seed=34, n_grains=33, T=7)
    ob, ms = to_device(case, dev)
    lat = api.Lattice.cubic(case.cfg.a, case.cfg.hmax, case.cfg.centering, device=dev)
    om = torch.tensor(case.om, dtype=torch.float32, device=dev)
    n_em, k, eps_final, steps = 6, 4, 1.0, 3
    pose = lambda: (torch.tensor(case.R.reshape(-1, 9), dtype=torch.float32, device=dev) + 0.0,
                    torch.tensor(case.x + 0.02, dtype=torch.float32, device=dev))
    R, x = pose()
    h = api.Handle(dev)
    h.reserve(7, n_obs=int(ob.p.shape[0]), n_model=ms.n, n_grains=33, n_planes=int(lat.w_d0.shape[0]))
    h.set_launch_shape(*shapes)
    kept = api.em(h, GEOM, lat, ob, ms, om, R, x, eps_final, n_em, n_iter, case.c_out, k_first=k, k_last=k,
                  dust_mode=mode, mstep=kind, n_newton=steps)
    Ra, xa = pose()
    ha = api.Handle(dev)
    ha.set_launch_shape(*shapes)
    eps = float(np.float32(api.anneal_eps(eps_final, n_em, k, 100.0)))
    api.refresh(ha, GEOM, lat, Ra, xa, om, ms)
    anew = api.cost_sinkhorn(ha, GEOM, ob, ms, eps, case.c_out, n_iter, dust_mode=mode)
    if kind == "plain":
        api.mstep(ha, GEOM, lat, ob, ms, anew["f"], anew["g"], eps, om, Ra, xa, n_newton=steps)
    else:
        api.mstep_adjoint(ha, GEOM, lat, ob, ms, anew["f"], anew["g"], eps, om, Ra, xa, n_steps=steps, lam=1e-3)
    torch.cuda.synchronize()
    for name in ("f", "g", "dust", "assign", "margin"):
        assert torch.equal(kept[name][:len(anew[name])], anew[name]), name
    assert torch.equal(R, Ra) and torch.equal(x, xa)
    assert not torch.equal(x, pose()[1])


@pytest.mark.parametrize("rho", [4, 33])
def test_sparse_search_follows_the_workspace(env, rho):
    """The sparse E-step in exactly the size that has room for the order (the
    search over the cones) and in exactly its own needs (over every pair)."""
    api, torch, dev = env["api"], env["torch"], env["dev"]
    data = _blocks([(300, 170), (1, 40), (0, 9), (40, 0), (513, 64)], 35, GEOM)
    ob, ms = _lists(env, data)
    h = api.Handle(dev)
    L, size, least = h.L, ctypes.c_size_t(), ctypes.c_size_t()
    dims = (5, int(ob.p.shape[0]), ms.n, rho)
    assert L.laue_sparse_workspace_size(*dims, ctypes.byref(size)) == 0
    assert L.laue_sparse_workspace_min_size(*dims, ctypes.byref(least)) == 0
    assert least.value < size.value
    h.ws = torch.empty(size.value, dtype=torch.uint8, device=dev)
    out = []
    for n in (size.value, least.value):
        assert L.laue_set_workspace(h.h, ctypes.c_void_p(h.ws.data_ptr()), n, None) == 0
        out.append(api.cost_sinkhorn_sparse(h, GEOM, ob, ms, 2.0, 2.25, 15, rho=rho, dust_mode=1, col_harvest=True,
                                            neighbours=True))
        torch.cuda.synchronize()
    for k in out[0]:
        assert torch.equal(out[0][k].nan_to_num(9e9), out[1][k].nan_to_num(9e9)), k
    assert L.laue_set_workspace(h.h, ctypes.c_void_p(h.ws.data_ptr()), least.value // 256 * 256 - 256, None) == 0
    with pytest.raises(api.LaueError):
        api.cost_sinkhorn_sparse(h, GEOM, ob, ms, 2.0, 2.25, 15, rho=rho, dust_mode=1)
