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
