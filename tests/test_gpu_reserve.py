"""A device without room for the whole workspace (the lists of the passes, the
order of the sparse search): the calls run in their own needs, with the same
results, and the size that could not be had is not asked for again."""
import pytest

import synthgen as sg
from _cases import GEOM, make_case, to_device
from test_gpu_lists import env  # noqa: F401

pytestmark = pytest.mark.gpu


def test_calls_run_in_what_the_device_can_give(env, monkeypatch):
    api, torch, dev = env["api"], env["torch"], env["dev"]
    case = make_case(sg.CONFIGS["medium"], seed=61, n_grains=40, T=6)
    ob, ms = to_device(case, dev)
    cfg = case.cfg
    lat = api.Lattice.cubic(cfg.a, cfg.hmax, cfg.centering, device=dev)
    om = torch.tensor(case.om, dtype=torch.float32, device=dev)
    R0 = torch.tensor(case.R.reshape(-1, 9), dtype=torch.float32, device=dev)
    x0 = torch.tensor(case.x, dtype=torch.float32, device=dev)

    def calls():
        h = api.Handle(dev)
        out = []
        e = api.cost_sinkhorn(h, GEOM, ob, ms, 2.0, case.c_out, 30)
        out += [e[k] for k in ("f", "g", "dust", "assign", "margin")]
        R, x = R0.clone(), x0.clone()
        api.mstep(h, GEOM, lat, ob, ms, e["f"], e["g"], 2.0, om, R, x)
        out += [R, x, *api.objective_grad(h, GEOM, lat, ob, ms, e["f"], e["g"], 2.0, om, R0, x0)]
        for _ in range(2):
            s = api.cost_sinkhorn_sparse(h, GEOM, ob, ms, 2.0, case.c_out, 20, rho=16)
            out += [s[k] for k in ("f", "g", "assign")]
        torch.cuda.synchronize()
        return out

    want = calls()
    empty, denied = torch.empty, []
    probe = api.Handle(dev)
    nI, nJ = int(ob.p.shape[0]), ms.n
    full = probe.workspace_size(6, n_obs=nI, n_model=nJ)
    d, least = api.N.LaueProblemDims(6, nI, nJ, 0, 0, 0, 0), api.ctypes.c_size_t()
    assert probe.L.laue_workspace_min_size(probe.h, api.ctypes.byref(d), api.ctypes.byref(least)) == 0
    assert least.value < full

    def limited(*size, **kw):
        if kw.get("dtype") is torch.uint8 and size[0] > most:
            denied.append(size[0])
            raise torch.cuda.OutOfMemoryError("out of memory (test)")
        return empty(*size, **kw)

    s_least, s_full = api.ctypes.c_size_t(), api.ctypes.c_size_t()
    probe.L.laue_sparse_workspace_min_size(6, nI, nJ, 16, api.ctypes.byref(s_least))
    probe.L.laue_sparse_workspace_size(6, nI, nJ, 16, api.ctypes.byref(s_full))
    most = max(probe.workspace_size(6, n_obs=nI, n_model=nJ, n_grains=40, n_planes=int(lat.w_d0.shape[0]))
               - (full - least.value), s_least.value) + 256
    assert most < min(full, s_full.value)
    monkeypatch.setattr(torch, "empty", limited)
    got = calls()
    monkeypatch.undo()
    assert len(denied) == len(set(denied)) and denied
    for a, b in zip(want, got):
        assert torch.equal(a, b)
    # and where not even the calls' own needs can be had, the error is the allocator's
    most = 4096
    monkeypatch.setattr(torch, "empty", limited)
    with pytest.raises(torch.cuda.OutOfMemoryError):
        api.cost_sinkhorn(api.Handle(dev), GEOM, ob, ms, 2.0, case.c_out, 30)


@pytest.mark.parametrize("T,n_obs,n_model", [(90, 1200000, 700000), (1000000, 2000000, 2000000), (1, 10, 10)])
def test_room_for_lists_is_bounded(env, T, n_obs, n_model):
    api = env["api"]
    h = api.Handle(env["dev"])
    d, b = api.N.LaueProblemDims(T, n_obs, n_model, 0, 0, 0, 0), api.ctypes.c_size_t()
    assert h.L.laue_workspace_min_size(h.h, api.ctypes.byref(d), api.ctypes.byref(b)) == 0
    assert 0 <= h.workspace_size(T, n_obs=n_obs, n_model=n_model) - b.value <= 3 << 30
