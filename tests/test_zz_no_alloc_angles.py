"""The no-allocation E-step takes every problem whose spots, order and tables
need at most 64 MiB, also where the angles hold few spots each and what the
passes keep beside them needs more than that.  The limits on T here are those of
the layout without the passes' own tables."""
import numpy as np
import pytest

from _cases import GEOM
from test_gpu_lists import _blocks, env  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_obs,n_model,T", [(10, 7, 67000), (1, 1, 225456), (2, 0, 220000)])
def test_many_small_angles(env, n_obs, n_model, T):
    api, torch, dev = env["api"], env["torch"], env["dev"]
    p, _, m, _ = _blocks([(n_obs, max(n_model, 1))], 51, GEOM)
    f4 = lambda a, w: torch.tensor(np.concatenate([a, np.asarray(w, float).reshape(-1, 1)], 1), dtype=torch.float32,
                                   device=dev)
    rep = lambda a: a.repeat(T, 1)[:max(T * n_model, 1)]
    ob = api.ObsSpots(f4(p, np.zeros(n_obs)).repeat(T, 1), torch.arange(T + 1, dtype=torch.int32, device=dev) * n_obs)
    label = torch.zeros(max(T * n_model, 1), dtype=torch.int32, device=dev)
    ms = api.ModelSpots(T, T * n_model, torch.arange(T + 1, dtype=torch.int32, device=dev) * n_model, label, label,
                        label, rep(torch.tensor(m["ray"], dtype=torch.float32, device=dev)),
                        rep(f4(m["center"], np.zeros(len(m["center"])))), rep(f4(m["spot"], m["det"])))
    want = api.cost_sinkhorn(api.Handle(dev), GEOM, ob, ms, 2.0, 2.25, 3, dust_mode=1)
    f, g = torch.empty(T * n_obs, device=dev), torch.empty(max(T * n_model, 1), device=dev)
    dust, assign = torch.zeros(2 * T, device=dev), torch.empty(T * n_obs, dtype=torch.int32, device=dev)
    margin, status = torch.empty(T * n_obs, device=dev), torch.full((1,), 99, dtype=torch.int32, device=dev)
    rc = api.cost_sinkhorn_noalloc(GEOM, ob, ms, 2.0, 2.25, 3, f, g, dust, assign, margin, status=status, dust_mode=1)
    torch.cuda.synchronize()
    assert rc == 0 and int(status) == 0
    for k, v in (("f", f), ("g", g[:T * n_model]), ("dust", dust), ("assign", assign), ("margin", margin)):
        assert torch.equal(v, want[k]), k


@pytest.mark.parametrize("n_obs,n_model,T", [(10, 7, 67100), (1, 1, 225500), (100, 70, 8200)])
def test_larger_problems_are_refused(env, n_obs, n_model, T):
    api, torch, dev = env["api"], env["torch"], env["dev"]
    p, I_off, m, J_off = _blocks([(4, 4)], 52, GEOM)
    ob = api.ObsSpots.from_numpy(p, I_off, device=dev)
    ms = api.ModelSpots.from_numpy(J_off, m["grain"], m["plane"], m["ray"], m["center"], m["spot"], m["det"], device=dev)
    o_s, m_s, g_s, prm = ob.struct(), ms.struct(), api.geometry_struct(GEOM), api.ot_params(2.0, 2.25, 3)
    o_s.T = m_s.T = T  # refused on the host, before anything reads the arrays
    o_s.n, m_s.n, m_s.capacity = T * n_obs, T * n_model, T * n_model
    from paper_2404_06478_gb300 import _native as N
    f = torch.zeros(8, device=dev)
    ref = api.ctypes.byref
    rc = N.lib().laue_cost_sinkhorn_noalloc(ref(g_s), ref(o_s), ref(m_s), ref(prm), api._ptr(f), api._ptr(f), None, None,
                                            None, None, None, None, api._stream())
    assert rc == N.LAUE_ERR_CAPACITY
