"""The sparse E-step where the neighbour lists hold more records than 32 bits
count (33.6 million model spots of 64 neighbours).  The angle blocks are copies
of one another, with dustbins of their own, so every block has the potentials of
a solve of one block alone, bit for bit."""
import numpy as np
import pytest

from _cases import GEOM
from test_gpu_lists import _blocks, env  # noqa: F401

pytestmark = pytest.mark.gpu


def test_records_past_32_bits(env):
    api, torch, dev = env["api"], env["torch"], env["dev"]
    T, ni, nj, rho = 65536, 64, 513, 64
    assert T * nj * rho > 2 ** 31
    if torch.cuda.mem_get_info(dev)[0] < 60 << 30:
        pytest.skip("needs 45 GB of device memory")
    p, _, m, _ = _blocks([(ni, nj)], 41, GEOM)
    f4 = lambda a, w: torch.tensor(np.concatenate([a, w.reshape(-1, 1)], 1), dtype=torch.float32, device=dev)
    p4, c4 = f4(p, np.zeros(ni)), f4(m["center"], np.zeros(nj))
    r4, s4 = torch.tensor(m["ray"], dtype=torch.float32, device=dev), f4(m["spot"], np.asarray(m["det"], float))

    def solve(T):
        h = api.Handle(dev)
        off = lambda n: torch.arange(T + 1, dtype=torch.int32, device=dev) * n
        label = torch.zeros(T * nj, dtype=torch.int32, device=dev)
        ob = api.ObsSpots(p4.repeat(T, 1), off(ni))
        ms = api.ModelSpots(T, T * nj, off(nj), label, label, label, r4.repeat(T, 1), c4.repeat(T, 1), s4.repeat(T, 1))
        out = api.cost_sinkhorn_sparse(h, GEOM, ob, ms, 2.0, 2.25, 3, rho=rho, dust_mode=1, harvest=True,
                                       col_harvest=True)
        torch.cuda.synchronize()
        assert h.device_status() == 0
        return out

    one, many = solve(1), solve(T)
    for k, n in (("f", ni), ("g", nj), ("margin", ni), ("q", nj)):
        assert bool((many[k].view(T, n) == one[k]).all()), k
    assert bool((many["dust"].view(2, T) == one["dust"].view(2, 1)).all())
    first = torch.arange(T, dtype=torch.int32, device=dev).view(T, 1) * nj
    want = torch.where(one["assign"] < 0, one["assign"], one["assign"] + first)
    assert bool((many["assign"].view(T, ni) == want).all())
    assert int((one["assign"] >= 0).sum()) > 0
