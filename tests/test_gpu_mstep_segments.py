"""The two ways to count an angle's model spots by grain: one CTA an angle, and
the count spread over the spots where an angle holds many.  Empty angles behind
a full one lower the mean and leave every sum as it is, so the poses and
gradients of the two are equal bit for bit."""
import numpy as np
import pytest

import synthgen as sg
from _cases import GEOM

pytestmark = pytest.mark.gpu


def _block(rng, n_obs, grain):
    n = len(grain)
    s = np.concatenate([rng.uniform(-128, 128, (n, 2)), np.where(rng.random((n, 1)) < 0.5, 200.0, -200.0)], 1)
    c = rng.uniform(-2.5, 2.5, (n, 3))
    r = (s - c) / np.linalg.norm(s - c, axis=1, keepdims=True)
    p = s[rng.integers(0, n, n_obs)].copy()
    p[:, :2] += rng.normal(size=(n_obs, 2)) * 0.5
    return p, s, c, r


@pytest.mark.parametrize("n", [8191, 8192, 8193, 20011])
def test_counts_of_long_angles(n):
    import torch
    from paper_2404_06478_gb300 import api, build
    build.build()
    dev = torch.device("cuda", 0)
    cfg = sg.CONFIGS["medium"]
    lat = api.Lattice.cubic(cfg.a, cfg.hmax, cfg.centering, device=dev)
    M, N = int(lat.w_d0.shape[0]), n // 60 + 3  # the last grains see nothing
    rng = np.random.default_rng(n)
    grain = np.sort(rng.integers(0, N - 2, n))
    first = np.searchsorted(grain, grain)
    plane = (np.arange(n) - first) % M  # distinct within a grain
    assert np.bincount(grain).max() <= M
    p, s, c, r = _block(rng, 700, grain)
    ray = np.concatenate([r, np.full((n, 1), 2.0)], 1)
    w = rng.uniform(0.5, 1.5, n)
    out = []
    for empty in (0, 3):
        T = 1 + empty
        ob = api.ObsSpots.from_numpy(p, np.array([0] + [700] * T), device=dev)
        ms = api.ModelSpots.from_numpy(np.array([0] + [n] * T), grain, plane, ray, c, s, (s[:, 2] < 0).astype(int),
                                       device=dev)
        h = api.Handle(dev)
        f = torch.full((700,), -3.0, device=dev)
        g = torch.tensor(np.log(w), dtype=torch.float32, device=dev)
        om = torch.tensor(np.linspace(0.0, 0.3, T), dtype=torch.float32, device=dev)
        R = torch.tensor(np.tile(np.eye(3).reshape(9), (N, 1)), dtype=torch.float32, device=dev)
        x = torch.zeros(N, 3, device=dev)
        grad, val = api.objective_grad(h, GEOM, lat, ob, ms, f, g, 2.0, om, R, x)
        norms = torch.empty(N, 2, device=dev)
        api.mstep(h, GEOM, lat, ob, ms, f, g, 2.0, om, R, x, step_norms=norms)
        torch.cuda.synchronize()
        out.append((grad, val, R, x, norms))
    for a, b in zip(*out):
        assert torch.equal(a, b)
    assert int((out[0][1] != 0).sum()) > N // 2
    assert not out[0][0][-2:].any()
