"""Selection of a set's spots where the window's axes are not spread evenly:
many equal distances, clusters and gaps around the seed.

A distance 1 - |n . n0| of unit axes has an error of at most 3 roundings of
products near 1 and of the axes themselves, below 4e-7 together; spots whose
distances differ by less may take either order.  Equal axes have equal
distances, and the lower index comes first."""
import numpy as np
import pytest

import oracle.proposal as op
import synthgen as sg

pytestmark = pytest.mark.gpu

GEOM = sg.Geometry()
TOL = 4e-7


def _sets(p, seeds):
    """(ids, axes in 64 bits) of sets over one angle of spots p."""
    import torch
    from paper_2404_06478_gb300 import api, build, proposal as pr
    build.build()
    dev = torch.device("cuda", 0)
    h = api.Handle(dev)
    n, B = len(p), len(seeds)
    p4 = np.zeros((n, 4), np.float32)
    p4[:, :3] = p
    ti = lambda a: torch.tensor(np.asarray(a), dtype=torch.int32, device=dev)
    batch = pr.Batch(h, B)
    axes = torch.empty(n, 4, dtype=torch.float32, device=dev)
    pr.make_sets(h, GEOM, torch.tensor(p4, device=dev), ti([0, n]), torch.zeros(1, device=dev), ti(seeds),
                 ti(np.zeros(B)), ti(np.ones(B)), batch, axes)
    torch.cuda.synchronize()
    assert h.device_status() == 0
    return batch.ids.cpu().numpy().reshape(B, op.KSET), axes.cpu().numpy()[:, :3].astype(np.float64)


def _points(xy, z=-200.0):
    return np.concatenate([xy, np.full((len(xy), 1), z)], 1)


@pytest.mark.parametrize("n_equal", [60, 127, 128, 260, 600, 4000, 4200, 9000])
@pytest.mark.parametrize("n_nearer", [0, 50])
def test_equal_axes_in_index_order(n_equal, n_nearer):
    """n_equal spots at one place, which the seed sees behind n_nearer others:
    the nearer ones and the lowest indices of the equal ones."""
    rng = np.random.default_rng(n_equal + n_nearer)
    here = np.array([31.0, -17.0])
    near = here + rng.uniform(2.0, 4.0, (n_nearer, 2))
    equal = np.repeat(here[None] + 9.0, n_equal, 0)
    rest = rng.uniform(-120.0, -60.0, (700, 2))
    xy = np.concatenate([here[None], near, equal, rest])
    order = rng.permutation(len(xy))
    kind = np.concatenate([[0], np.full(n_nearer, 1), np.full(n_equal, 2), np.full(700, 3)])[order]
    seed = int(np.nonzero(kind == 0)[0][0])
    ids, _ = _sets(_points(xy[order]), [seed])
    take = min(op.KSET - 1 - n_nearer, n_equal)
    assert ids[0, 0] == seed
    assert sorted(ids[0, 1:1 + n_nearer]) == sorted(np.nonzero(kind == 1)[0])
    np.testing.assert_array_equal(ids[0, 1 + n_nearer:1 + n_nearer + take], np.nonzero(kind == 2)[0][:take])
    assert (kind[ids[0, 1 + n_nearer + take:]] == 3).all()


@pytest.mark.parametrize("groups", [
    [(6000, (20.0, 22.0)), (2000, (-120.0, 120.0))],    # more around the seed than the first distance should hold
    [(20000, (20.0, 20.5))],                            # all of them
    [(40, (20.0, 22.0)), (6000, (-120.0, -60.0))],      # fewer
    [(200, (20.0, 20.1)), (9000, (60.0, 61.0))],        # some around it, many at one distance behind
    [(4096, (-120.0, 120.0))], [(4098, (-120.0, 120.0))],  # the buffer's size, seed included
], ids=["dense", "all_dense", "sparse", "gap", "buffer", "over"])
def test_uneven_windows(groups):
    rng = np.random.default_rng(len(groups) + groups[0][0])
    xy = np.concatenate([rng.uniform(lo, hi, (n, 2)) for n, (lo, hi) in groups])
    seeds = np.concatenate([rng.integers(0, groups[0][0], 6), rng.integers(0, len(xy), 6)])
    ids, n = _sets(_points(xy), seeds)
    for b, i0 in enumerate(seeds):
        assert ids[b, 0] == i0
        got = ids[b, 1:]
        d = 1.0 - np.abs(n @ n[i0])
        d[i0] = np.inf
        kth = np.sort(d)[op.KSET - 2]
        assert len(set(got.tolist())) == op.KSET - 1 and (got >= 0).all()
        assert d[got].max() <= kth + TOL
        assert set(np.nonzero(d < kth - TOL)[0]) <= set(got.tolist())
        assert (np.diff(d[got]) >= -TOL).all()
