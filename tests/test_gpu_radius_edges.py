"""adop_point_radius at the ends of its ranges, against an exhaustive FP64 search."""
import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu


def _exhaustive(xyz, k):
    import torch
    x = torch.from_numpy(xyz).cuda().double()
    out = torch.empty(len(xyz), dtype=torch.float64, device="cuda")
    for o in range(0, len(xyz), 2048):
        q = x[o:o + 2048]
        d2 = sum((q[:, None, a] - x[None, :, a]) ** 2 for a in range(3))
        d2[torch.arange(len(q)), torch.arange(o, o + len(q))] = float("inf")
        out[o:o + 2048] = torch.topk(d2, k, dim=1, largest=False).values[:, -1].sqrt()
    return out.cpu().numpy()


@pytest.mark.parametrize("median", [1e19, 1e-15])
def test_radius_of_huge_and_tiny_clouds(adop, median):
    """Cells whose square is beyond FP32, or about as small as it goes.  (Distances from 1.8e19 on,
    whose squares are no FP32 numbers, are +inf.)"""
    import torch
    n = 4000
    x = np.random.default_rng(3).random((n, 3)) * median / np.cbrt(3 * 4 / (4 * np.pi * n))
    xyz = np.ascontiguousarray(x, np.float32)
    got = adop.adop_point_radius(torch.from_numpy(xyz).cuda(), 4).cpu().numpy().astype(np.float64)
    want = _exhaustive(xyz, 4)
    near = want < 1.8e19
    assert 0.9 < near.mean()
    # an FP32 difference, square, sum and root of FP32 positions: a few units of 2^-24
    assert np.all(np.abs(got - want)[near] <= 4e-7 * want[near])
    assert np.all(got[~near] >= want[~near] * (1 - 4e-7))


@pytest.mark.parametrize("order", ["surface", "shuffled"])
@pytest.mark.parametrize("n,k", [(32768, 4), (32769, 4), (32769, 16), (32800, 4), (32801, 5)])
def test_radius_where_the_sample_bound_stops_covering_the_cloud(adop, n, k, order):
    """Up to 32768 points the samples' first bound comes from the whole cloud and is exact; past that a
    pass over the cloud lists what is within it, the last group of 32 points full or not."""
    import torch
    xyz = scenes.tiny_spheres(n, 1, seed=n).xyz
    if order == "shuffled":
        xyz = xyz[np.random.default_rng(n).permutation(n)]
    xyz = np.ascontiguousarray(xyz, np.float32)
    got = adop.adop_point_radius(torch.from_numpy(xyz).cuda(), k).cpu().numpy().astype(np.float64)
    want = _exhaustive(xyz, k)
    # exact while the neighbour is less than 8 cells of 1.5 medians away; FP32 as above
    near = want < 8 * 1.5 * np.median(want)
    assert near.mean() > 0.95
    assert np.all(np.abs(got - want)[near] <= 4e-7 * want[near])
    assert np.all(got[~near] >= want[~near] * (1 - 4e-7))
