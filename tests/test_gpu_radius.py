"""adop_point_radius against an exhaustive FP64 search, where its paths change:
clouds the samples' subset covers and just does not (65536 points), both
orders in memory, curves, surfaces, volumes, more copies of a place than a
sample's list holds, and every list length."""
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


def _cloud(kind, n):
    rng = np.random.default_rng(n)
    if kind == "curve":
        t = np.sort(rng.random(n)) * 6.0
        x = np.stack([np.cos(t), np.sin(t), 0.2 * t], 1)
    elif kind == "volume":
        x = rng.random((n, 3)) * [2.0, 1.0, 0.5] - 0.3
    elif kind == "copies":
        x = scenes.tiny_spheres(n, 1, seed=n).xyz.copy()
        x[n // 4:n // 4 + 6000] = x[n // 4]
    else:
        x = scenes.tiny_spheres(n, 1, seed=n).xyz.copy()
        if kind == "shuffled":
            x = x[rng.permutation(n)]
    return np.ascontiguousarray(x, np.float32)


@pytest.mark.parametrize("kind,n,k", [
    ("surface", 5, 4), ("surface", 31, 4), ("surface", 300, 4), ("surface", 65536, 4), ("surface", 65537, 4),
    ("shuffled", 65537, 4), ("shuffled", 90001, 1), ("surface", 90001, 5), ("shuffled", 70000, 16),
    ("curve", 20011, 4), ("volume", 80021, 4), ("volume", 4099, 3), ("copies", 80000, 4)])
def test_radius_is_the_exhaustive_distance(adop, kind, n, k):
    import torch
    xyz = _cloud(kind, n)
    got = adop.adop_point_radius(torch.from_numpy(xyz).cuda(), k).cpu().numpy().astype(np.float64)
    want = _exhaustive(xyz, k)
    # an FP32 difference, square, sum and root of FP32 positions: a few units of 2^-24;
    # exact while the k-th neighbour is less than 8 cells of 1.5 medians away
    near = want < 8 * 1.5 * np.median(want) if np.median(want) > 0 else want >= 0
    assert np.all(np.abs(got - want)[near] <= 4e-7 * want[near])
    assert np.all(got[~near] >= want[~near] * (1 - 4e-7))
    assert near.mean() > 0.95
