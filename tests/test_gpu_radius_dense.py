"""adop_point_radius where the points lie so densely that a search cell holds
more candidates than the first search looks at (65536), beside a sparse
remainder that sets the cell size, against an exhaustive FP64 search."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _exhaustive(xyz, at, k):
    import torch
    x = torch.from_numpy(xyz).cuda().double()
    out = []
    for o in range(0, len(at), 512):
        i = torch.from_numpy(at[o:o + 512]).cuda()
        d2 = sum((x[i][:, None, a] - x[None, :, a]) ** 2 for a in range(3))
        d2[torch.arange(len(i)), i] = float("inf")
        out.append(torch.topk(d2, k, dim=1, largest=False).values[:, -1].sqrt())
    return torch.cat(out).cpu().numpy()


def _cloud(kind, sparse, dense):
    """`sparse` points in the unit box and `dense` ones in a part of it as wide as a search cell,
    1.6 * 1.5 medians of the distance to the fourth neighbour: 4 points in a ball of that radius."""
    rng = np.random.default_rng(dense)
    x = rng.random((sparse + dense, 3))
    if kind == "plane":
        width = 2.4 * np.sqrt(4 / (np.pi * sparse))
        x[:sparse, 2] = 0.0
        x[sparse:] = [0.413, 0.377, 0.0] + width * x[sparse:] * [1, 1, 1e-3]
    else:
        width = 2.4 * np.cbrt(3 * 4 / (4 * np.pi * sparse))
        x[sparse:] = [0.413, 0.377, 0.521] + width * x[sparse:]
    if kind == "beside":  # a few sparse points next to the dense ones: their balls reach into these
        x[:600] = [0.413, 0.377, 0.521] + width * (1.0 + 0.3 * x[:600])
    return np.ascontiguousarray(rng.permutation(x), np.float32)


@pytest.mark.parametrize("kind,sparse,dense,k", [
    ("volume", 130000, 110000, 4), ("volume", 130000, 70000, 16), ("plane", 130000, 90000, 4),
    ("beside", 150000, 140000, 4), ("volume", 900000, 400000, 4)])
def test_radius_in_a_dense_part(adop, kind, sparse, dense, k):
    import torch
    xyz = _cloud(kind, sparse, dense)
    dev = torch.from_numpy(xyz).cuda()
    got = adop.adop_point_radius(dev, k).cpu().numpy().astype(np.float64)
    again = adop.adop_point_radius(dev, k).cpu().numpy().astype(np.float64)
    assert np.array_equal(got, again)  # exact results do not depend on the order of the sort
    # every kind of point: the smallest distances found are the dense part, the rest in order of index
    order = np.argsort(got, kind="stable")
    at = np.unique(np.concatenate([order[::len(xyz) // 3000], order[:dense][-1000:], order[dense:dense + 1000]]))
    want = _exhaustive(xyz, at, k)
    # an FP32 difference, square, sum and root of FP32 positions: a few units of 2^-24
    assert np.all(np.abs(got[at] - want) <= 4e-7 * want)
