"""The forward's launch-time choices against the oracle: sums seeded with each
pixel's nearest point (from 96 MB of pixel state) or cleared, one, two
or four points a lane in the accumulate pass (from 1167360 and 2334720 points on 152 SMs), every
depth-pass layer count, state kept or rendered again by the backward, and a
layer-mask buffer that is only 4-byte aligned."""
import numpy as np
import pytest

import scenes
from parity import compare, gpu_run, oracle_run

pytestmark = pytest.mark.gpu


def _camera(w, h, **kw):
    return scenes.Camera(w, h, 0.9 * w, 0.9 * w, w / 2, h / 2, k1=0.01, R=np.eye(3, dtype=np.float32),
                         t=np.array([-0.5, -0.5, 2.0], np.float32), **kw)


@pytest.mark.parametrize("n,c,dtype,levels,w,h,keep", [
    (1_167_359, 4, "f32", 4, 320, 200, True),   # one point a lane
    (1_167_361, 4, "f32", 4, 320, 200, True),   # two, and a last chunk of one point
    (2_334_721, 4, "f32", 4, 320, 200, False),  # four, and a last chunk of one point
    (400_003, 8, "bf16", 5, 333, 217, False),
    (350_001, 2, "f16", 2, 320, 200, True),
    (350_001, 1, "f32", 1, 320, 200, False),
    (40_001, 8, "bf16", 4, 2200, 1500, True),   # seeded
    (2_200_001, 8, "f32", 4, 2200, 1500, False),
    (40_001, 16, "f16", 3, 1400, 1000, True),
    (40_001, 3, "f32", 5, 2400, 2001, True),
    (20_011, 1, "f32", 8, 3000, 2400, False),
    (799_999, 4, "bf16", 4, 320, 200, True),    # backward in index order, and binned from 800000 on
    (800_003, 4, "bf16", 4, 320, 200, True),
    (800_003, 8, "f32", 4, 1600, 1100, False),  # in index order: fewer than 500 points a tile
    (4_200_003, 2, "f32", 2, 4128, 2080, True)])   # binned, more tiles than a block counts in shared memory
def test_forward_and_backward_paths(adop, orc, n, c, dtype, levels, w, h, keep):
    sc = scenes.tiny_spheres(n, c, seed=n % 1000)
    cams = [_camera(w, h)]
    G = [scenes.upstream_grad(w, h, levels, c, 7)]
    g = gpu_run(adop, sc, cams, dtype, levels=levels, grads=G, keep_state=keep, grad_assign=True)
    r = oracle_run(orc, sc, cams, dtype, levels=levels, grads=G)
    compare(g, r, dtype, check_state=keep)
    if keep:  # an empty pixel's sums are zero in a kept frame
        fr = g["frames"][0]
        acc = fr.acc.view(-1, c).cpu().numpy()
        assert not acc[r["cnt"][0] == 0].any()


@pytest.mark.parametrize("keep", [True, False])
def test_several_cameras_of_a_large_cloud(adop, keep):
    """From 4M points on the backward takes the cameras two at a time: the
    same gradients as one call per camera, summed, and the same pose rows
    (FP32 sums in another order)."""
    import torch
    from parity import assert_close
    n = (1 << 22) + 3
    sc = scenes.tiny_spheres(n, 4, seed=9)
    cams = [_camera(200 + 16 * k, 150) for k in range(3)]
    pts = adop.Points(torch.from_numpy(sc.xyz).cuda(), torch.from_numpy(sc.feat).cuda())
    params = adop.Params(4, 0.01, 1e-3, None, adop.ADOP_FLAG_GRAD_ASSIGN)
    G = [[torch.from_numpy(g).cuda() for g in scenes.upstream_grad(c.w, c.h, 4, 4, 30 + k)]
         for k, c in enumerate(cams)]

    def grads(sub, g):
        frames = [adop.Frame.alloc(c, 4, 4, torch.float32, keep, "cuda", n if keep else None) for c in sub]
        ws = adop.alloc_workspace(pts, sub, params)
        adop.adop_render_forward(pts, sub, params, frames, ws)
        out = [torch.full((n, 4), float("nan"), device="cuda"), torch.full((n, 3), float("nan"), device="cuda"),
               torch.zeros((len(sub), 6), device="cuda"), torch.zeros((len(sub), 6), device="cuda")]
        adop.adop_render_backward(pts, sub, params, frames, g, *out, ws)
        return [o.cpu().numpy().astype(np.float64) for o in out]

    got = grads(cams, G)
    one = [grads([c], [g]) for c, g in zip(cams, G)]
    for j in range(2):
        assert_close(got[j], sum(o[j] for o in one), 1e-5, "per-point gradients")
    for j in (2, 3):
        want = np.concatenate([o[j] for o in one])
        assert np.all(np.abs(got[j] - want) <= 1e-4 * np.abs(want).max())


@pytest.mark.parametrize("dtype", ["f32", "f16"])
def test_binned_gradient_buffers_only_aligned_as_asked(adop, dtype):
    """dL/dx 4 bytes past a 16-byte boundary, and dL/dtau in 16 bits, give the
    zero gradients and the others of an aligned call (binned, a point count
    that is no multiple of 32, buffers filled with NaN).  A point's sum over
    its layers is split where the list of a warp's pairs is, so that FP32
    rounding may differ, and with it one step of FP16."""
    import torch
    from parity import assert_close
    n, c = 800_021, 3
    sc = scenes.tiny_spheres(n, c, seed=3)
    cam = _camera(320, 200)
    pts = adop.Points(torch.from_numpy(sc.xyz).cuda(), torch.from_numpy(sc.feat).cuda())
    params = adop.Params(4, 0.01, 1e-3, None, adop.ADOP_FLAG_GRAD_ASSIGN)
    fr = adop.Frame.alloc(cam, c, 4, torch.float32, True, "cuda", n)
    ws = adop.alloc_workspace(pts, [cam], params)
    adop.adop_render_forward(pts, [cam], params, [fr], ws)
    G = [[torch.from_numpy(g).cuda() for g in scenes.upstream_grad(cam.w, cam.h, 4, c, 8)]]
    got = []
    for offset in (0, 1):
        gx = torch.full((n * 3 + 4,), float("nan"), device="cuda")[offset:offset + n * 3].view(n, 3)
        assert gx.data_ptr() % 16 == 4 * offset
        gf = torch.full((n, c), float("nan"), dtype=torch.float16 if dtype == "f16" else torch.float32, device="cuda")
        adop.adop_render_backward(pts, [cam], params, [fr], G, gf, gx, None, None, ws)
        got.append((gf.float().cpu().numpy(), gx.cpu().numpy()))
    assert_close(got[0][0], got[1][0], 1e-6 if dtype == "f32" else 2e-3, "dL/dtau")
    assert_close(got[0][1], got[1][1], 1e-5, "dL/dx")
    unseen = fr.vis.cpu().numpy() & 0xFF == 0
    assert unseen.any() and not got[0][0][unseen].any() and not got[0][1][unseen].any()


@pytest.mark.parametrize("c,dtype", [(4, "f32"), (3, "f16")])
def test_gradients_zeroed_ahead(adop, c, dtype):
    """From 16M points on, eight per pixel, the zero gradients are written
    ahead of the point pass: the same as gradients added onto zeros (FP32
    rounding of sums in another order, one step of FP16), every point written
    (buffers filled with NaN), dL/dx on a 16-byte boundary and off it."""
    import torch
    from parity import assert_close
    n = (1 << 24) + 5
    rng = np.random.default_rng(1)
    xyz = torch.from_numpy(rng.random((n, 3), dtype=np.float32)).cuda()
    feat = torch.from_numpy(rng.random((n, c), dtype=np.float32)).cuda()
    cam = _camera(320, 200)
    pts = adop.Points(xyz, feat)
    params = adop.Params(4, 0.01, 1e-3, None, adop.ADOP_FLAG_GRAD_ASSIGN)
    fr = adop.Frame.alloc(cam, c, 4, torch.float32, True, "cuda", n)
    ws = adop.alloc_workspace(pts, [cam], params)
    adop.adop_render_forward(pts, [cam], params, [fr], ws)
    G = [[torch.from_numpy(g).cuda() for g in scenes.upstream_grad(cam.w, cam.h, 4, c, 8)]]
    want = [torch.zeros((n, c), device="cuda"), torch.zeros((n, 3), device="cuda")]
    adop.adop_render_backward(pts, [cam], adop.Params(4, 0.01, 1e-3, None, 0), [fr], G, *want, None, None, ws)
    want = [w.cpu().numpy() for w in want]
    seen = fr.vis.cpu().numpy() & 0xFF != 0
    assert seen.any() and not seen.all()
    for offset in (0, 1):
        gx = torch.full((n * 3 + 4,), float("nan"), device="cuda")[offset:offset + n * 3].view(n, 3)
        gf = torch.full((n, c), float("nan"), dtype=torch.float16 if dtype == "f16" else torch.float32, device="cuda")
        adop.adop_render_backward(pts, [cam], params, [fr], G, gf, gx, None, None, ws)
        gf, gx = gf.float().cpu().numpy(), gx.cpu().numpy()
        assert not gf[~seen].any() and not gx[~seen].any()
        assert_close(gf[seen], want[0][seen], 1e-6 if dtype == "f32" else 2e-3, "dL/dtau")
        assert_close(gx[seen], want[1][seen], 1e-5, "dL/dx")


def test_layer_masks_only_4_byte_aligned(adop):
    import torch
    sc = scenes.tiny_spheres(2_334_731, 4, seed=5)
    cam = _camera(320, 200)
    pts = adop.Points(torch.from_numpy(sc.xyz).cuda(), torch.from_numpy(sc.feat).cuda())
    params = adop.Params(4, 0.01, 1e-3, None, 0)
    got = []
    for offset in (0, 1):
        fr = adop.Frame.alloc(cam, 4, 4, torch.float32, True, "cuda", sc.n)
        buf = torch.full((sc.n + 2,), -1, dtype=torch.int32, device="cuda")
        fr.vis = buf[offset:offset + sc.n]
        ws = adop.alloc_workspace(pts, [cam], params)
        adop.adop_render_forward(pts, [cam], params, [fr], ws)
        got.append(fr.vis.cpu().numpy())
        assert buf[offset + sc.n] == -1 and (offset == 0 or buf[0] == -1)
    assert np.array_equal(got[0], got[1])
    assert (got[0] == 0).any() and (got[0] & 0xFF != 0).any()
