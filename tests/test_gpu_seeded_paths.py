"""Sums seeded with each pixel's nearest point (from 96 MB of pixel state, a
kept one only with a point per 32 pixels) with everything that decides which
points count and what an empty pixel shows, in several cameras of one launch
and in the server; and the backward's choices that follow the channel count
and the number of screen tiles.  Against the oracle, or the render alone."""
import numpy as np
import pytest

import scenes
from parity import RTOL_FEAT_F32, assert_close, compare, gpu_run, oracle_run

pytestmark = pytest.mark.gpu


def _camera(w, h, **kw):
    return scenes.Camera(w, h, 0.9 * w, 0.9 * w, w / 2, h / 2, k1=0.01, R=np.eye(3, dtype=np.float32),
                         t=np.array([-0.5, -0.5, 2.0], np.float32), **kw)


N = 150_001  # more than a point per 32 of the 4.4M pixels


@pytest.mark.parametrize("keep", [True, False])
@pytest.mark.parametrize("what", ["plain", "log", "discard", "normals", "env", "tangential"])
def test_seeded_forward_and_backward(adop, orc, what, keep):
    sc = scenes.tiny_spheres(N, 8, seed=11)
    if what == "log":
        sc = scenes.Scene(sc.xyz, (sc.feat * 0.5).astype(np.float32), sc.normals)
    cams = [_camera(2200, 1500)]
    if what == "tangential":  # each camera's state is below 96 MB, their sum is not
        cams = [_camera(1400, 1000), _camera(1400, 1000, p1=2e-3, p2=-1e-3)]
    G = [scenes.upstream_grad(c.w, c.h, 4, 8, 20 + k) for k, c in enumerate(cams)]
    gpu, ref = {}, {}
    if what == "log":
        gpu, ref = {"flags": adop.ADOP_FLAG_LOG_DESCRIPTORS}, {"log_desc": True}
    if what == "normals":
        gpu, ref = {"flags": adop.ADOP_FLAG_NORMAL_CULL, "normals": True}, {"normals": True}
    if what == "discard":
        rng = np.random.default_rng(12)
        d = (rng.uniform(0.5e-3, 4e-3, N).astype(np.float32), rng.random(N).astype(np.float32), 1.5)
        gpu, ref = {"flags": adop.ADOP_FLAG_DISCARD, "discard": d}, {"discard": d}
    if what == "env":
        gpu = ref = {"env": scenes.env_map(8, 64, 128, seed=13)}
    g = gpu_run(adop, sc, cams, "f32", grads=G, keep_state=keep, **gpu)
    r = oracle_run(orc, sc, cams, "f32", grads=G, **ref)
    assert (r["cnt"][0] == 0).any() and (r["cnt"][0] > 1).any()
    compare(g, r, check_state=keep, env=what == "env")


@pytest.mark.parametrize("n,c,w,h,levels,keep", [
    (299_999, 16, 1280, 720, 4, True),    # in index order
    (300_001, 16, 1280, 720, 4, False),   # binned
    (40_001, 16, 320, 200, 8, True),      # the accumulate pass with 16 channels and more than five layers
    (849_999, 8, 1920, 1080, 4, False),   # in index order: fewer than 500 points a tile
    (850_001, 8, 1920, 1080, 4, True),    # binned
    (850_001, 8, 3200, 1600, 4, False),   # binned, 5000 tiles
    (153_000, 4, 640, 480, 4, True)])     # a point pass of less than a wave of blocks
def test_backward_choices(adop, orc, n, c, w, h, levels, keep):
    sc = scenes.tiny_spheres(n, c, seed=n % 1000)
    cams = [_camera(w, h)]
    G = [scenes.upstream_grad(w, h, levels, c, 7)]
    g = gpu_run(adop, sc, cams, "bf16", levels=levels, grads=G, keep_state=keep, grad_assign=True)
    r = oracle_run(orc, sc, cams, "bf16", levels=levels, grads=G)
    compare(g, r, "bf16", check_state=keep)


@pytest.mark.parametrize("room", [True, False])
def test_server_with_seeded_sums(adop, room):
    """Two clouds (four points a lane, a last chunk of one point) at 2200x1500, with room in the pool for
    the depth pass's bytes and without: the images of the render alone."""
    import torch
    n, levels = 2_334_721, 4
    pts = []
    for seed in (5, 6):
        sc = scenes.tiny_spheres(n, 8, seed=seed)
        pts.append(adop.Points(torch.from_numpy(sc.xyz).cuda(), torch.from_numpy(sc.feat).cuda()))
    cams = [_camera(2200, 1500), _camera(2200, 1500, p1=1e-3)]
    state = sum((2200 >> l) * (1500 >> l) for l in range(levels)) * (8 + 4 + 32) + 3 * 256
    srv = adop.Server(mem_budget_bytes=2 * state + (16 << 20 if room else 1 << 20), max_slots=2, streams=1, max_batch=2,
                      levels=levels, batch_window_us=900_000)
    ids = [srv.load_cloud(p) for p in pts]
    outs = [torch.empty(adop.output_numel(c, 8, levels), dtype=torch.float32, device="cuda") for c in cams]
    torch.cuda.synchronize()
    tickets = [srv.submit(i, c, o) for i, c, o in zip(ids, cams, outs)]
    for t in tickets:
        assert srv.wait(t, 60_000) == 0
    st = srv.stats()
    srv.close()
    assert st["batches"] == 1 and (st["mem_peak"] >= 2 * (state - 768 + n)) == room, st
    for p, c, o in zip(pts, cams, outs):
        params = adop.Params(levels, 0.01, 1e-3, None, 0)
        fr = adop.Frame.alloc(c, 8, levels, torch.float32, True, "cuda")
        ws = adop.alloc_workspace(p, [c], params, None, "cuda")
        adop.adop_render_forward(p, [c], params, [fr], ws)
        torch.cuda.synchronize()
        want = np.concatenate([im.cpu().numpy().ravel() for im in fr.images])
        assert_close(o.cpu().numpy(), want, RTOL_FEAT_F32, "image")


@pytest.mark.parametrize("keep", [True, False])
@pytest.mark.parametrize("w,h", [(1100, 900), (320, 200)])
def test_several_cameras_of_a_large_cloud(adop, w, h, keep):
    """From 4M points on the backward takes three cameras two at a time where their pixel records (126 MB
    here, 8 MB) are more than 96 MB: the gradients of one call per camera, summed, and the same pose rows
    (FP32 sums in another order)."""
    import torch
    n = (1 << 22) + 3
    sc = scenes.tiny_spheres(n, 4, seed=9)
    cams = [_camera(w, h + 16 * k) for k in range(3)]
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
