"""The render server where a cloud's byte per point outweighs the pixel states:
requests that fit the pool together run together."""
import numpy as np
import pytest

import scenes
from parity import RTOL_FEAT_F32, assert_close

pytestmark = pytest.mark.gpu

LEVELS = 4


def _alone(adop, torch, pts, cam):
    params = adop.Params(LEVELS, 0.01, 1e-3, None, 0)
    fr = adop.Frame.alloc(cam, pts.feat.shape[1], LEVELS, torch.float32, True, "cuda")
    ws = adop.alloc_workspace(pts, [cam], params, None, "cuda")
    adop.adop_render_forward(pts, [cam], params, [fr], ws)
    torch.cuda.synchronize()
    return np.concatenate([im.cpu().numpy().ravel() for im in fr.images])


def test_small_views_of_a_large_cloud_share_a_batch(adop):
    """16 views of 180 KB of state each over 4M points in a 40 MiB pool: one batch of 16."""
    import torch
    sc = scenes.tiny_spheres(4_000_000, 8, seed=9)
    pts = adop.Points(torch.from_numpy(sc.xyz).cuda(), torch.from_numpy(sc.feat).cuda())
    srv = adop.Server(mem_budget_bytes=40 << 20, max_slots=64, streams=1, max_batch=16, levels=LEVELS,
                      batch_window_us=900_000)  # a batch that is not full waits this long
    cid = srv.load_cloud(pts)
    cams = []
    for k in range(16):
        eye = np.array([np.cos(0.4 * k), 0.2, np.sin(0.4 * k)]) * 2.5 + 0.5
        R, t = scenes.look_at(eye, np.full(3, 0.5))
        cams.append(scenes.Camera(64, 48, 58.0, 58.0, 32.0, 24.0, R=R, t=t))
    outs = [torch.empty(adop.output_numel(c, 8, LEVELS), dtype=torch.float32, device="cuda") for c in cams]
    torch.cuda.synchronize()
    tickets = [srv.submit(cid, c, o) for c, o in zip(cams, outs)]
    for t in tickets:
        assert srv.wait(t, 60_000) == 0
    st = srv.stats()
    srv.close()
    assert st["completed"] == 16 and st["batches"] == 1 and st["mean_batch"] == 16.0, st
    for k in (0, 7, 15):
        assert_close(outs[k].cpu().numpy(), _alone(adop, torch, pts, cams[k]), RTOL_FEAT_F32, f"request {k}")
