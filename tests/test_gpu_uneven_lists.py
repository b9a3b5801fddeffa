"""Raster regions made smaller where a few lists are much longer than the rest: a
sync-mode pass, which knows the lists' lengths, against a no-sync one of a
context that has seen none (regions by the tile count alone).  Images bit for
bit (a pixel's arithmetic does not depend on its region), gradients to the
float32 order of their sums (1e-5 of the array's norm)."""
import numpy as np
import pytest
import torch

from synth import workloads
from synth.scene import Camera, look_at
from tests._util import ensure_built, to_gpu_model

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [(16, 16), (8, 32), (32, 8)])
def test_regions_by_list_lengths(tile):
    ensure_built()
    from paper_2408_12677_gb300 import abi
    from paper_2408_12677_gb300.torch_api import Context, camera_struct
    cam = Camera(500.0, 500.0, 320.0, 240.0, 637, 479)
    pose = look_at([0.1, 0.2, -0.1], [0.7, 3.0, 0.2])
    rng = np.random.default_rng(4)
    n = 9000
    P = workloads.random_gaussians(rng, n, cam, pose, 1, log_scale_range=(-6.0, -5.0), sh_rest_std=0.1)
    mid = P["means"].mean(0)
    P["means"][:3000] = (mid + 0.01 * rng.standard_normal((3000, 3))).astype(np.float32)
    P["opacity_logits"][:3000] = -4.5
    cu = lambda a: torch.as_tensor(a.astype(np.float32), device="cuda")
    wc, wd = cu(rng.standard_normal((3, cam.height, cam.width))), cu(rng.standard_normal((cam.height, cam.width)))
    rcfg, camS, view = abi.raster_cfg(tile_w=tile[0], tile_h=tile[1]), camera_struct(cam), abi.make_viewmat(pose.R, pose.t)
    out = []
    for sync in (True, False):
        ctx, model = Context(0), to_gpu_model(P)
        if not sync:
            abi.gs_ctx_reserve(ctx.handle, n, cam.width * cam.height, 1 << 20)
            abi.gs_ctx_set_sync(ctx.handle, False)
        col, dep, alp = torch.empty_like(wc), torch.empty_like(wd), torch.empty_like(wd)
        abi.gs_render_fwd(ctx.handle, model.gaussians(), camS, view, rcfg, col, dep, alp)
        ranges = torch.empty((-(-cam.width // tile[0]) * -(-cam.height // tile[1]), 2), dtype=torch.int32, device="cuda")
        abi.gs_get_tile_ranges(ctx.handle, ranges)
        lens = (ranges[:, 1] - ranges[:, 0]).long()
        assert len(lens) >= 6 * 152 and 1024 <= int(lens.max()) <= 4096
        assert int(lens.max()) * 24 * 152 > 8 * int(lens.sum())  # two pixels per lane instead of four
        abi.gs_render_bwd(ctx.handle, model.gaussians(), camS, view, rcfg, wc, wd, None, model.grads())
        torch.cuda.synchronize()
        abi.gs_sync_status(ctx.handle)
        out.append((col.cpu().numpy(), dep.cpu().numpy(), alp.cpu().numpy(), model.grad.cpu().numpy().astype(np.float64)))
        ctx.close()
    for a, b in zip(out[0][:3], out[1][:3]):
        assert np.array_equal(a, b)
    assert np.linalg.norm(out[0][3] - out[1][3]) <= 1e-5 * np.linalg.norm(out[1][3])
