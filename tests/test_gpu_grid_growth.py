"""The difference grids of rectangles over more than 1024 tiles are sized with the
tiles: a batch whose grids have more cells than any before, but whose tiles fit,
allocates nothing (an allocation would free what a captured graph uses, and its
clearing would have to be ordered with the caller's stream).  One large view
covered by huge splats and fifteen of one tile's width (two cells per tile), on a
side stream, images and gradients against a fresh context's: images bit for bit,
gradients to the order of float32 atomics (1e-5 of the norm)."""
import numpy as np
import pytest
import torch

from synth import workloads
from synth.scene import Camera, look_at
from tests._util import ensure_built, gpu_render, to_gpu_model

pytestmark = pytest.mark.gpu


def test_grids_do_not_outgrow_the_tiles():
    ensure_built()
    from paper_2408_12677_gb300 import abi
    from paper_2408_12677_gb300.torch_api import Context, camera_struct
    pose = look_at([0.1, 0.2, -0.1], [0.7, 3.0, 0.2])
    wide = Camera(700.0, 700.0, 650.0, 500.0, 1300, 1000)  # 5166 tiles, 5312 cells
    cams = [Camera(700.0, 700.0, 512.0, 320.0, 1024, 640)]  # 2560 tiles, 2665 cells
    cams += [Camera(700.0, 700.0, 8.0, 1800.0, 16, 3600)] * 15  # 3375 tiles, 6780 cells
    P = workloads.random_gaussians(np.random.default_rng(8), 600, cams[0], pose, 1, z_range=(1.5, 3.0), sh_rest_std=0.1)
    P["log_scales"][:40] = 0.5
    many = workloads.random_gaussians(np.random.default_rng(9), 16 * 600, wide, pose, 1)
    rng = np.random.default_rng(3)
    cu = lambda *s: torch.as_tensor(rng.standard_normal(s).astype(np.float32), device="cuda")
    wc, wd = [cu(3, c.height, c.width) for c in cams], [cu(c.height, c.width) for c in cams]
    cs, views = [camera_struct(c) for c in cams], [abi.make_viewmat(pose.R, pose.t)] * len(cams)
    out = []
    for fresh in (False, True):
        ctx, model = Context(0), to_gpu_model(P)
        h = ctx.handle
        abi.gs_ctx_reserve(h, 0, 0, 1 << 22)
        if not fresh:
            gpu_render(ctx, to_gpu_model(many), wide, pose)
            abi.gs_ctx_inject_alloc_failure(h, 1)
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            img = [[torch.empty_like(a) for a in (c, d, d)] for c, d in zip(wc, wd)]
            rcfg = abi.raster_cfg()
            abi.gs_render_fwd_batched(h, model.gaussians(), cs, views, rcfg, *[list(x) for x in zip(*img)])
            abi.gs_ctx_inject_alloc_failure(h, 0)
            abi.gs_render_bwd_batched(h, model.gaussians(), cs, views, rcfg, wc, wd, None, model.grads())
        torch.cuda.synchronize()
        out.append(([a.cpu().numpy() for i in img for a in i], model.grad.cpu().numpy().astype(np.float64)))
        ctx.close()
    assert max(float(a.max()) for a in out[1][0]) > 0.5
    for a, b in zip(out[0][0], out[1][0]):
        assert np.array_equal(a, b)
    assert np.linalg.norm(out[0][1] - out[1][1]) <= 1e-5 * np.linalg.norm(out[1][1])
