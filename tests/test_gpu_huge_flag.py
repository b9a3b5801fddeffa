"""After a pass with rectangles of more than 1024 tiles, a context's passes without any bin as
fast as before: the scan integrates the difference grids only in passes that use them.  Four
views of 900 to 1056 tiles (one scan block, the grids one after the other, about 9 us when it
integrates them): medians of the scan and scatter stage over 60 passes, within 3 us."""
import numpy as np
import pytest
import torch

from synth import workloads
from synth.scene import Camera, look_at
from tests._util import ensure_built, to_gpu_model

pytestmark = pytest.mark.gpu


def test_grids_are_integrated_only_when_used():
    ensure_built()
    from paper_2408_12677_gb300 import abi
    from paper_2408_12677_gb300.torch_api import Context, camera_struct
    cams = [Camera(500.0, 500.0, 264.0, 256.0, 528, 512)] * 3 + [Camera(500.0, 500.0, 240.0, 240.0, 480, 480)]
    pose = look_at([0.1, 0.2, -0.1], [0.7, 3.0, 0.2])
    P = workloads.random_gaussians(np.random.default_rng(8), 5000, cams[0], pose, 0, z_range=(1.5, 3.0),
                                   log_scale_range=(-6.0, -5.0))
    Q = {k: v.copy() if hasattr(v, "copy") else v for k, v in P.items()}
    Q["log_scales"][:10] = 1.0
    ctx = Context(0)
    h = ctx.handle
    img = [[torch.empty(c + (k.height, k.width), device="cuda") for k in cams] for c in ((3,), (), ())]
    cs, views, rcfg = [camera_struct(c) for c in cams], [abi.make_viewmat(pose.R, pose.t)] * 4, abi.raster_cfg()

    def passes(model, n):
        us = []
        for _ in range(n):
            abi.gs_set_profiling(h, True)
            abi.gs_render_fwd_batched(h, model.gaussians(), cs, views, rcfg, *img)
            ms, count = abi.gs_profile_read(h)["duplicate"]
            us.append(1e3 * ms)
        abi.gs_set_profiling(h, False)
        return float(np.median(us))

    small, huge = to_gpu_model(P), to_gpu_model(Q)
    passes(small, 10)
    before = passes(small, 60)
    passes(huge, 1)
    after = passes(small, 60)
    assert after <= before + 3.0, (before, after)
    ctx.close()


def test_no_grids_for_views_of_few_tiles():
    """Views of at most 1024 tiles hold no such rectangle: 5000 tiles of eight views are scanned in three launches,
    with the projection, the scatter, the sort and the raster pass seven."""
    ensure_built()
    from paper_2408_12677_gb300 import abi
    from paper_2408_12677_gb300.torch_api import Context, camera_struct
    cam, pose = Camera(400.0, 400.0, 200.0, 200.0, 400, 400), look_at([0.1, 0.2, -0.1], [0.7, 3.0, 0.2])
    P = workloads.random_gaussians(np.random.default_rng(8), 3000, cam, pose, 0, log_scale_range=(-6.0, -5.0))
    ctx, model = Context(0), to_gpu_model(P)
    img = [[torch.empty(c + (400, 400), device="cuda") for _ in range(8)] for c in ((3,), (), ())]
    args = model.gaussians(), [camera_struct(cam)] * 8, [abi.make_viewmat(pose.R, pose.t)] * 8, abi.raster_cfg(), *img
    abi.gs_render_fwd_batched(ctx.handle, *args)
    before = ctx.stats()["kernel_launches"]
    abi.gs_render_fwd_batched(ctx.handle, *args)
    assert ctx.stats()["kernel_launches"] - before == 7
    ctx.close()
