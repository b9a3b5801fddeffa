"""Thin slanted splats (30:1, at all angles): their bounding boxes hold many times the pixels
that they reach, so the raster passes also test the ellipse's extent over each row of blocks.
Images, the blended-pair counter and gradients against the oracle (tolerances as in
test_gpu_render and test_gpu_grad), with one, two and four pixels per lane and every tile shape;
and the evaluated pixels: a row of up to four pixels' height evaluates at most the ellipse's
width plus four columns, under four times the pixels blended (a box 60 px wide would evaluate
over ten times as many)."""
import numpy as np
import pytest

from oracle import render as R
from synth import workloads
from synth.scene import Camera, look_at
from tests._util import compare, ensure_built, gpu_backward, gpu_render, oracle_params, to_gpu_model
from tests.test_gpu_grad import check_grad_arrays

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w,h,n,tile", [(93, 70, 120, (16, 16)), (333, 221, 250, (8, 32)), (611, 420, 300, (16, 16)),
                                        (611, 420, 300, (32, 8))])
def test_thin_splats(w, h, n, tile):
    ensure_built()
    from paper_2408_12677_gb300 import abi
    from paper_2408_12677_gb300.torch_api import Context
    cam, pose = Camera(150.0, 150.0, w / 2, h / 2, w, h), look_at([0.1, 0.2, -0.1], [0.7, 3.0, 0.2])
    rng = np.random.default_rng(17)
    P = workloads.random_gaussians(rng, n, cam, pose, 1, z_range=(1.5, 4.0), sh_rest_std=0.1)
    P["log_scales"][:] = np.log(0.2) + rng.uniform(-0.3, 0.3, (n, 3)) + np.array([0.0, -3.4, -3.4])
    ctx, model = Context(0), to_gpu_model(P)
    cfg = dict(tile_w=tile[0], tile_h=tile[1])
    abi.gs_set_eval_counting(ctx.handle, True)
    images = gpu_render(ctx, model, cam, pose, **cfg)
    st = ctx.stats()
    abi.gs_set_eval_counting(ctx.handle, False)
    R64, t64 = pose.R.astype(np.float64), pose.t.astype(np.float64)
    o = R.render(oracle_params(P), 1, cam, R64, t64, prefilter=True)
    m = R.decision_margins(P, 1, cam, R64, t64)
    near = int((m["pixel"] <= 1e-4).sum())
    for name, a in zip(("color", "depth", "alpha"), images):
        b = o[name].detach().numpy()
        mg = np.broadcast_to(m["pixel"].reshape(b.shape[-2:]), b.shape)
        compare(name, a, b, 1e-4, 1e-6, 1e-4, 3 * max(1, near), None, margins=mg)
    assert abs(st["evals_blended"] - R.gaussian_pixel_evals(o)) <= max(1, near)
    assert st["evals_blended"] > 3000 and st["evals_tiled"] <= 4 * st["evals_blended"], st
    wc, wd = (rng.standard_normal(s).astype(np.float32) for s in ((3, h, w), (h, w)))
    g = gpu_backward(ctx, model, cam, pose, wc, wd, None, **cfg)
    jj, ii = np.meshgrid(np.arange(h), np.arange(w), indexing="ij")
    og, _ = R.weighted_pixel_gradients(P, 1, cam, R64, t64, np.stack([ii.ravel(), jj.ravel()], 1),
                                       wc.reshape(3, -1).astype(np.float64), wd.ravel().astype(np.float64), prefilter=True)
    check_grad_arrays(g, og, m, flip_gaussians=near)
    ctx.close()
