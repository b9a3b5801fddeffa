"""Which binning a sync-mode pass with a list of more than 4096 entries takes, by the stages it
times (only the full binning has a ranges stage), and that the results agree: images bit for
bit, gradients to the order of float32 atomics (1e-5 of the norm)."""
import numpy as np
import pytest
import torch

from oracle import render as R
from synth import workloads
from synth.scene import Camera, look_at
from tests._util import compare, ensure_built, gpu_backward, gpu_render, oracle_params, to_gpu_model
from tests.test_gpu_grad import check_grad_arrays

pytestmark = pytest.mark.gpu

POSE = look_at([0.1, 0.2, -0.1], [0.7, 3.0, 0.2])


def _pass(ctx, model, cam):
    """Images, gradients, and how often the pass rastered and binned in full."""
    from paper_2408_12677_gb300 import abi
    abi.gs_set_profiling(ctx.handle, True)
    images = gpu_render(ctx, model, cam, POSE)
    stages = abi.gs_profile_read(ctx.handle)
    abi.gs_set_profiling(ctx.handle, False)
    rng = np.random.default_rng(2)
    wc, wd = (rng.standard_normal(s).astype(np.float32) for s in ((3, cam.height, cam.width), (cam.height, cam.width)))
    return images, gpu_backward(ctx, model, cam, POSE, wc, wd, None), (stages["raster_fwd"][1], stages["ranges"][1])


def test_few_long_lists_are_binned_in_full():
    """Some lists over 4096 in a scene of a mean of about 1000: one pass over the full lists, against the oracle."""
    ensure_built()
    from paper_2408_12677_gb300 import abi
    from paper_2408_12677_gb300.torch_api import Context
    cam = Camera(70.0, 70.0, 60.0, 45.0, 123, 90)
    rng = np.random.default_rng(11)
    n = 8000
    P = workloads.random_gaussians(rng, n, cam, POSE, 1, z_range=(1.5, 4.0), sh_rest_std=0.1)
    P["means"][:6000] = (np.array([0.6, 2.6, 0.15]) + np.array([0.05, 0.4, 0.05]) * rng.standard_normal((6000, 3))).astype(np.float32)
    P["log_scales"][:6000] = rng.uniform(-2.0, -1.6, (6000, 3))
    P["opacity_logits"][:6000] = -2.0
    ctx, model = Context(0), to_gpu_model(P)
    images, g, route = _pass(ctx, model, cam)
    st = ctx.stats()
    ranges = torch.empty((st["n_tiles"], 2), dtype=torch.int32, device="cuda")
    abi.gs_get_tile_ranges(ctx.handle, ranges)
    lens = (ranges[:, 1] - ranges[:, 0]).cpu().numpy()
    assert lens.sum() == st["n_pairs"] and lens.max() > 4096 and 768 <= lens.mean() < 2048, (lens.max(), lens.mean())
    assert route == (1, 1)
    R64, t64 = POSE.R.astype(np.float64), POSE.t.astype(np.float64)
    o = R.render(oracle_params(P), 1, cam, R64, t64, prefilter=True)
    m = R.decision_margins(P, 1, cam, R64, t64)
    near = int((m["pixel"] <= 1e-4).sum())
    for name, a in zip(("color", "depth", "alpha"), images):
        b = o[name].detach().numpy()
        mg = np.broadcast_to(m["pixel"].reshape(b.shape[-2:]), b.shape)
        compare(name, a, b, 1e-4, 1e-6, 1e-4, 3 * max(1, near), None, margins=mg)
    rng = np.random.default_rng(2)
    wc, wd = (rng.standard_normal(s) for s in ((3, cam.height, cam.width), (cam.height, cam.width)))
    jj, ii = np.meshgrid(np.arange(cam.height), np.arange(cam.width), indexing="ij")
    og, _ = R.weighted_pixel_gradients(P, 1, cam, R64, t64, np.stack([ii.ravel(), jj.ravel()], 1),
                                       wc.reshape(3, -1).astype(np.float32).astype(np.float64),
                                       wd.ravel().astype(np.float32).astype(np.float64), prefilter=True)
    check_grad_arrays(g, og, m, flip_gaussians=near)
    ctx.close()


def test_lists_that_no_pixel_ends_are_binned_in_full():
    """200k faint splats, lists of about 5000 that are read to their ends in every tile: after the second attempt the
    pass is binned in full, and the next one at once.  Then a map of which a strip is faint: cut, its open tiles'
    lists gathered, in a fresh context; in full in the first one."""
    ensure_built()
    from paper_2408_12677_gb300.torch_api import Context
    cam = Camera(100.0, 100.0, 64.0, 64.0, 128, 128)
    rng = np.random.default_rng(12)
    n = 200_000
    P = workloads.random_gaussians(rng, n, cam, POSE, 0, z_range=(2.0, 3.0), log_scale_range=(-2.7, -2.5))
    P["opacity_logits"][:] = -5.2
    ctx, faint = Context(0), to_gpu_model(P)
    a, ga, route = _pass(ctx, faint, cam)
    assert route == (3, 1), (route, ctx.stats())
    b, gb, route = _pass(ctx, faint, cam)
    assert route == (1, 1), route
    pc = P["means"].astype(np.float64) @ POSE.R.astype(np.float64).T + POSE.t.astype(np.float64)
    P["opacity_logits"][pc[:, 0] / pc[:, 2] * cam.fx + cam.cx > 26.0] = 2.0
    strip, other = to_gpu_model(P), Context(0)
    c, gc, route = _pass(other, strip, cam)
    assert route == (3, 0), (route, other.stats())
    d, gd, route = _pass(ctx, strip, cam)
    assert route == (1, 1), route
    for x, y, gx, gy in ((a, b, ga, gb), (c, d, gc, gd)):
        for p, q in zip(x, y):
            assert np.array_equal(p, q)
        for k in gx:
            assert np.linalg.norm(gx[k].astype(np.float64) - gy[k]) <= 1e-5 * np.linalg.norm(gy[k].astype(np.float64)), k
    ctx.close()
    other.close()
