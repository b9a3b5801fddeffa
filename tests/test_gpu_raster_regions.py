"""The raster passes' pixels-per-lane variants (1, 2 and 4 pixels, chosen by the
tile count) in every tile shape, at sizes whose borders cut tiles, regions and
blocks: images and gradients against the oracle on the pixels of a sample of
tiles.  A quarter of the Gaussians lie on top of each other in the middle, so
that lists run past the warp's ring of 128 entries, pixels stop early, and
opaque ones reach the 0.99 clamp.  Tolerances as in test_gpu_render and
test_gpu_grad."""
import numpy as np
import pytest

from oracle import render as R
from synth import workloads
from synth.scene import Camera, look_at
from tests._util import compare, ensure_built, gpu_backward, gpu_render, oracle_params, to_gpu_model
from tests.test_gpu_grad import check_grad_arrays

pytestmark = pytest.mark.gpu


def _scene(cam, pose, n=800):
    rng = np.random.default_rng(7)
    P = workloads.random_gaussians(rng, n, cam, pose, 1, log_scale_range=(-4.5, -2.5), sh_rest_std=0.1)
    k = n // 4
    mid = P["means"].mean(0)
    P["means"][:k] = mid + 0.05 * rng.standard_normal((k, 3)).astype(np.float32)
    P["log_scales"][:k] = -2.0
    P["opacity_logits"][:k] = np.where(np.arange(k) % 3 == 0, 6.0, -2.5)
    return P


@pytest.mark.parametrize("tile", [(16, 16), (8, 32), (32, 8)])
@pytest.mark.parametrize("size", [(45, 31), (211, 203), (491, 487)])  # 6 to 14, 175 to 196, 976 to 992 tiles
def test_regions_match_the_oracle(size, tile):
    ensure_built()
    from paper_2408_12677_gb300.torch_api import Context
    W, H = size
    cam = Camera(0.9 * W, 0.9 * W, W / 2.0, H / 2.0, W, H)
    pose = look_at([0.1, 0.2, -0.1], [0.7, 3.0, 0.2])
    P = _scene(cam, pose)
    ctx = Context(0)
    model = to_gpu_model(P)
    cfg = dict(tile_w=tile[0], tile_h=tile[1])
    col, dep, alp = gpu_render(ctx, model, cam, pose, **cfg)
    # the pixels of up to 40 16 x 16 squares: the corners, the middle and random ones
    rng = np.random.default_rng(3)
    nx, ny = -(-W // 16), -(-H // 16)
    pick = {(0, 0), (nx - 1, ny - 1), (nx // 2, ny // 2), (nx - 1, 0)}
    while len(pick) < min(40, nx * ny):
        pick.add((int(rng.integers(nx)), int(rng.integers(ny))))
    px = np.array([(x, y) for tx, ty in sorted(pick) for y in range(16 * ty, min(16 * ty + 16, H))
                   for x in range(16 * tx, min(16 * tx + 16, W))])
    R64, t64 = pose.R.astype(np.float64), pose.t.astype(np.float64)
    o = R.render(oracle_params(P), 1, cam, R64, t64, pixels=px, prefilter=True)
    m = R.decision_margins(P, 1, cam, R64, t64, pixels=px)
    at = (px[:, 1], px[:, 0])
    budget = max(1, int(1e-5 * len(px)))
    mk = dict(margins=m["pixel"], kinds=m["pixel_kind"])
    for c in range(3):
        compare(f"color{c}", col[c][at], o["color"][c].detach().numpy(), 1e-4, 1e-6, 1e-4, budget, None, **mk)
    compare("depth", dep[at], o["depth"].detach().numpy(), 1e-4, 1e-6, 1e-4, budget, None, **mk)
    compare("alpha", alp[at], o["alpha"].detach().numpy(), 1e-4, 1e-6, 1e-4, budget, None, **mk)
    w = [np.zeros((H, W), np.float32) for _ in range(5)]
    for k in w:
        k[at] = rng.standard_normal(len(px)).astype(np.float32)
    wc = np.stack(w[:3])
    g = gpu_backward(ctx, model, cam, pose, wc, w[3], w[4], **cfg)
    og, _ = R.weighted_pixel_gradients(P, 1, cam, R64, t64, px, wc[:, px[:, 1], px[:, 0]].astype(np.float64),
                                       w[3][at].astype(np.float64), w[4][at].astype(np.float64), prefilter=True)
    check_grad_arrays(g, og, m)
    ctx.close()
