"""A Gaussian whose opacity is NaN is drawn with the clamp opacity (0.99) over
its 3-sigma support and nowhere else, and its opacity takes no gradient: pixels
outside the support equal the render without it bit for bit, inside it the rest
of the map is seen through 0.01, and the other Gaussians' gradients are those
of that image.  The Gaussian is the nearest one and the map too thin for a pixel
to stop, so the expected image and gradients follow from a render without it
(about 20 blends and float32 atomics: 1e-5 of an image of values up to 1 and of
the gradients' norm).  Sizes with one, two and four pixels per lane."""
import numpy as np
import pytest
import torch

from synth import workloads
from synth.scene import Camera, look_at
from tests._util import ensure_built, gpu_backward, gpu_render, to_gpu_model

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w,h", [(61, 47), (333, 221), (637, 479)])
def test_nan_opacity_stays_within_its_support(w, h):
    ensure_built()
    from paper_2408_12677_gb300.torch_api import Context
    cam = Camera(0.8 * w, 0.8 * w, w / 2, h / 2, w, h)
    pose = look_at([0.1, 0.2, -0.1], [0.7, 3.0, 0.2])
    rng = np.random.default_rng(6)
    P = workloads.random_gaussians(rng, 300, cam, pose, 0, z_range=(1.5, 4.0), log_scale_range=(-4.0, -2.5))
    P["opacity_logits"][:] = -2.0
    z, s = 1.0, 0.05  # the NaN one: isotropic, on the optical axis
    axis = np.array(pose.R, np.float64)[2] * z - np.array(pose.R, np.float64).T @ np.array(pose.t, np.float64)
    P["means"][0], P["log_scales"][0], P["sh"][0] = axis.astype(np.float32), np.log(s), 0.0  # colour 0.5
    up = [rng.standard_normal(a).astype(np.float32) for a in ((3, h, w), (h, w))]
    ctx, got = Context(0), []
    for logit in (np.nan, -np.inf):
        P["opacity_logits"][0] = logit
        model = to_gpu_model(P)
        images = gpu_render(ctx, model, cam, pose)
        got.append((images, gpu_backward(ctx, model, cam, pose, *up, None)))
        up = [u * np.where(got[0][0][2] > 0.9899, np.float32(0.01), np.float32(1.0)) for u in up]
    (col, dep, alp), grads = got[0]
    (rcol, rdep, ralp), rgrads = got[1]
    assert ralp.max() < 0.95
    i, j = np.meshgrid(np.arange(w) + 0.5 - cam.cx, np.arange(h) + 0.5 - cam.cy)
    q = (i * i + j * j) / ((cam.fx * s / z) ** 2 + 0.3)
    inside = alp > 0.9899
    assert np.array_equal(inside[abs(q - 9) > 1e-3], (q <= 9)[abs(q - 9) > 1e-3]) and inside.sum() > 50
    for a, b, front in ((col, rcol, 0.5), (dep, rdep, z), (alp, ralp, 1.0)):
        assert np.array_equal(a[..., ~inside], b[..., ~inside])
        assert np.abs(a - (0.99 * front + 0.01 * b))[..., inside].max() <= 1e-5
    for k in ("means", "log_scales", "quats", "opacity_logits", "sh"):
        a, b = grads[k][1:], rgrads[k][1:]
        assert np.isfinite(a).all() and np.linalg.norm(a - b) <= 1e-5 * np.linalg.norm(b), k
    ctx.close()
