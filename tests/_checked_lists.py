"""Renders maps of long tile lists through one build of the library and saves the images, for
tests/test_gpu_checked_lists.py.

usage: python -m tests._checked_lists {normal|checked} OUT.npz

The cases, with the routes that tests/test_gpu_cut_rules.py checks: lists cut once, lists cut three
times with the open tiles' gathered whole, a few long lists binned in full; and a small map at an
odd size.  gs_sync_status raises if a kernel met an index out of bounds."""
import os
import sys

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def scenes():
    from synth import workloads
    from synth.scene import Camera, look_at
    pose = look_at([0.1, 0.2, -0.1], [0.7, 3.0, 0.2])
    cam = Camera(60.0, 60.0, 32.0, 24.0, 61, 47)
    P = workloads.random_gaussians(np.random.default_rng(75), 6000, cam, pose, 0, z_range=(1.5, 4.0), log_scale_range=(1.0, 1.5))
    P["opacity_logits"][:] = 2.0
    yield "cut", cam, pose, P
    cam = Camera(100.0, 100.0, 64.0, 64.0, 128, 128)
    P = workloads.random_gaussians(np.random.default_rng(12), 200_000, cam, pose, 0, z_range=(2.0, 3.0), log_scale_range=(-2.7, -2.5))
    pc = P["means"].astype(np.float64) @ pose.R.astype(np.float64).T + pose.t.astype(np.float64)
    P["opacity_logits"][:] = np.where(pc[:, 0] / pc[:, 2] * cam.fx + cam.cx > 26.0, 2.0, -5.2)
    yield "gathered", cam, pose, P
    cam, rng = Camera(70.0, 70.0, 60.0, 45.0, 123, 90), np.random.default_rng(11)
    P = workloads.random_gaussians(rng, 8000, cam, pose, 1, z_range=(1.5, 4.0), sh_rest_std=0.1)
    P["means"][:6000] = (np.array([0.6, 2.6, 0.15]) + np.array([0.05, 0.4, 0.05]) * rng.standard_normal((6000, 3))).astype(np.float32)
    P["log_scales"][:6000] = rng.uniform(-2.0, -1.6, (6000, 3))
    P["opacity_logits"][:6000] = -2.0
    yield "in_full", cam, pose, P
    cam = Camera(150.0, 150.0, 166.5, 38.5, 333, 77)
    yield "odd", cam, pose, workloads.random_gaussians(np.random.default_rng(72), 3000, cam, pose, 1, sh_rest_std=0.1)


def main():
    which, out_path = sys.argv[1], sys.argv[2]
    from paper_2408_12677_gb300 import abi
    abi.load(abi.CHECKED_LIB_PATH if which == "checked" else abi.LIB_PATH)
    from paper_2408_12677_gb300.torch_api import Context
    from tests._util import gpu_render, to_gpu_model
    ctx, out = Context(0), {"checked": np.array(abi.gs_bounds_checked())}
    for name, cam, pose, P in scenes():
        abi.gs_set_profiling(ctx.handle, True)
        images = gpu_render(ctx, to_gpu_model(P), cam, pose)
        stages = abi.gs_profile_read(ctx.handle)
        abi.gs_set_profiling(ctx.handle, False)
        for k, a in zip(("color", "depth", "alpha"), images):
            out[f"{name}_{k}"] = a
        out[f"{name}_route"] = np.array([stages["raster_fwd"][1], stages["ranges"][1]])
        abi.gs_sync_status(ctx.handle)
    np.savez(out_path, **out)


if __name__ == "__main__":
    main()
