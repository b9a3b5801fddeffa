"""Lists longer than the per-tile sort holds, binned by their nearest entries
(csrc/prefix.cu), against the oracle: pixels that stop within the first
attempt's lists, only within the longest ones the sort holds, and never (all
of the list).  Images, gradients, the blended-pair counter, the full
lists' ranges, and the training step's loss and valid-depth count after
repeated attempts; two views of one map.  Tolerances as in test_gpu_render and
test_gpu_grad."""
import numpy as np
import pytest
import torch

from oracle import render as R
from synth import workloads
from synth.scene import Camera, look_at
from tests._util import compare, ensure_built, gpu_backward, gpu_render, oracle_params, to_gpu_model
from tests.test_gpu_grad import check_grad_arrays

pytestmark = pytest.mark.gpu

CAM = Camera(60.0, 60.0, 32.0, 24.0, 61, 47)
POSE = look_at([0.1, 0.2, -0.1], [0.7, 3.0, 0.2])


def _scene(kind, n=6000):
    """Gaussians over the whole image ("stop": opaque, "faint": a pixel needs a
    few hundred of them) or on one spot of it ("never": most pixels see none)."""
    rng = np.random.default_rng(11)
    P = workloads.random_gaussians(rng, n, CAM, POSE, 1, z_range=(1.5, 4.0), sh_rest_std=0.1)
    if kind == "never":
        mid = np.array([0.6, 2.6, 0.15], np.float32)
        P["means"] = (mid + np.array([0.03, 0.4, 0.03]) * rng.standard_normal((n, 3))).astype(np.float32)
        P["log_scales"][:] = rng.uniform(-4.0, -3.0, (n, 3))
        P["opacity_logits"][:] = -3.0
    else:
        P["log_scales"][:] = rng.uniform(1.0, 1.5, (n, 3))
        P["opacity_logits"][:] = 2.0 if kind == "stop" else -3.9
    return P


@pytest.mark.parametrize("kind", ["stop", "faint", "never"])
def test_cut_lists_match_the_oracle(kind):
    ensure_built()
    from paper_2408_12677_gb300 import abi
    from paper_2408_12677_gb300.torch_api import Context, Trainer
    P = _scene(kind)
    ctx = Context(0)
    h = ctx.handle
    model = to_gpu_model(P)
    abi.gs_set_eval_counting(h, True)
    col, dep, alp = gpu_render(ctx, model, CAM, POSE)
    st = ctx.stats()
    abi.gs_set_eval_counting(h, False)
    ranges = torch.empty((st["n_tiles"], 2), dtype=torch.int32, device="cuda")
    abi.gs_get_tile_ranges(h, ranges)
    lens = (ranges[:, 1] - ranges[:, 0]).cpu().numpy()
    assert lens.sum() == st["n_pairs"] and lens.max() > 4096
    with pytest.raises(abi.GsError):
        abi.gs_get_tile_order(h, torch.empty(st["n_tiles"], dtype=torch.int32, device="cuda"))
    R64, t64 = POSE.R.astype(np.float64), POSE.t.astype(np.float64)
    o = R.render(oracle_params(P), 1, CAM, R64, t64, prefilter=True)
    m = R.decision_margins(P, 1, CAM, R64, t64)
    mk = dict(margins=m["pixel"], kinds=m["pixel_kind"])
    near = int((m["pixel"] <= 1e-4).sum())
    for c in range(3):
        compare(f"color{c}", col[c], o["color"][c].detach().numpy(), 1e-4, 1e-6, 1e-4, max(1, near), None, **mk)
    compare("depth", dep, o["depth"].detach().numpy(), 1e-4, 1e-6, 1e-4, max(1, near), None, **mk)
    compare("alpha", alp, o["alpha"].detach().numpy(), 1e-4, 1e-6, 1e-4, max(1, near), None, **mk)
    # (a stop that flips by float32 rounding adds or drops one blend of a pixel)
    assert abs(st["evals_blended"] - R.gaussian_pixel_evals(o)) <= max(1, near)
    rng = np.random.default_rng(2)
    wc, wd = (rng.standard_normal(s).astype(np.float32) for s in ((3, CAM.height, CAM.width), (CAM.height, CAM.width)))
    gpu_render(ctx, model, CAM, POSE)
    g = gpu_backward(ctx, model, CAM, POSE, wc, wd, None)
    jj, ii = np.meshgrid(np.arange(CAM.height), np.arange(CAM.width), indexing="ij")
    og, _ = R.weighted_pixel_gradients(P, 1, CAM, R64, t64, np.stack([ii.ravel(), jj.ravel()], 1),
                                       wc.reshape(3, -1).astype(np.float64), wd.ravel().astype(np.float64), prefilter=True)
    check_grad_arrays(g, og, m, flip_gaussians=near)
    # the training step in one call (loss and valid depths taken in the forward pass) and as three
    rgb = torch.as_tensor(rng.uniform(0, 1, wc.shape).astype(np.float32), device="cuda")
    dep = torch.as_tensor((rng.uniform(0.5, 4.0, wd.shape) * (rng.uniform(size=wd.shape) < 0.7)).astype(np.float32), device="cuda")
    out = []
    for one_call in (True, False):
        tr = Trainer(to_gpu_model(P), CAM, POSE.R, POSE.t, ctx=ctx, one_call=one_call)
        tr.step(rgb, dep)
        out.append((float(tr.loss), tr.model.m.cpu().numpy()))
    assert abs(out[0][0] - out[1][0]) <= 1e-6 * abs(out[1][0])
    assert np.linalg.norm(out[0][1] - out[1][1]) <= 1e-5 * np.linalg.norm(out[1][1])
    ctx.close()


def test_cut_lists_of_two_views():
    ensure_built()
    from paper_2408_12677_gb300.torch_api import BatchedTrainer, Context
    P = _scene("stop")
    views = [(CAM, POSE.R, POSE.t)]
    other = Camera(45.0, 45.0, 20.0, 15.0, 40, 29)
    pose = look_at([0.3, -0.1, 0.1], [0.7, 3.0, 0.2])
    views.append((other, pose.R, pose.t))
    ctx = Context(0)
    tr = BatchedTrainer(to_gpu_model(P), views, ctx=ctx)
    tr.forward()
    for k, (cam, Rm, t) in enumerate(views):  # images of a batch are the single views', bit for bit
        one = gpu_render(ctx, tr.model, cam, type(POSE)(Rm, t))
        for a, b in zip((tr.color[k], tr.depth[k], tr.alpha[k]), one):
            assert np.array_equal(a.cpu().numpy(), b)
    ctx.close()
