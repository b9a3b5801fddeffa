"""Benchmark: fwd + bwd + Adam iterations of the Gaussian map optimisation
(GSFusion's online optimisation, Sec. III-B.3) on one synthetic view at
1200x680 with about 300k quadtree-seeded Gaussians, SH degree 3, float32.

One step = gs_train_step on the same view (inputs resident in HBM): the
forward pass (projection, binning, compositing) with the L1 loss in its
epilogue, then the backward pass fused with the Adam update, replayed as one
CUDA graph.  Prints one JSON line; besides the single-view numbers it carries
the measured ALU peaks of the raster passes' roofline, the clocks sampled
during the timed region, the FP64 oracle timed on the host cores
(cpu_baseline) and a compact batched-vs-view-by-view comparison of the
8-view multi-view iteration (``multi_view``).

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

--gpus N > 1 runs N independent replicas under torchrun (one process per GPU,
no collective on the data path); the value is the sum over replicas.
--impl reference times the FP64 CPU oracle on whole iterations of the same
workload (the only other place this script runs the oracle).
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "fwd+bwd+Adam iterations/sec and Gaussian-pixel evals/sec at 1 GB300, % HBM roofline"
WORKLOAD = "single_view 1200x680, ~300k quadtree-seeded Gaussians, SH degree 3, fp32, loss 0.8 L1(rgb) + 0.2 L1(depth)"


def load_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        d = json.load(open(p))
        return d.get("hbm_gbs", 6800.0), "measured"
    return 6800.0, "fallback"


# ---------------------------------------------------------------------------
# algorithmic traffic and work per launch
# ---------------------------------------------------------------------------
def algorithmic_bytes(n, deg, pairs, npx, n_tiles):
    """Bytes each stage must move at least (one launch, single view)."""
    K = (deg + 1) ** 2
    pbytes = 4 * (11 + 3 * K)  # parameters of one Gaussian (236 B at degree 3)
    rec = 48                    # projected record
    return {
        "project_fwd": n * (pbytes + rec + 4 + 8 + 4),        # params in; record, depth key, rect, count out
        "duplicate": n * 2 * 12 + pairs * 4 + n_tiles * 12,   # rects + counts read twice; ids out; tile tables
        "pair_sort": pairs * 12,                              # ids in, depth keys gathered, ids out
        "raster_fwd": pairs * (4 + rec) + npx * 28,           # ids + records in; rgb, depth, alpha, T, last out
        "loss": npx * 48,                                     # rgb, depth, targets in; image gradients out
        "raster_bwd": pairs * (4 + rec) + npx * 24 + n * rec, # ids + records, pixel state + grads in; records out
        "project_bwd": n * (pbytes + rec + 2 * pbytes + 3 * pbytes),  # fused with Adam: p, record, m, v in; p, m, v out
        "adam": 0,                                            # folded into project_bwd (fused path)
    }


# algorithmic FP32 operations per blended (pixel, Gaussian) pair: the
# exponent and opacity test (13), then the blend (14) or the gradient (55)
FLOPS_PER_BLEND = {"raster_fwd": 27, "raster_bwd": 68}


def alu_roofline(dom, e_blend, dom_ms, alu):
    """ALU roofline of a raster pass: algorithmic FP32 flops per blended pair
    x blended pairs per launch over the launch time, against the FP32 FMA rate
    measured by gs_measure_alu_peaks on this GPU."""
    flops = e_blend * FLOPS_PER_BLEND[dom]
    achieved = flops / (dom_ms * 1e-3) / 1e12 if dom_ms else 0.0
    peak = alu["fma_tflops"]
    return {"kernel": dom, "bound": "alu", "achieved": achieved, "peak": peak, "unit": "TFLOP/s",
            "frac": achieved / peak if peak else None, "traffic": load_traffic(dom),
            "peak_kind": f"measured: FP32 FMA probe (gs_measure_alu_peaks) at {alu['fma_sm_mhz']:.0f} MHz",
            "alg_flops_per_launch": flops, "ms_per_launch": dom_ms}


class ClockSampler:
    """nvidia-smi clocks during the timed region (median SM clock, reasons)."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu: int):
        self.gpu = gpu
        self.proc = None
        self.path = None

    def start(self):
        """Starts sampling every 50 ms and returns once the first sample is
        in, so that the samples after it fall in the region timed next (the
        first one is dropped)."""
        self.skip = 0
        try:
            fd, self.path = tempfile.mkstemp(suffix=".csv")
            os.close(fd)
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "50"],
                                         stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None
            return
        t_end = time.perf_counter() + 3.0
        while time.perf_counter() < t_end and self.proc.poll() is None:
            with open(self.path) as f:
                n = sum(1 for line in f if line.count(",") >= 8)
            if n:
                self.skip = n
                break
            time.sleep(0.01)

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        rows = []
        for line in open(self.path):
            f = [x.strip() for x in line.split(",")]
            if len(f) >= 9:
                rows.append(f)
        os.unlink(self.path)
        rows = rows[self.skip:]  # taken before the timed region
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4) if r[5 + i].lower() == "active"})
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(rows)}


# ---------------------------------------------------------------------------
# our arm
# ---------------------------------------------------------------------------
def run_ours(args, rank, world, local_rank):
    import numpy as np
    import torch

    from paper_2408_12677_gb300 import abi
    from paper_2408_12677_gb300.torch_api import Context, GaussianModel, Trainer
    from synth import workloads

    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    abi.load()
    w = workloads.single_view()
    v = w.views[0]
    H, W = v.cam.height, v.cam.width
    ctx = Context(local_rank)
    model = GaussianModel(w.params, device=dev)
    tr = Trainer(model, v.cam, v.pose.R, v.pose.t, ctx=ctx, device=local_rank)
    trgb = torch.as_tensor(v.target_rgb, device=dev)
    tdep = torch.as_tensor(v.target_depth, device=dev)
    stream = torch.cuda.current_stream(dev)

    # issue rates of the FP32 and MUFU pipes (the raster passes' ALU roofline)
    alu = abi.gs_measure_alu_peaks(local_rank, 50000)

    # warm-up
    for _ in range(args.warmup):
        tr.step(trgb, tdep)
    torch.cuda.synchronize(dev)

    # counts per iteration (pairs, evals) from one counted iteration
    abi.gs_set_eval_counting(ctx.handle, True)
    tr.step(trgb, tdep)
    st = ctx.stats()
    abi.gs_set_eval_counting(ctx.handle, False)
    pairs, e_blend, e_tiled = st["n_pairs"], st["evals_blended"], st["evals_tiled"]

    def barrier():
        if world > 1:
            import torch.distributed as dist
            dist.barrier()
        torch.cuda.synchronize(dev)

    # one iteration = one replay of a CUDA graph of fwd + loss + bwd + Adam
    # (no-sync mode: pair buffers reserved, Adam step counted on the device)
    tr.capture(trgb, tdep)
    for _ in range(args.warmup):
        tr.replay()
    torch.cuda.synchronize(dev)

    # The map trains while it is timed (the iterations are the online
    # optimisation, so its Gaussians and their pairs grow from step to step).
    # The timed region, the per-stage run and the end-to-end run each start
    # from this state (parameters, Adam moments and step restored), so all
    # three measure the same K iterations.
    snap = trainer_snapshot(tr)

    def restore():
        trainer_restore(tr, snap)

    # timed region: K graph replays, CUDA events on the launch stream.  It is
    # repeated (the map restored between repeats) until the sampled region
    # lasts at least 0.5 s, so that the clock sampler (50 ms period) sees it;
    # ms_per_step is the median repeat.
    clocks = ClockSampler(local_rank)
    clocks.start()
    reps = []
    t_region = time.perf_counter()
    while True:
        restore()
        barrier()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(args.steps):
            tr.replay()
        e1.record(stream)
        barrier()
        reps.append(e0.elapsed_time(e1))
        if time.perf_counter() - t_region >= 0.5 or len(reps) >= 200:
            break
    clk = clocks.stop()
    ms_total = statistics.median(reps)
    tr.check_capacity()
    loss_end = float(tr.loss)

    # per-stage device times: the same K iterations run eagerly (same kernels,
    # same no-sync mode) with the library's CUDA event pairs around each stage
    restore()
    launches0 = ctx.stats()["kernel_launches"]
    abi.gs_set_profiling(ctx.handle, True)
    p0 = torch.cuda.Event(enable_timing=True)
    p1 = torch.cuda.Event(enable_timing=True)
    p0.record(stream)
    for _ in range(args.steps):
        tr._step_device_counter(trgb, tdep)
    p1.record(stream)
    stages = abi.gs_profile_read(ctx.handle)
    abi.gs_set_profiling(ctx.handle, False)
    ms_eager = p0.elapsed_time(p1)
    launches = ctx.stats()["kernel_launches"] - launches0

    # end to end through the public API with host buffers: per step, H2D of
    # that step's target RGB-D frame from pinned memory, the iteration and a
    # D2H copy of the loss.  First choice: Trainer.capture_from_host, two
    # graphs that each run one iteration on one target buffer while a forked
    # branch uploads the next step's frame into the other (one launch call
    # per step; the first frame is uploaded inside the timed region before
    # the first replay).  Fallback if the copies cannot be captured: the same
    # double buffering with a copy stream and events.
    h_rgb = torch.from_numpy(v.target_rgb).pin_memory()
    h_dep = torch.from_numpy(v.target_depth).pin_memory()
    h_loss = torch.empty(1).pin_memory()
    restore()
    bufs = [(trgb, tdep), (trgb.clone(), tdep.clone())]
    e2e_mode = "two captured graphs: iteration on one buffer + upload of the next frame into the other + D2H loss"
    try:
        g_h2h = tr.capture_from_host(h_rgb, h_dep, h_loss, bufs)
        torch.cuda.synchronize(dev)
    except Exception as exc:  # pragma: no cover - depends on the torch build
        g_h2h = None
        e2e_mode = f"double-buffered streams (graph capture of the copies failed: {type(exc).__name__})"
    if g_h2h is not None:
        barrier()
        f0 = torch.cuda.Event(enable_timing=True)
        f1 = torch.cuda.Event(enable_timing=True)
        t_host0 = time.perf_counter()
        f0.record(stream)
        bufs[0][0].copy_(h_rgb, non_blocking=True)
        bufs[0][1].copy_(h_dep, non_blocking=True)
        for k in range(args.steps):
            g_h2h[k % 2].replay()
            tr.step_count += 1
        f1.record(stream)
        barrier()
    else:
        graphs = [tr.graph, tr.capture(*bufs[1])]
        copy_stream = torch.cuda.Stream(dev)
        ev_copied = [torch.cuda.Event(), torch.cuda.Event()]
        ev_done = [torch.cuda.Event(), torch.cuda.Event()]

        def upload(b):
            bufs[b][0].copy_(h_rgb, non_blocking=True)
            bufs[b][1].copy_(h_dep, non_blocking=True)
            ev_copied[b].record(copy_stream)

        barrier()
        f0 = torch.cuda.Event(enable_timing=True)
        f1 = torch.cuda.Event(enable_timing=True)
        t_host0 = time.perf_counter()
        f0.record(stream)
        copy_stream.wait_event(f0)
        with torch.cuda.stream(copy_stream):
            upload(0)
        for k in range(args.steps):
            b = k % 2
            stream.wait_event(ev_copied[b])
            graphs[b].replay()
            tr.step_count += 1
            h_loss.copy_(tr.loss, non_blocking=True)
            ev_done[b].record(stream)
            if k + 1 < args.steps:
                with torch.cuda.stream(copy_stream):
                    if k >= 1:
                        copy_stream.wait_event(ev_done[1 - b])  # step k - 1 read buffer 1 - b
                    upload(1 - b)
        f1.record(stream)
        barrier()
    e2e_ms = f0.elapsed_time(f1)
    e2e_host_s = time.perf_counter() - t_host0
    h2d = h_rgb.numel() * 4 + h_dep.numel() * 4

    ms_total, e2e_ms = max_over_ranks([ms_total, e2e_ms], world)

    # roofline of the dominant kernel (per launch, CUDA events over the timed region)
    npx = H * W
    n_tiles = ((W + 15) // 16) * ((H + 15) // 16)
    alg = algorithmic_bytes(w.n, w.sh_degree, pairs, npx, n_tiles)
    per_stage = {k: {"ms_per_launch": (ms / c if c else 0.0), "launches": c, "share": None}
                 for k, (ms, c) in stages.items()}
    tot_stage = sum(ms for ms, _ in stages.values())
    for k, (ms, c) in stages.items():
        per_stage[k]["share"] = ms / tot_stage if tot_stage else None
    dom = max(stages, key=lambda k: stages[k][0])
    hbm_peak, peak_kind = load_peaks()
    dom_ms = per_stage[dom]["ms_per_launch"]
    traffic = load_traffic(dom)
    if dom in FLOPS_PER_BLEND:
        roof = alu_roofline(dom, e_blend, dom_ms, alu)
    else:
        achieved = alg[dom] / (dom_ms * 1e-3) / 1e9 if dom_ms else 0.0
        roof = {"kernel": dom, "bound": "hbm", "achieved": achieved, "peak": hbm_peak, "unit": "GB/s",
                "frac": achieved / hbm_peak, "traffic": traffic, "peak_kind": peak_kind,
                "alg_bytes_per_launch": alg[dom], "ms_per_launch": dom_ms}
    it_s = whole_job_rate(args.steps, world, ms_total)
    b_alg_iter = sum(alg.values())
    out = {
        "metric": METRIC, "value": it_s, "unit": "it/s", "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms_total / args.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": WORKLOAD, "n_gaussians": w.n, "width": W, "height": H, "sh_degree": w.sh_degree,
                   "tile": "16x16", "pairs": pairs, "parallelism": f"replicas{world}",
                   "timing": "CUDA graph replay per step; per-stage times from an eager profiled run of the same steps",
                   "l2": "no flush: per-step working set (params, grads, Adam moments, pairs, images) > 129 MB L2"},
        "gaussian_pixel_evals_per_s": e_blend * it_s, "evals_blended_per_iter": e_blend,
        "evals_tiled_per_iter": e_tiled,
        "hbm_roofline_frac_iteration": b_alg_iter * it_s / world / (hbm_peak * 1e9),
        "alg_bytes_per_iter": b_alg_iter,
        "roofline": roof,
        "stages": per_stage,
        "e2e": {"value": whole_job_rate(args.steps, world, e2e_ms), "unit": "it/s", "h2d_bytes_per_step": h2d,
                "d2h_bytes_per_step": 4, "host_wall_s": e2e_host_s, "mode": e2e_mode},
        "gpu_launches": launches,
        "eager_ms_per_step": ms_eager / args.steps,
        "clocks": clk,
        "timed_repeats": {"count": len(reps), "ms": reps, "note": "K steps each, map restored between repeats; "
                          "ms_per_step from the median"},
        "alu_peaks": {"fp32_fma_tflops": alu["fma_tflops"], "mufu_ex2_gops": alu["ex2_gops"],
                      "fma_per_sm_clk": alu["fma_per_sm_clk"], "ex2_per_sm_clk": alu["ex2_per_sm_clk"],
                      "sm_mhz": alu["fma_sm_mhz"], "num_sms": alu["num_sms"]},
        "loss_end": loss_end,
    }
    return out


def run_scale_stress(args, rank, world, local_rank):
    """The scale-stress configuration: 1752x1168 (fx 1200), 1M quadtree-seeded
    Gaussians of which 20% are large (log-scale U[-1, 0], logit +2), SH
    degree 3: about 1.1e9 (tile, Gaussian) pairs, every tile list beyond the
    per-tile sort, so the lists are cut to their nearest entries, whose counts
    the forward pass reads back (sync mode: the iteration runs eagerly, one
    gs_train_step per step).  Reported on Gaussian-pixel evals/s (blended
    pairs per second) like the single view, which it is compared with."""
    import torch

    from paper_2408_12677_gb300 import abi
    from paper_2408_12677_gb300.torch_api import Context, GaussianModel, Trainer
    from synth import workloads

    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    abi.load()
    t_gen = time.perf_counter()
    w = workloads.scale_stress()
    t_gen = time.perf_counter() - t_gen
    v = w.views[0]
    ctx = Context(local_rank)
    tr = Trainer(GaussianModel(w.params, device=dev), v.cam, v.pose.R, v.pose.t, ctx=ctx, device=local_rank)
    trgb = torch.as_tensor(v.target_rgb, device=dev)
    tdep = torch.as_tensor(v.target_depth, device=dev)
    stream = torch.cuda.current_stream(dev)
    alu = abi.gs_measure_alu_peaks(local_rank, 50000)
    for _ in range(args.warmup):
        tr.step(trgb, tdep)
    abi.gs_set_eval_counting(ctx.handle, True)
    tr.step(trgb, tdep)
    st = ctx.stats()
    abi.gs_set_eval_counting(ctx.handle, False)
    pairs, e_blend, e_tiled = st["n_pairs"], st["evals_blended"], st["evals_tiled"]
    snap = trainer_snapshot(tr)
    clocks = ClockSampler(local_rank)
    clocks.start()
    torch.cuda.synchronize(dev)
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(args.steps):
        tr.step(trgb, tdep)
    e1.record(stream)
    torch.cuda.synchronize(dev)
    clk = clocks.stop()
    ms = e0.elapsed_time(e1)
    trainer_restore(tr, snap)
    launches0 = ctx.stats()["kernel_launches"]
    abi.gs_set_profiling(ctx.handle, True)
    for _ in range(args.steps):
        tr.step(trgb, tdep)
    stages = abi.gs_profile_read(ctx.handle)
    abi.gs_set_profiling(ctx.handle, False)
    launches = ctx.stats()["kernel_launches"] - launches0
    ms, = max_over_ranks([ms], world)
    it_s = whole_job_rate(args.steps, world, ms)
    per_stage = {k: {"ms_per_launch": (t / c if c else 0.0), "launches": c} for k, (t, c) in stages.items()}
    dom = max(stages, key=lambda k: stages[k][0])
    dom_ms = per_stage[dom]["ms_per_launch"]
    if dom in FLOPS_PER_BLEND:
        roof = alu_roofline(dom, e_blend, dom_ms, alu)
    else:
        n_tiles = ((v.cam.width + 15) // 16) * ((v.cam.height + 15) // 16)
        alg = algorithmic_bytes(w.n, w.sh_degree, pairs, v.cam.width * v.cam.height, n_tiles)
        alg["pair_sort"] = 256 * n_tiles * 4 * 2  # the ids of lists cut to about 256 entries, read + write
        alg["duplicate"] = w.n * 12 + 256 * n_tiles * 4
        hbm_peak, peak_kind = load_peaks()
        achieved = alg.get(dom, 0) / (dom_ms * 1e-3) / 1e9 if dom_ms else 0.0
        roof = {"kernel": dom, "bound": "hbm", "achieved": achieved, "peak": hbm_peak, "unit": "GB/s",
                "frac": achieved / hbm_peak, "traffic": None, "peak_kind": peak_kind,
                "alg_bytes_per_launch": alg.get(dom), "ms_per_launch": dom_ms}
    return {
        "metric": METRIC, "value": it_s, "unit": "it/s", "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms / args.steps, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": "scale_stress 1752x1168 (fx 1200), 1M quadtree-seeded Gaussians, 20% large "
                               "(log-scale U[-1,0], logit +2), SH degree 3, fp32, loss 0.8 L1(rgb) + 0.2 L1(depth)",
                   "n_gaussians": w.n, "width": v.cam.width, "height": v.cam.height, "tile": "16x16",
                   "pairs": pairs, "binning": "every tile list > 4096, cut to its nearest entries", "parallelism": f"replicas{world}",
                   "timing": "eager gs_train_step per step (sync mode: one host read of the pair count)",
                   "l2": "no flush: per-step working set (1.4 GB of parameters and moments) > 129 MB L2", "host_generation_s": t_gen},
        "gaussian_pixel_evals_per_s": e_blend * it_s, "evals_blended_per_iter": e_blend,
        "evals_tiled_per_iter": e_tiled,
        "roofline": roof, "stages": per_stage,
        "e2e": None, "gpu_launches": launches, "clocks": clk,
        "alu_peaks": {"fp32_fma_tflops": alu["fma_tflops"], "mufu_ex2_gops": alu["ex2_gops"]},
    }


def run_profile_driver(args, local_rank):
    """``--profile-iterations N``: N eager gs_train_step iterations of the
    single-view workload, for profiler captures of single launches: the
    first in sync mode, the others in the no-sync mode of the bench's graph
    (the same kernels and launch configuration, no graph, no timing loop)."""
    import torch

    from paper_2408_12677_gb300 import abi
    from paper_2408_12677_gb300.torch_api import Context, GaussianModel, Trainer
    from synth import workloads
    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    abi.load()
    w = workloads.single_view()
    v = w.views[0]
    tr = Trainer(GaussianModel(w.params, device=dev), v.cam, v.pose.R, v.pose.t, ctx=Context(local_rank),
                 device=local_rank)
    trgb = torch.as_tensor(v.target_rgb, device=dev)
    tdep = torch.as_tensor(v.target_depth, device=dev)
    tr.step(trgb, tdep)  # sync mode: counting-scatter binning, sizes the buffers
    torch.cuda.synchronize(dev)
    # the rest as the graph replays run them: no-sync mode, bucket binning
    h = tr.ctx.handle
    abi.gs_ctx_reserve(h, tr.model.n, v.cam.width * v.cam.height, int(abi.gs_get_stats(h)["n_pairs"] * 1.5) + 4096)
    abi.gs_ctx_set_sync(h, False)
    for _ in range(args.profile_iterations - 1):
        tr.step(trgb, tdep)
    torch.cuda.synchronize(dev)
    abi.gs_sync_status(h)
    return {"profile_iterations": args.profile_iterations, "loss": float(tr.loss)}


def trainer_snapshot(tr):
    """Parameters, Adam moments and step of a trainer (device copies)."""
    m = tr.model
    return [t.clone() for t in (m.flat, m.m, m.v)], tr.step_count


def trainer_restore(tr, snap):
    """Puts a trainer back to ``snap`` (also the context's device Adam step),
    so that timed phases start from the same map."""
    import torch

    from paper_2408_12677_gb300 import abi
    torch.cuda.synchronize()
    m = tr.model
    for dst, src in zip((m.flat, m.m, m.v), snap[0]):
        dst.copy_(src)
    tr.step_count = snap[1]
    abi.gs_ctx_set_adam_step(tr.ctx.handle, snap[1])
    torch.cuda.synchronize()


def run_sequential(args, w, views, trgb, tdep, rcfg, timed, local_rank, snap=None):
    """The batched iteration run view by view with the single-view calls:
    eager (one host read of the pair count per view) and graph-captured; each
    timed phase starts from ``snap`` (the batched run's map after its
    warm-up) when given."""
    import torch

    from paper_2408_12677_gb300.torch_api import BatchedTrainer, Context, GaussianModel

    dev = torch.device("cuda", local_rank)
    ctx_s = Context(local_rank)
    ts = BatchedTrainer(GaussianModel(w.params, device=dev), views, raster_cfg=rcfg, ctx=ctx_s)
    for _ in range(args.warmup):
        ts.step_sequential(trgb, tdep)
    if snap is not None:
        trainer_restore(ts, snap)
    ms_s_eager = timed(lambda: ts.step_sequential(trgb, tdep), args.steps)
    ts.capture_sequential(trgb, tdep)
    for _ in range(args.warmup):
        ts.replay()
    if snap is not None:
        trainer_restore(ts, snap)
    ms_s = timed(ts.replay, args.steps)
    ts.check_capacity()
    return ms_s, ms_s_eager, float(ts.loss_views.sum())


def run_multi_view(args, rank, world, local_rank):
    """Batched multi-view iteration: 8 views of uneven resolution (2 x 640x480,
    4 x 1200x680, 2 x 1752x1168) against one 500k-Gaussian map, one step =
    batched forward + loss + backward fused with one Adam step, tile shape
    from the autotuner, CUDA-graph replay; compared with the same iteration
    run view by view through the single-view calls (eager with its per-view
    host reads of the pair count, and graph-captured in no-sync mode)."""
    import torch

    from paper_2408_12677_gb300 import abi
    from paper_2408_12677_gb300.torch_api import BatchedTrainer, Context, GaussianModel
    from synth import workloads

    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    abi.load()
    t_gen = time.perf_counter()
    w = workloads.multi_view(workers=min(8, os.cpu_count() or 1))
    t_gen = time.perf_counter() - t_gen
    alu = abi.gs_measure_alu_peaks(local_rank, 50000)
    views = [(v.cam, v.pose.R, v.pose.t) for v in w.views]
    trgb = [torch.as_tensor(v.target_rgb, device=dev) for v in w.views]
    tdep = [torch.as_tensor(v.target_depth, device=dev) for v in w.views]
    stream = torch.cuda.current_stream(dev)
    npx = sum(v.cam.width * v.cam.height for v in w.views)

    def timed(fn, k):
        torch.cuda.synchronize(dev)
        a = torch.cuda.Event(enable_timing=True)
        b = torch.cuda.Event(enable_timing=True)
        a.record(stream)
        for _ in range(k):
            fn()
        b.record(stream)
        torch.cuda.synchronize(dev)
        return a.elapsed_time(b)

    # batched
    ctx_b = Context(local_rank)
    tb = BatchedTrainer(GaussianModel(w.params, device=dev), views, ctx=ctx_b)
    tune_ms = tb.autotune(reps=3)
    tile = (tb.rcfg.tile_w, tb.rcfg.tile_h)
    for _ in range(args.warmup):
        tb.step(trgb, tdep)
    abi.gs_set_eval_counting(ctx_b.handle, True)
    tb.step(trgb, tdep)
    st = ctx_b.stats()
    abi.gs_set_eval_counting(ctx_b.handle, False)
    pairs, e_blend = st["n_pairs"], st["evals_blended"]
    # every timed phase (both forms) starts from this map: the map trains
    # while it is timed, and its pairs grow with it
    snap = trainer_snapshot(tb)
    ms_b_eager = timed(lambda: tb.step(trgb, tdep), args.steps)  # sync mode: one host read per call
    tb.capture(trgb, tdep)
    for _ in range(args.warmup):
        tb.replay()
    trainer_restore(tb, snap)
    clocks = ClockSampler(local_rank)
    clocks.start()
    ms_b = timed(tb.replay, args.steps)
    clk = clocks.stop()
    tb.check_capacity()
    loss_b = float(tb.loss)
    trainer_restore(tb, snap)
    launches0 = ctx_b.stats()["kernel_launches"]
    abi.gs_set_profiling(ctx_b.handle, True)
    timed(lambda: tb._iteration(trgb, tdep, 0), args.steps)
    stages = abi.gs_profile_read(ctx_b.handle)
    abi.gs_set_profiling(ctx_b.handle, False)
    launches = ctx_b.stats()["kernel_launches"] - launches0

    # end to end: per step, H2D of all 8 target frames from pinned memory and D2H of the loss
    h_rgb = [torch.from_numpy(v.target_rgb).pin_memory() for v in w.views]
    h_dep = [torch.from_numpy(v.target_depth).pin_memory() for v in w.views]
    h_loss = torch.empty(1).pin_memory()

    trainer_restore(tb, snap)

    def e2e_step():
        for k in range(len(views)):
            trgb[k].copy_(h_rgb[k], non_blocking=True)
            tdep[k].copy_(h_dep[k], non_blocking=True)
        h_loss.copy_(tb.replay(), non_blocking=True)
    ms_e2e = timed(e2e_step, args.steps)
    h2d = sum(x.numel() * 4 for x in h_rgb + h_dep)

    if args.no_compare:
        ms_s = ms_s_eager = float("nan")
        loss_s = None
    else:
        ms_s, ms_s_eager, loss_s = run_sequential(args, w, views, trgb, tdep, tb.rcfg, timed, local_rank, snap)
    ms_b, ms_e2e = max_over_ranks([ms_b, ms_e2e], world)
    per_stage = {k: {"ms_per_launch": (ms / c if c else 0.0), "launches": c} for k, (ms, c) in stages.items()}
    dom = max(stages, key=lambda k: stages[k][0])
    dom_ms = per_stage[dom]["ms_per_launch"]
    it_s = whole_job_rate(args.steps, world, ms_b)
    roof = alu_roofline(dom, e_blend, dom_ms, alu) if dom in FLOPS_PER_BLEND else None
    return {
        "metric": METRIC, "value": it_s, "unit": "it/s", "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms_b / args.steps, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": "multi_view: 8 views (2x640x480, 4x1200x680, 2x1752x1168), 500k-Gaussian map, "
                               "SH degree 3, fp32, one Adam step on the summed loss per iteration",
                   "n_gaussians": w.n, "views": [[c.width, c.height] for c, _, _ in views], "pixels": npx,
                   "tile": f"{tile[0]}x{tile[1]}", "autotune_ms": dict(zip(["16x16", "8x32", "32x8"], tune_ms)),
                   "pairs": pairs, "parallelism": f"replicas{world}",
                   "timing": "CUDA graph replay per step", "l2": "no flush: per-step working set > 129 MB L2",
                   "host_generation_s": t_gen},
        "gaussian_pixel_evals_per_s": e_blend * it_s, "evals_blended_per_iter": e_blend,
        "comparison": None if args.no_compare else {
            "batched_graph_ms": ms_b / args.steps, "batched_eager_ms": ms_b_eager / args.steps,
            "sequential_graph_ms": ms_s / args.steps, "sequential_eager_ms": ms_s_eager / args.steps,
            "speedup_vs_sequential_graph": ms_s / ms_b, "speedup_vs_sequential_eager": ms_s_eager / ms_b,
            "loss_batched": loss_b, "loss_sequential": loss_s,
        },
        "roofline": roof,
        "stages": per_stage,
        "e2e": {"value": whole_job_rate(args.steps, world, ms_e2e), "unit": "it/s", "h2d_bytes_per_step": h2d,
                "d2h_bytes_per_step": 4},
        "gpu_launches": launches,
        "clocks": clk,
    }


def multi_view_compare(local_rank, steps=100, warmup=5):
    """The batched multi-view iteration (8 views of uneven size, 2 x 640x480,
    4 x 1200x680, 2 x 1752x1168, one 500k-Gaussian map) against the same
    iteration run view by view, both graph-captured and starting from the
    same map: the batched-vs-sequential comparison in compact form for the
    default bench line."""
    import argparse as _ap

    import torch

    from paper_2408_12677_gb300.torch_api import BatchedTrainer, Context, GaussianModel
    from synth import workloads

    dev = torch.device("cuda", local_rank)
    t_gen = time.perf_counter()
    w = workloads.multi_view(workers=min(8, os.cpu_count() or 1))
    t_gen = time.perf_counter() - t_gen
    views = [(v.cam, v.pose.R, v.pose.t) for v in w.views]
    trgb = [torch.as_tensor(v.target_rgb, device=dev) for v in w.views]
    tdep = [torch.as_tensor(v.target_depth, device=dev) for v in w.views]
    stream = torch.cuda.current_stream(dev)

    def timed(fn, k):
        torch.cuda.synchronize(dev)
        a = torch.cuda.Event(enable_timing=True)
        b = torch.cuda.Event(enable_timing=True)
        a.record(stream)
        for _ in range(k):
            fn()
        b.record(stream)
        torch.cuda.synchronize(dev)
        return a.elapsed_time(b)

    ctx_b = Context(local_rank)
    tb = BatchedTrainer(GaussianModel(w.params, device=dev), views, ctx=ctx_b)
    tb.autotune(reps=2)
    for _ in range(warmup):
        tb.step(trgb, tdep)
    snap = trainer_snapshot(tb)
    tb.capture(trgb, tdep)
    for _ in range(warmup):
        tb.replay()
    trainer_restore(tb, snap)
    ms_b = timed(tb.replay, steps)
    tb.check_capacity()
    loss_b = float(tb.loss)
    a = _ap.Namespace(steps=steps, warmup=warmup)
    ms_s, ms_s_eager, loss_s = run_sequential(a, w, views, trgb, tdep, tb.rcfg, timed, local_rank, snap)
    ctx_b.close()
    return {"views": [[c.width, c.height] for c, _, _ in views], "n_gaussians": w.n,
            "tile": f"{tb.rcfg.tile_w}x{tb.rcfg.tile_h}", "steps": steps,
            "batched_graph_ms": ms_b / steps, "sequential_graph_ms": ms_s / steps,
            "sequential_eager_ms": ms_s_eager / steps, "speedup_vs_sequential_graph": ms_s / ms_b,
            "loss_batched": loss_b, "loss_sequential": loss_s, "host_generation_s": t_gen,
            "note": "both forms from the same map after warm-up; the losses are after the same K steps"}


STREAM_SEEDING = {"var_thr": 0.035, "min_size": 2}  # about 50k Gaussians from the first 1200x680 frame
PAPER_SEEDING = {"var_thr": 0.01, "max_size": 64, "min_size": 1}  # quadtree threshold 0.1 (as a std), 1 px leaves


def _stream_frame(args):
    """Ray-cast frame k of the streaming sequence (worker process)."""
    n_frames, k = args
    from synth import workloads
    return workloads.streaming(n_frames=n_frames).frame(k)


def _stream_seed(rgb, depth, cam, pose, mask):
    from synth.quadtree import seed_gaussians
    return seed_gaussians(rgb, depth, cam, pose, 3, mask=mask, **STREAM_SEEDING)


def run_streaming(args, rank, world, local_rank):
    """Per-frame streaming optimisation at 1200x680: each frame is fused into
    the TSDF grid and seeds Gaussians where the voxel weight is 1 (or, with
    --novelty alpha, where the map's rendered alpha is below 0.5), then 10
    batched iterations over the frame and up to 4 random earlier keyframes.
    The frames are ray-cast on the host cores before the GPU starts (a spawn
    process pool); value = optimisation iterations per second of GPU time
    (CUDA events around each frame's iterations), e2e = frames per second of
    the whole loop (fusion, seeding, uploads, iterations)."""
    import multiprocessing as mp

    t_gen = time.perf_counter()
    with mp.get_context("spawn").Pool(min(16, os.cpu_count() or 1)) as pool:
        frames = pool.map(_stream_frame, [(args.frames, k) for k in range(args.frames)])
    t_gen = time.perf_counter() - t_gen

    import torch

    from paper_2408_12677_gb300 import abi
    from paper_2408_12677_gb300.streaming import StreamingOptimizer
    from synth import workloads

    torch.cuda.set_device(local_rank)
    abi.load()
    st = workloads.streaming(n_frames=args.frames)
    novelty = "alpha" if args.host_seeding else args.novelty
    seeding = STREAM_SEEDING if novelty == "alpha" else PAPER_SEEDING
    opt = StreamingOptimizer(st.cam, 3, _stream_seed if args.host_seeding else None, iters=10, n_past=4,
                             capacity=1 << 16, device=local_rank, seeding=seeding, novelty=novelty)
    clocks = ClockSampler(local_rank)
    clocks.start()
    launches0 = opt.ctx.stats()["kernel_launches"]
    t0 = time.perf_counter()
    stats = [opt.process_frame(rgb, dep, st.poses[k]) for k, (rgb, dep) in enumerate(frames)]
    wall = time.perf_counter() - t0
    clk = clocks.stop()
    launches = opt.ctx.stats()["kernel_launches"] - launches0
    from paper_2408_12677_gb300.streaming import global_optimize
    glob = global_optimize(opt, epochs=args.global_epochs, views_per_step=16) if args.global_epochs > 0 else None
    gpu_ms = sum(s.gpu_ms for s in stats)
    iters = sum(len(s.views_per_iter) for s in stats)
    views = sum(sum(s.views_per_iter) for s in stats)
    tsdf_ms = sum(s.tsdf_ms for s in stats)
    tsdf_updated = sum(s.tsdf_updated for s in stats)
    gpu_ms, wall, tsdf_ms = max_over_ranks([gpu_ms, wall, tsdf_ms], world)
    return {
        "metric": METRIC, "value": world * iters / (gpu_ms * 1e-3), "unit": "it/s", "n_gpus": world,
        "steps": iters, "warmup": 0, "ms_per_step": gpu_ms / iters, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": f"streaming: {args.frames} frames at 1200x680 (fx 600), "
                               + ("TSDF fusion (1 cm voxels, eps 8 cm) and seeding where the voxel weight is 1"
                                  if novelty == "tsdf" else "novelty seeding where rendered alpha < 0.5")
                               + ", 10 batched iterations per frame over the frame and up to 4 "
                               "random earlier keyframes, SH degree 3, fp32",
                   "frames": args.frames, "seeding": seeding, "novelty": novelty,
                   "tsdf_grid": None if opt.tsdf is None else {
                       "voxel_size_m": opt.tsdf.voxel_size, "truncation_m": opt.tsdf.truncation,
                       "max_weight": opt.tsdf.max_weight,
                       "eq9": "as printed" if opt.tsdf.fusion == 0 else "unit measurement weight"},
                   "seeding_on": "host" if args.host_seeding else "device", "host_generation_s": t_gen,
                   "parallelism": f"replicas{world}", "timing": "CUDA events around each frame's iterations"},
        "stream": {
            "gaussians_first_frame": stats[0].n_gaussians, "gaussians_last_frame": stats[-1].n_gaussians,
            "capacity_last": stats[-1].capacity, "keyframes": sum(s.keyframe for s in stats),
            "views_per_iteration_mean": views / iters, "gpu_ms_per_frame": gpu_ms / len(stats),
            "host_ms_per_frame": 1e3 * wall / len(stats), "loss_first": stats[0].loss, "loss_last": stats[-1].loss,
            "new_per_frame": [s.new_gaussians for s in stats],
        },
        # TSDF fusion (allocation + integration kernels, CUDA events): algorithmic bytes = 16 per updated
        # voxel (float2 read + write) + 4 per depth pixel
        "tsdf": None if novelty != "tsdf" else {
            "ms_per_frame": tsdf_ms / len(stats), "blocks_last": stats[-1].tsdf_blocks,
            "touched_per_frame": sum(s.tsdf_touched for s in stats) / len(stats),
            "updated_voxels_per_frame": tsdf_updated / len(stats),
            "roofline": tsdf_roofline(16 * tsdf_updated + 4 * st.cam.width * st.cam.height * len(stats), tsdf_ms,
                                      len(stats)),
        },
        # e2e step = one frame: its RGB-D upload, the alpha read-back for the novelty mask, the new
        # Gaussians' upload and one loss read
        # the offline optimisation over the keyframe list after the sequence (16 keyframes per batched step);
        # context: the paper's 10 global iterations over ~340 ScanNet++ keyframes at 876x584 take 60.1 s on an
        # RTX 3060, about 17.7 ms per view-iteration
        "global_optimisation": None if glob is None else {
            "epochs": glob.epochs, "keyframes": glob.keyframes, "batched_steps": glob.steps,
            "view_iterations": glob.view_iterations, "gpu_ms": glob.gpu_ms,
            "ms_per_view_iteration": glob.ms_per_view_iteration, "loss_first_step": glob.loss_first,
            "loss_last_step": glob.loss_last},
        "e2e": {"value": world * len(stats) / wall, "unit": "frames/s",
                "h2d_bytes_per_step": 16 * st.cam.width * st.cam.height
                + int(sum(s.new_gaussians for s in stats) / len(stats)) * 4 * (11 + 48),
                "d2h_bytes_per_step": (4 * st.cam.width * st.cam.height if novelty == "alpha" else 16 + 4) + 4 + 4},
        "gpu_launches": launches,
        "clocks": clk,
    }


def tsdf_roofline(alg_bytes, ms, frames):
    """HBM roofline of the TSDF fusion launches (allocation + integration),
    timed with CUDA events around each frame's gs_tsdf_integrate; algorithmic
    bytes: 16 per updated voxel (float2 read + write), 4 per depth pixel."""
    peak, kind = load_peaks()
    achieved = alg_bytes / (ms * 1e-3) / 1e9 if ms else 0.0
    return {"kernel": "tsdf_alloc + tsdf_integrate", "bound": "hbm", "achieved": achieved, "peak": peak,
            "unit": "GB/s", "frac": achieved / peak, "traffic": None, "peak_kind": kind,
            "alg_bytes_per_frame": alg_bytes / max(frames, 1)}


def max_over_ranks(values, world):
    """Element-wise maximum of per-rank timings (gloo/NCCL all-reduce)."""
    import torch
    t = torch.tensor([float(v) for v in values], dtype=torch.float64)
    if world > 1:
        import torch.distributed as dist
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return [float(x) for x in t]


def whole_job_rate(steps, world, max_ms):
    """Iterations per second of the whole job: every rank ran ``steps``."""
    return world * steps / (max_ms * 1e-3)


def load_traffic(kernel):
    """DRAM bytes per launch of ``kernel`` from the committed ncu summary, or
    None if there is none or the kernel's source changed since the capture."""
    import hashlib
    p = os.path.join(ROOT, "profiles", "traffic.txt")
    if not os.path.exists(p):
        return None
    for line in open(p):
        f = line.split()
        if len(f) == 4 and f[0] == kernel:
            src = os.path.join(ROOT, f[2])
            if os.path.exists(src) and hashlib.sha256(open(src, "rb").read()).hexdigest()[:16] == f[3]:
                return int(f[1])
    return None


# ---------------------------------------------------------------------------
# oracle timing (cpu_baseline / reference arm)
# ---------------------------------------------------------------------------
def _oracle_setup(w):
    """float64 leaves, the view, its 16 x 16 tiles and each tile's pixels."""
    import numpy as np

    from oracle import render as R
    v = w.views[0]
    tx, ty = -(-v.cam.width // 16), -(-v.cam.height // 16)
    return v, tx * ty, np.asarray(v.pose.R, np.float64), np.asarray(v.pose.t, np.float64), R


def oracle_iteration(w, tiles=None):
    """One iteration of the FP64 oracle on the host cores, as it stands:
    projection of every Gaussian, compositing (Eq. 11) of the pixels of
    ``tiles`` (16 x 16 tiles, every tile when None) with the Gaussians whose
    3-sigma box meets each tile (exact selection: the others have q > 9
    there), the L1 loss (Eq. 12 + depth term) of those pixels, autograd
    backward to every parameter, and a float64 Adam step over ALL parameters.
    Returns seconds of (projection + compositing forward, backward, Adam) and
    the blended (pixel, Gaussian) pairs."""
    import numpy as np
    import torch

    from oracle import adam as oadam
    v, n_tiles, Rm, t, R = _oracle_setup(w)
    pix, sizes = R.tile_pixels(v.cam, range(n_tiles) if tiles is None else tiles, sizes=True)
    lin = pix[:, 1] * v.cam.width + pix[:, 0]
    trgb = torch.as_tensor(np.asarray(v.target_rgb, np.float64).reshape(3, -1)[:, lin])
    tdep = torch.as_tensor(np.asarray(v.target_depth, np.float64).reshape(-1)[lin])
    t0 = time.perf_counter()
    P = R.to_tensors({k: np.asarray(w.params[k], np.float64) for k in R.PARAM_NAMES}, requires_grad=True)
    out = R.render(P, w.sh_degree, v.cam, Rm, t, pixels=pix, prefilter="bbox", chunk_px=sizes)
    if len(pix):
        L = R.loss_l1(out["color"], out["depth"], trgb, tdep)
    else:  # the projection alone: differentiate the sum of its outputs
        L = sum(out["proj"][k].sum() for k in ("mean2d", "cov2d", "depth", "rgb", "opacity"))
    t1 = time.perf_counter()
    g = torch.autograd.grad(L, [P[k] for k in R.PARAM_NAMES])
    t2 = time.perf_counter()
    cfg = oadam.AdamCfg()
    flat = oadam.flatten(w.params)
    oadam.adam_step(flat, np.concatenate([x.numpy().ravel() for x in g]), np.zeros_like(flat),
                    np.zeros_like(flat), 1, oadam.lr_per_element(w.n, w.sh_degree, cfg), cfg)
    t3 = time.perf_counter()
    return t1 - t0, t2 - t1, t3 - t2, int(out["n_contrib"].sum())


def oracle_whole_iteration(w):
    """One whole iteration of the oracle on the single-view workload (every
    pixel, every Gaussian, Adam on every parameter), the same procedure as
    the reference arm's steps.  Returns (seconds, description, threads)."""
    import torch
    t_f, t_b, t_a, blended = oracle_iteration(w)
    v = w.views[0]
    desc = (f"one whole iteration: projection and compositing of all {v.cam.width}x{v.cam.height} pixels "
            f"({blended} blended pairs) {t_f:.2f} s, L1 loss and backward {t_b:.2f} s, float64 Adam on all "
            f"parameters {t_a:.2f} s")
    return t_f + t_b + t_a, desc, torch.get_num_threads()


def oracle_small_iteration():
    """A whole oracle iteration (brute force, every Gaussian at every pixel)
    on the 64 x 48 / 500-Gaussian configuration: seconds."""
    import numpy as np

    from oracle import adam as oadam
    from oracle import render as R
    from synth import workloads
    w = workloads.tiny_random()
    v = w.views[0]
    t0 = time.perf_counter()
    _, g, _ = R.gradients(w.params, w.sh_degree, v.cam, np.asarray(v.pose.R, np.float64),
                          np.asarray(v.pose.t, np.float64), v.target_rgb, v.target_depth, with_pose=False)
    cfg = oadam.AdamCfg()
    flat = oadam.flatten(w.params)
    oadam.adam_step(flat, np.concatenate([g[k].numpy().ravel() for k in R.PARAM_NAMES]), np.zeros_like(flat),
                    np.zeros_like(flat), 1, oadam.lr_per_element(w.n, w.sh_degree, cfg), cfg)
    return time.perf_counter() - t0


def run_reference(args):
    """The reference arm: the FP64 oracle, as it stands, on the host cores,
    timing WHOLE iterations of the single-view workload (every pixel, every
    Gaussian, Adam on every parameter).  An iteration takes tens of seconds,
    so the arm runs as many as fit in about two minutes (at least one) and
    reports that true count in ``steps`` (``warmup`` 0); the requested
    --steps / --warmup are echoed under ``requested``."""
    from synth import workloads
    w = workloads.single_view()
    times, blended = [], 0
    t_start = time.perf_counter()
    while len(times) < max(1, args.steps) and (not times or time.perf_counter() - t_start + times[-1] < 120.0):
        t_f, t_b, t_a, blended = oracle_iteration(w)
        times.append(t_f + t_b + t_a)
    import torch
    value = len(times) / sum(times)
    desc = (f"{len(times)} whole iterations (projection, compositing of all {w.views[0].cam.width}x"
            f"{w.views[0].cam.height} pixels with {blended} blended pairs, L1 loss, backward, Adam on all "
            f"parameters), {[round(x, 2) for x in times]} s")
    return {
        "impl": "reference", "metric": METRIC, "value": value, "unit": "it/s", "n_gpus": 1, "steps": len(times),
        "warmup": 0, "ms_per_step": 1e3 / value, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": WORKLOAD, "n_gaussians": w.n},
        "requested": {"steps": args.steps, "warmup": args.warmup},
        "cpu_baseline": {"value": value, "unit": "it/s", "cores": torch.get_num_threads(), "kind": "oracle",
                         "sample": desc},
        "e2e": {"value": value, "unit": "it/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=300)
    ap.add_argument("--warmup", type=int, default=10)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--workload", default="single_view",
                    choices=["single_view", "multi_view", "streaming", "scale_stress"],
                    help="multi_view: the batched 8-view iteration vs the same iteration view by view")
    ap.add_argument("--frames", type=int, default=40, help="streaming: frames of the sequence")
    ap.add_argument("--novelty", choices=("tsdf", "alpha"), default="tsdf",
                    help="streaming: seed where the TSDF voxel weight is 1 (the paper) or where rendered alpha < 0.5")
    ap.add_argument("--host-seeding", action="store_true",
                    help="streaming: seed new Gaussians with the host quadtree instead of gs_seed_quadtree")
    ap.add_argument("--global-epochs", type=int, default=2,
                    help="streaming: passes of the offline optimisation over the keyframe list afterwards")
    ap.add_argument("--no-multi-view", action="store_true",
                    help="single_view: skip the compact batched-vs-sequential multi-view comparison")
    ap.add_argument("--profile-iterations", type=int, default=0,
                    help="run this many eager single-view iterations and exit (a short driver for ncu captures)")
    ap.add_argument("--no-compare", action="store_true",
                    help="multi_view: skip the view-by-view comparison arm (e.g. for a profiler capture)")
    args = ap.parse_args()
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))
    if args.impl == "reference":
        if rank == 0:
            print(json.dumps(run_reference(args)))
        return
    if args.profile_iterations > 0:
        print(json.dumps(run_profile_driver(args, local_rank)))
        return
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("gloo")
    if args.workload in ("multi_view", "streaming", "scale_stress"):
        run = {"multi_view": run_multi_view, "streaming": run_streaming, "scale_stress": run_scale_stress}[args.workload]
        out = run(args, rank, world, local_rank)
        if rank == 0:
            print(json.dumps(out))
        if world > 1:
            import torch.distributed as dist
            dist.destroy_process_group()
        return
    out = run_ours(args, rank, world, local_rank)
    if rank == 0 and not args.no_multi_view:
        out["multi_view"] = multi_view_compare(local_rank)
    if rank == 0:
        if not args.no_cpu_baseline:
            from synth import workloads
            t_iter, desc, cores = oracle_whole_iteration(workloads.single_view())
            out["cpu_baseline"] = {"value": 1.0 / t_iter, "unit": "it/s", "cores": cores, "kind": "oracle",
                                   "sample": desc, "whole_iteration_64x48_500_s": oracle_small_iteration()}
        print(json.dumps(out))
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
