"""Benchmark: RGB + depth + normal + semantic forward+backward views/s.

Workload: the 1M-Gaussian synthetic room (log-scales N(-4.5, 1) clipped at -1,
SH degree 3, 64 logits, k factor), seen at 1280x720.  One step renders and
back-propagates a batch of 16 views on the orbit:

* batched (the headline ``value``): one plan over the 16 cameras, SH and
  logits stored as bfloat16, FP32 arithmetic, the whole preprocess + sort +
  forward + normal-from-depth + backward sequence captured in one CUDA graph
  and replayed per step;
* per_view: the plain path, FP32 features, one camera per call sequence with
  the instance count read back each call (16 sequences per step).

Inputs (parameters, workspace, outputs) are far larger than the 129 MB L2, so
no flush is needed between steps.  ``--impl reference`` times the FP64 CPU
oracle on a bounded sample of the same workload.

``e2e`` runs the same 16 views through the public API with the combined loss
of Sec. 3.4 driving the backward, the targets copied from pinned host memory
every step and the loss record read back.  ``train_step`` times one training
iteration (forward, loss, backward, Adam) of the 6M-Gaussian, 8 x 1080p
workload and the HBM-bound Adam and loss kernels against the HBM peak.

Multi-GPU: the path renders independent views, so N ranks are N replicas
(weak scaling, no collective); ``value`` sums the views of all ranks.
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

METRIC = "RGB+D+N+sem fwd+bwd views/s at 1M Gaussians 720p; batched vs per-view"
N_GAUSS = 1_000_000
N_VIEWS = 16
WORKLOAD = "1M-Gaussian synthetic room, 16 orbit views at 1280x720, 64 logits, SH3, fwd+bwd"


def workload_config(n_gauss: int = N_GAUSS) -> dict:
    """The workload both arms measure (identical in their JSON lines)."""
    return {"workload": WORKLOAD, "gaussians": n_gauss, "views_per_step": N_VIEWS,
            "resolution": "1280x720", "n_sem": 64, "sh_degree": 3,
            "features": "SH and logits rounded to bfloat16 (the oracle takes the same values)",
            "l2": "inputs larger than L2 (no flush)"}


def _dist():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    return ws, rank


class ClockSampler:
    """nvidia-smi clocks / throttle reasons sampled every 200 ms."""

    QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        self.path = os.path.join(tempfile.gettempdir(), f"unigs_clocks_{os.getpid()}.csv")

    def __enter__(self):
        try:
            os.makedirs(os.path.dirname(self.path), exist_ok=True)
            self.f = open(self.path, "w")
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--id={self.gpu}", f"--query-gpu={self.QUERY}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=self.f, stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None
        return self

    def __exit__(self, *a):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()
            self.f.close()

    def summary(self):
        if self.proc is None or not os.path.exists(self.path):
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        sm, smax, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax = float(parts[2])
            except ValueError:
                continue
            for n, v in zip(names, parts[5:9]):
                if v.lower() == "active":
                    reasons.add(n)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": smax,
                "reasons": sorted(reasons), "samples": len(sm)}


# DRAM bytes (read + write) of one launch of the backward composite on this
# workload (render_bwd_tc_kernel<64>), from a one-pass ncu capture of the
# full run (dram__bytes_read.sum 6.827 GB + dram__bytes_write.sum 1.086 GB;
# the two metrics take one pass), valid only for the kernel sources whose
# digest is recorded here; any change to them reports null until re-captured.
BWD_TRAFFIC_BYTES = 7_913_533_184
BWD_TRAFFIC_SOURCES = ('render_bwd.cu', 'render_bwd_tc.cu', 'bwd_pair.cuh', 'splat.cuh',
                       'unigs_internal.cuh', 'ff.cuh', 'sh.cuh', 'tcgen05.cuh', 'ewa_ff.cuh')
BWD_TRAFFIC_DIGEST = "e088559ec0bc1e1b3cfc7c44e468995b5d0188098c9e65f52ea084b517cdbd4f"


def bwd_traffic():
    import hashlib
    h = hashlib.sha256()
    for f in BWD_TRAFFIC_SOURCES:
        with open(os.path.join(ROOT, "paper_2510_12174_gb300", "csrc", f), "rb") as fh:
            h.update(fh.read())
    return BWD_TRAFFIC_BYTES if h.hexdigest() == BWD_TRAFFIC_DIGEST else None


def hbm_bytes_per_step(n: int, sh_degree: int, n_sem: int, pixels: int, instances: int,
                       feat_bytes: int) -> int:
    """Algorithmic HBM bytes of one batched forward + backward step: every
    parameter read once in each pass (P twice), each parameter gradient written
    once (G), each output (O) and upstream gradient (U, plus the
    normal-from-depth gradient) touched once, and 44 B per (tile, Gaussian)
    instance (written, sorted once, read by both composites).  P and G are paid
    once for all views of the step; pixels is the total over the views."""
    n_sh = (sh_degree + 1) ** 2
    P = n * (48 + (3 * n_sh + n_sem) * feat_bytes)
    G = n * (12 + 3 * n_sh + n_sem) * 4
    O = pixels * (8 + n_sem + 2) * 4
    U = pixels * (8 + n_sem) * 4 + 3 * pixels * 4
    return 2 * P + G + O + U + 44 * instances


def launch_shape(cfg, paths: int) -> dict:
    """The composites' kernels and launch shapes after the library's defaults
    (``paths``: unigs_plan_paths of the plan)."""
    from paper_2510_12174_gb300 import abi
    fwd_tc = bool(paths & abi.UNIGS_PATH_FWD_TC)
    bwd_tc = bool(paths & abi.UNIGS_PATH_BWD_TC)
    bwd = (16, 2) if bwd_tc else (int(cfg.batch) or 8, int(cfg.ctas_per_sm) or 3)
    if not fwd_tc:
        fwd = (int(cfg.batch_fwd) or 32, int(cfg.ctas_per_sm_fwd) or 2)
    else:
        fwd = (int(cfg.batch_fwd) or 16, min(int(cfg.ctas_per_sm_fwd) or 4, 4))
    return {"tile": [int(cfg.tile_w) or 16, int(cfg.tile_h) or 16],
            "fwd": {"batch": fwd[0], "ctas_per_sm": fwd[1],
                    "logits": "tensor cores" if fwd_tc else "fp32 pipes"},
            "bwd": {"batch": bwd[0], "ctas_per_sm": bwd[1],
                    "logits": "tensor cores" if bwd_tc else "fp32 pipes"}}


def parse_tile(text: str) -> tuple:
    """'WxH' -> (W, H); one of the library's 256-pixel tile shapes."""
    from paper_2510_12174_gb300 import abi
    w, h = (int(v) for v in text.lower().split("x"))
    if (w, h) not in abi.TILE_SHAPES:
        raise SystemExit(f"--tile {text}: not one of {abi.TILE_SHAPES}")
    return w, h


def aggregate(ms_local: float, world: int, device) -> tuple:
    """Whole-job time and throughput of N independent replicas: the slowest
    rank's ms per step, and the views of every rank over that time."""
    ms_all = float(ms_local)
    if world > 1:
        import torch
        import torch.distributed as dist
        t = torch.tensor([ms_all], dtype=torch.float64, device=device)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        ms_all = float(t.item())
    return ms_all, world * N_VIEWS / (ms_all / 1000.0)


def _peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return json.load(f), "measured"
    except Exception:
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "sm_max_mhz": 2070.0}, "fallback"


def measure_fp32_peak(dev) -> dict:
    """FP32 FMA throughput of this GPU, measured with the library's probe
    (unigs_probe_fma: 8 independent FMA chains per thread, 8 CTAs of 256
    threads per SM), scalar and packed-pair FMAs, best of 5 launches each;
    the SM count comes from the device."""
    import ctypes

    import torch

    from paper_2510_12174_gb300 import abi
    sink = torch.empty(abi.unigs_probe_fma_sink_floats(), device=dev)
    st = torch.cuda.current_stream(dev)
    res = {"sm_count": torch.cuda.get_device_properties(dev).multi_processor_count}
    for name, packed in (("fma", 0), ("fma2", 1)):
        fl = ctypes.c_int64(0)
        best = 0.0
        for rep in range(6):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(st)
            abi.check(abi.unigs_probe_fma(sink.data_ptr(), 2048, packed, fl, st.cuda_stream),
                      "unigs_probe_fma")
            e1.record(st)
            torch.cuda.synchronize(dev)
            if rep:
                best = max(best, fl.value / (e0.elapsed_time(e1) / 1000.0) / 1e12)
        res[f"{name}_tflops"] = best
    res["tflops"] = max(res["fma_tflops"], res["fma2_tflops"])
    return res


# FP32 operations per (pixel, Gaussian) pair of the backward composite, counted
# from its source (FMA = 2): alpha recomputation ~24 per evaluated pair; per
# blended pair ~ 80 (geometry recompute) + 2*(8 + n_sem) (G_i dot) + ~190
# (alpha, depth, normal chains) + 2*n_sem (semantic gradients).
def bwd_flops(n_eval, n_blend, n_sem, tensor_logits=False):
    """FP32-pipe flops of the backward; with ``tensor_logits`` the 4 n_sem of
    the logit terms (G_i's logit dot product and the logit-feature gradient)
    run on the tensor cores and are not counted."""
    sem = 0 if tensor_logits else 4 * n_sem
    return 24.0 * n_eval + (80 + 16 + 190 + sem) * n_blend


def fwd_flops(n_eval, n_blend, n_sem):
    return 24.0 * n_eval + (80 + 2 * (11 + n_sem) + 10) * n_blend


def _time_ms(fn, steps: int, warmup: int, dev) -> float:
    """Mean ms per call of fn() on the current stream (CUDA events)."""
    import torch
    for _ in range(warmup):
        fn()
    torch.cuda.synchronize(dev)
    st = torch.cuda.current_stream(dev)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(st)
    for _ in range(steps):
        fn()
    e1.record(st)
    torch.cuda.synchronize(dev)
    return e0.elapsed_time(e1) / steps


def _capture(fn, dev):
    """fn() captured in a CUDA graph (after two runs on a side stream)."""
    import torch
    side = torch.cuda.Stream(device=dev)
    side.wait_stream(torch.cuda.current_stream(dev))
    with torch.cuda.stream(side):
        for _ in range(2):
            fn()
    torch.cuda.current_stream(dev).wait_stream(side)
    torch.cuda.synchronize(dev)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        fn()
    torch.cuda.synchronize(dev)
    return g


def _device_upstream(r, n_sem, seed, dev):
    """N(0,1) upstream gradients for a renderer's flat outputs, drawn on the
    device from a seeded generator (the timing does not depend on them)."""
    import torch
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    P = r.n_pixels
    ch = {"rgb": 3, "depth": 1, "normal_g": 3, "kmap": 1, "logits": n_sem, "normal_d": 3}
    return {k: torch.randn(c * P, generator=gen, device=dev) for k, c in ch.items()}


def measure_configs(dev, fp32_tflops: float, hbm_gbs: float, steps: int) -> dict:
    """Throughput of the neighbouring workload configurations (the parity tests
    cover their numerics): config 1 forward-only, 10k Gaussians at 256x256
    (microseconds per view through the per-call path, which reads the instance
    count back, and as a replayed graph); config 2 forward + backward, 200k
    Gaussians at 640x480, 32 logits, FP32 (per call and as a graph); config 4,
    3M Gaussians over 16 orbit views of mixed resolution with BF16 features,
    the batched graph against the same views looped one camera at a time
    through the plain FP32 path.  Each entry carries the ALU fraction (FP32
    work of the pair model over the measured FP32 peak) and the HBM fraction
    (algorithmic bytes over the measured copy bandwidth)."""
    import torch

    from paper_2510_12174_gb300 import abi
    from paper_2510_12174_gb300 import rasterizer as rz
    from paper_2510_12174_gb300 import scenes

    res = {}
    n_rep = max(3, min(steps, 10))

    def fracs(flops, nbytes, ms):
        return {"alu_frac": flops / (ms / 1000.0) / 1e12 / fp32_tflops,
                "hbm_frac": nbytes / (ms / 1000.0) / 1e9 / hbm_gbs,
                "flops": flops, "bytes": nbytes}

    # ---- config 1: forward only
    sc, cams = scenes.config1()
    ds = rz.DeviceScene.from_scene(sc, device=dev)
    r = rz.Renderer(ds, cams)
    out = r.forward()
    torch.cuda.synchronize(dev)
    n_inst = int(r.last_instances)
    n_eval, n_blend = r.stats()
    call_ms = _time_ms(lambda: r.forward(out), 20 * n_rep, 5, dev)
    rg = rz.Renderer(ds, cams, capacity=int(n_inst * 1.15) + 4096)
    og = rg.alloc_outputs()
    g = _capture(lambda: rg.forward(og, readback=False), dev)
    graph_ms = _time_ms(g.replay, 20 * n_rep, 5, dev)
    del g
    n_sh = (sc.sh_degree + 1) ** 2
    pix = sum(c.width * c.height for c in cams)
    fwd_bytes = sc.n * (48 + (3 * n_sh + sc.n_sem) * 4) + pix * (10 + sc.n_sem) * 4 + 40 * n_inst
    res["config1"] = {"workload": "10k Gaussians, 1 view 256x256, 16 logits, forward only, FP32",
                      "us_per_view_call": call_ms * 1000.0, "us_per_view_graph": graph_ms * 1000.0,
                      "instances": n_inst, "pairs_evaluated": n_eval, "pairs_blended": n_blend,
                      **fracs(fwd_flops(n_eval, n_blend, sc.n_sem), fwd_bytes, graph_ms)}
    del r, rg, ds, out, og

    # ---- config 2: forward + backward, FP32, one view
    sc, cams = scenes.config2()
    ds = rz.DeviceScene.from_scene(sc, device=dev)
    r = rz.Renderer(ds, cams)
    out = r.forward()
    torch.cuda.synchronize(dev)
    n_inst = int(r.last_instances)
    n_eval, n_blend = r.stats()
    up = _device_upstream(r, sc.n_sem, 41, dev)
    grads = r.alloc_grads()
    gbuf = torch.empty(r.n_pixels, device=dev)

    def call2():
        r.forward(out)
        r.backward(out, up, grads=grads, g_depth_buf=gbuf)

    call_ms = _time_ms(call2, 5 * n_rep, 3, dev)
    rg = rz.Renderer(ds, cams, capacity=int(n_inst * 1.15) + 65536)
    og, gg = rg.alloc_outputs(), rg.alloc_grads()
    gb2 = torch.empty(rg.n_pixels, device=dev)
    g = _capture(lambda: (rg.forward(og, readback=False),
                          rg.backward(og, up, grads=gg, g_depth_buf=gb2)), dev)
    graph_ms = _time_ms(g.replay, 5 * n_rep, 3, dev)
    del g
    pix = sum(c.width * c.height for c in cams)
    nbytes = hbm_bytes_per_step(sc.n, sc.sh_degree, sc.n_sem, pix, n_inst, 4)
    res["config2"] = {"workload": "200k Gaussians, 1 view 640x480, 32 logits, SH3, forward + "
                                  "backward, FP32",
                      "views_per_s_call": 1000.0 / call_ms, "views_per_s_graph": 1000.0 / graph_ms,
                      "ms_per_view_graph": graph_ms, "instances": n_inst,
                      "pairs_evaluated": n_eval, "pairs_blended": n_blend,
                      **fracs(fwd_flops(n_eval, n_blend, sc.n_sem)
                              + bwd_flops(n_eval, n_blend, sc.n_sem), nbytes, graph_ms)}
    del r, rg, ds, out, og, grads, gg, up, gbuf, gb2

    # ---- config 4: 3M Gaussians, 16 views of mixed resolution
    sc, cams = scenes.config4()
    ds = rz.DeviceScene.from_scene(sc, device=dev, feat_bf16=True)
    r = rz.Renderer(ds, cams)
    out = r.forward()
    torch.cuda.synchronize(dev)
    n_inst = int(r.last_instances)
    n_eval, n_blend = r.stats()
    rb = rz.Renderer(ds, cams, capacity=int(n_inst * 1.15) + 65536)
    del r, out
    ob, gb = rb.alloc_outputs(), rb.alloc_grads()
    up = _device_upstream(rb, sc.n_sem, 42, dev)
    gbufb = torch.empty(rb.n_pixels, device=dev)
    g = _capture(lambda: (rb.forward(ob, readback=False),
                          rb.backward(ob, up, grads=gb, g_depth_buf=gbufb)), dev)
    batched_ms = _time_ms(g.replay, n_rep, 2, dev)
    del g
    offs = rb.pixel_offsets()
    ch = {"rgb": 3, "depth": 1, "normal_g": 3, "kmap": 1, "logits": sc.n_sem, "normal_d": 3}
    up_views = [{k: up[k][offs[i] * c: offs[i + 1] * c] for k, c in ch.items()}
                for i in range(len(cams))]
    tc4 = bool(abi.unigs_plan_paths(rb.plan) & abi.UNIGS_PATH_BWD_TC)
    del rb, ob, gb, gbufb
    torch.cuda.empty_cache()
    ds32 = rz.DeviceScene.from_scene(sc, device=dev, feat_bf16=False)
    rend = [rz.Renderer(ds32, [c]) for c in cams]
    outs = [rr.forward() for rr in rend]
    gr32 = [rr.alloc_grads() for rr in rend]

    def looped():
        for i, rr in enumerate(rend):
            rr.forward(outs[i])
            rr.backward(outs[i], up_views[i], grads=gr32[i])

    looped_ms = _time_ms(looped, max(2, n_rep // 2), 1, dev)
    pix = sum(c.width * c.height for c in cams)
    nbytes = hbm_bytes_per_step(sc.n, sc.sh_degree, sc.n_sem, pix, n_inst, 2)
    flops = fwd_flops(n_eval, n_blend, sc.n_sem) + bwd_flops(n_eval, n_blend, sc.n_sem, tc4)
    res["config4"] = {"workload": "3M Gaussians, 16 orbit views drawn from 640x480, 1280x720 "
                                  "and 1920x1080, 64 logits, SH3, forward + backward",
                      "batched_views_per_s": len(cams) * 1000.0 / batched_ms,
                      "batched_ms_per_step": batched_ms,
                      "looped_fp32_views_per_s": len(cams) * 1000.0 / looped_ms,
                      "looped_ms_per_step": looped_ms,
                      "batched_over_looped": looped_ms / batched_ms,
                      "resolutions": sorted({f"{c.width}x{c.height}" for c in cams}),
                      "instances": n_inst, "pairs_evaluated": n_eval, "pairs_blended": n_blend,
                      **fracs(flops, nbytes, batched_ms)}
    del rend, outs, gr32, ds, ds32, up, up_views
    torch.cuda.empty_cache()
    return res


def run_ours(args):
    import numpy as np
    import torch

    import __graft_entry__ as ge
    from paper_2510_12174_gb300 import abi
    from paper_2510_12174_gb300 import rasterizer as rz
    from paper_2510_12174_gb300 import scenes

    world, rank = _dist()
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    ge.build()
    dev = torch.device("cuda", local)

    def barrier():
        if world > 1:
            import torch.distributed as dist
            dist.barrier()

    sc, cams = scenes.config3_orbit(N_VIEWS, n=args.n_gauss, feat_bf16=True)
    n_sem = sc.n_sem
    up = scenes.upstream_grads(cams, n_sem, seed=5)
    keys = ("rgb", "depth", "normal_g", "kmap", "logits", "normal_d")
    host_up = {k: torch.from_numpy(np.concatenate([a.ravel() for a in up[k]])) for k in keys}
    dev_up = {k: v.to(dev) for k, v in host_up.items()}

    # ------------------------------------------------ batched (BF16, graph)
    ds = rz.DeviceScene.from_scene(sc, device=dev, feat_bf16=True)
    cfg = abi.unigs_config_default()
    cfg.batch, cfg.ctas_per_sm = args.batch, args.ctas
    cfg.batch_fwd, cfg.ctas_per_sm_fwd = args.batch_fwd, args.ctas_fwd
    cfg.tile_w, cfg.tile_h = parse_tile(args.tile)
    if args.simt_logits:
        cfg.flags |= abi.UNIGS_FLAG_SIMT_LOGITS
    r = rz.Renderer(ds, cams, cfg=cfg)
    out = r.forward()                      # sizes the capacity (one read-back)
    torch.cuda.synchronize()
    n_inst = int(r.last_instances)
    cap = int(n_inst * 1.15) + 65536
    r = rz.Renderer(ds, cams, cfg=cfg, capacity=cap)
    out = r.alloc_outputs()
    grads = r.alloc_grads()
    gbuf = torch.empty(r.n_pixels, device=dev)

    def step():
        r.forward(out, readback=False)
        r.backward(out, dev_up, grads=grads, g_depth_buf=gbuf)

    s_side = torch.cuda.Stream(device=dev)
    s_side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s_side):
        for _ in range(2):
            step()
    torch.cuda.current_stream().wait_stream(s_side)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step()
    torch.cuda.synchronize()
    for _ in range(args.warmup):
        graph.replay()
    torch.cuda.synchronize()
    st, need = r.status()
    if st != 0:
        raise RuntimeError(f"device status {st} (need {need}) after warm-up")
    n_eval, n_blend = r.stats()

    stream = torch.cuda.current_stream()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    barrier()
    torch.cuda.synchronize()
    with ClockSampler(local) as clk:
        e0.record(stream)
        for _ in range(args.steps):
            graph.replay()
        e1.record(stream)
        torch.cuda.synchronize()
    barrier()
    ms = e0.elapsed_time(e1) / args.steps
    ms_all, value = aggregate(ms, world, dev)

    # stage times (same kernels, outside the graph, CUDA events on the stream)
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(5)]
    reps = max(2, min(5, args.steps))
    acc = np.zeros(4)
    for _ in range(reps):
        ev[0].record(stream)
        r.preprocess_and_sort(readback=False)
        ev[1].record(stream)
        abi.check(abi.unigs_render_fwd(r.plan, ds.struct(), r.ws.data_ptr(),
                                       r._out_struct(out), r._stream()))
        abi.check(abi.unigs_depth_normal_fwd(r.plan, r.cams, out["depth"].data_ptr(),
                                             out["normal_d"].data_ptr(), r._stream()))
        ev[2].record(stream)
        abi.check(abi.unigs_depth_normal_bwd(r.plan, r.cams, out["depth"].data_ptr(),
                                             dev_up["normal_d"].data_ptr(),
                                             dev_up["depth"].data_ptr(), gbuf.data_ptr(),
                                             r._stream()))
        ev[3].record(stream)
        go = abi.unigs_grad_outputs()
        go.rgb, go.depth = dev_up["rgb"].data_ptr(), gbuf.data_ptr()
        go.normal_g, go.kmap = dev_up["normal_g"].data_ptr(), dev_up["kmap"].data_ptr()
        go.logits = dev_up["logits"].data_ptr()
        pg = abi.unigs_param_grads()
        for k in ("mean", "quat", "scale", "opacity", "kfac", "sh", "sem"):
            setattr(pg, k, grads[k].data_ptr())
        abi.check(abi.unigs_render_bwd(r.plan, ds.struct(), r.cams, r.ws.data_ptr(),
                                       r._out_struct(out), go, pg, r._stream()))
        ev[4].record(stream)
        torch.cuda.synchronize()
        acc += [ev[i].elapsed_time(ev[i + 1]) for i in range(4)]
    stage_ms = acc / reps

    # ------------------------------------------------ e2e through host buffers
    # The same 16 views through the public API, with the combined loss of
    # Sec. 3.4 driving the backward: every step copies that step's targets
    # from pinned host memory, renders, evaluates the loss, back-propagates
    # and reads the loss record back.  Targets are double-buffered: a copy
    # stream uploads step k+1's targets while step k computes (one captured
    # graph per buffer set).
    tg = scenes.synthetic_targets(cams, n_sem, seed=6)
    host_tg = {k: torch.from_numpy(np.concatenate([a.ravel() for a in tg[k]])).pin_memory()
               for k in tg}
    dev_tg = [{k: v.to(dev) for k, v in host_tg.items()} for _ in range(2)]
    records = [torch.zeros(16, device=dev) for _ in range(2)]
    lg = r.alloc_loss_grads()

    def e2e_step(i):
        r.forward(out, readback=False)
        r.loss(out, dev_tg[i], records[i], lg)
        r.backward(out, lg, grads=grads, g_depth_buf=gbuf)

    s_side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s_side):
        for i in range(2):
            e2e_step(i)
    torch.cuda.current_stream().wait_stream(s_side)
    torch.cuda.synchronize()
    graphs_e2e = []
    for i in range(2):
        g_i = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g_i):
            e2e_step(i)
        graphs_e2e.append(g_i)
    res_host = torch.empty(16, dtype=torch.float32).pin_memory()
    for g_i in graphs_e2e:
        g_i.replay()
    torch.cuda.synchronize()
    copy_stream = torch.cuda.Stream(device=dev)
    copied = [torch.cuda.Event() for _ in range(2)]
    used = [torch.cuda.Event() for _ in range(2)]

    def upload(j):
        with torch.cuda.stream(copy_stream):
            for k in dev_tg[j]:
                dev_tg[j][k].copy_(host_tg[k], non_blocking=True)
            copied[j].record(copy_stream)

    e2 = torch.cuda.Event(enable_timing=True)
    e3 = torch.cuda.Event(enable_timing=True)
    e2e_steps = max(2, min(args.steps, 6))
    e2.record(stream)
    copy_stream.wait_stream(stream)
    upload(0)
    for k in range(e2e_steps):
        i = k % 2
        if k + 1 < e2e_steps:
            if k >= 1:
                copy_stream.wait_event(used[1 - i])  # step k-1 has read that set
            upload(1 - i)
        stream.wait_event(copied[i])
        graphs_e2e[i].replay()
        used[i].record(stream)
        res_host.copy_(records[i], non_blocking=True)
    e3.record(stream)
    torch.cuda.synchronize()
    e2e_ms = e2.elapsed_time(e3) / e2e_steps
    h2d = sum(v.numel() * v.element_size() for v in host_tg.values())
    e2e_loss = float(res_host[0])
    del graphs_e2e, dev_tg, host_tg, lg

    # ------------------------------------------------ per-view FP32 path
    pv = None
    if not args.skip_per_view:
        ds32 = rz.DeviceScene.from_scene(sc, device=dev, feat_bf16=False)
        rend = [rz.Renderer(ds32, [c]) for c in cams]
        pv_up = []
        offs = r.pixel_offsets()
        for k in range(N_VIEWS):
            d = {}
            for key in keys:
                ch = {"rgb": 3, "depth": 1, "normal_g": 3, "kmap": 1, "logits": n_sem,
                      "normal_d": 3}[key]
                d[key] = dev_up[key][offs[k] * ch: offs[k + 1] * ch]
            pv_up.append(d)
        outs = [rr.forward() for rr in rend]
        gr32 = [rr.alloc_grads() for rr in rend]
        torch.cuda.synchronize()

        def pv_step():
            for k, rr in enumerate(rend):
                o = rr.forward(outs[k])
                rr.backward(o, pv_up[k], grads=gr32[k])

        for _ in range(max(1, args.warmup // 2)):
            pv_step()
        torch.cuda.synchronize()
        pv_steps = max(1, args.steps // 2)
        e0.record(stream)
        for _ in range(pv_steps):
            pv_step()
        e1.record(stream)
        torch.cuda.synchronize()
        pv_ms = e0.elapsed_time(e1) / pv_steps
        pv = {"value": N_VIEWS / (pv_ms / 1000.0), "unit": "views/s", "ms_per_step": pv_ms,
              "dtype": "f32", "note": "one camera per call sequence, instance count read back"}
        del rend, outs, gr32, ds32

    peaks, src = _peaks()
    clocks = clk.summary()
    paths = abi.unigs_plan_paths(r.plan)
    f_bwd = bwd_flops(n_eval, n_blend, n_sem, bool(paths & abi.UNIGS_PATH_BWD_TC))
    bwd_ms = stage_ms[3]
    fp32 = measure_fp32_peak(dev)
    fp32_peak = fp32["tflops"]
    achieved = f_bwd / (bwd_ms / 1000.0) / 1e12
    line = {
        "metric": METRIC, "value": value, "unit": "views/s", "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_all,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
        "data": "synthetic",
        "config": workload_config(args.n_gauss),
        "run": {"path": "batched, one CUDA graph per step", "parallelism": f"replicas{world}",
                "launch_shape": launch_shape(r.cfg, paths)},
        "per_view": pv,
        "stage_ms": {"preprocess+bin_sort": stage_ms[0], "render_fwd+normal_d": stage_ms[1],
                     "depth_normal_bwd": stage_ms[2], "render_bwd": stage_ms[3]},
        "work": {"pairs_evaluated": n_eval, "pairs_blended": n_blend,
                 "instances": n_inst,
                 "gaussian_pixel_evals_per_s": n_eval / (ms_all / 1000.0)},
        "roofline": {"bound": "alu",
                     "kernel": "render_bwd (composite backward + preprocess backward; the logit "
                               "terms on the tensor cores where the plan runs them there)",
                     "achieved": achieved, "peak": fp32_peak, "unit": "TFLOP/s",
                     "frac": achieved / fp32_peak,
                     "traffic": (bwd_traffic() if (args.n_gauss, args.batch, args.ctas) ==
                                 (N_GAUSS, 0, 0) else None),
                     "peak_source": "measured: FP32 FMA probe (unigs_probe_fma) on this GPU, "
                                    "best of scalar and packed-pair FMAs",
                     "peak_probe": fp32,
                     "flops_model": "FP32-pipe flops: per evaluated pair 24, per blended pair "
                                    f"{int(bwd_flops(0, 1, n_sem, bool(paths & abi.UNIGS_PATH_BWD_TC)))} "
                                    "(FMA = 2)"},
        "e2e": {"value": N_VIEWS / (e2e_ms / 1000.0) * world, "unit": "views/s",
                "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": 64,
                "note": "per step: targets (rgb, depth, normal, label) host->device from pinned "
                        "memory (double-buffered on a copy stream), forward, combined loss "
                        "(Sec. 3.4), backward, loss record device->host", "loss": e2e_loss},
        "gpu_launches": r.launches_per_step() * args.steps,
        "clocks": clocks,
    }
    hbm_b = hbm_bytes_per_step(args.n_gauss, sc.sh_degree, n_sem,
                               sum(c.width * c.height for c in cams), n_inst, 2)
    hbm_peak = float(peaks.get("hbm_gbs", 6800.0))
    line["hbm_view"] = {"bytes_per_step": hbm_b,
                        "achieved_gbs": hbm_b / (ms_all / 1000.0) / 1e9 * world,
                        "peak_gbs": hbm_peak,
                        "frac": hbm_b / (ms_all / 1000.0) / 1e9 * world / hbm_peak,
                        "note": "algorithmic bytes of the whole step against the measured "
                                "copy bandwidth; the step is ALU/issue-bound (see roofline)"}
    if not args.skip_train or not args.skip_configs:
        del graph, r, out, grads, gbuf, dev_up
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
    if not args.skip_configs:
        line["configs"] = measure_configs(dev, fp32_peak, hbm_peak, args.steps)
    if not args.skip_train:
        line["train_step"] = train_bench(args, dev, peaks)
    if rank == 0 and not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline(args.cpu_tiles)
    if rank == 0:
        print(json.dumps(line), flush=True)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


def train_bench(args, dev, peaks):
    """One training iteration of the 6M-Gaussian workload (8 orbit views at
    1920x1080, 64 logits, BF16 feature copies): forward, combined loss,
    backward, Adam over every parameter array - one CUDA graph per step.
    Also times the two HBM-bound training kernels alone against the HBM peak:
    Adam (bytes: every raw value, gradient and moment read; raw value and
    moments written; activated float32 or bfloat16 copy written) and the loss
    (both passes read every output and target channel; the gradient pass
    writes the gradient maps)."""
    import numpy as np
    import torch

    from paper_2510_12174_gb300 import rasterizer as rz
    from paper_2510_12174_gb300 import scenes
    from paper_2510_12174_gb300 import train as tr

    sc, cams = scenes.config5(n=args.train_gauss)
    tsc = scenes.perturb(sc, seed=5)
    # targets: renders of the perturbed scene (rgb, depth, normal-from-depth)
    # and uniform labels with 10% unlabelled
    rt = rz.Renderer(rz.DeviceScene.from_scene(tsc, device=dev, feat_bf16=True), cams)
    o = rt.forward()
    lab = scenes.synthetic_targets(cams, sc.n_sem, seed=7)["label"]
    targets = {"rgb": o["rgb"].clone(), "depth": o["depth"].clone(),
               "normal": o["normal_d"].clone(),
               "label": torch.as_tensor(np.concatenate([a.ravel() for a in lab]), device=dev)}
    del rt, o
    torch.cuda.synchronize()
    T = tr.Trainer.from_scene(sc, cams, targets, tr.TrainConfig(prune_every=0), device=dev)
    del sc, tsc
    T.step()                              # sizes the instance capacity (one read-back)
    torch.cuda.synchronize()

    def body():
        T.forward(readback=False)
        T.loss()
        T.backward()
        T.adam()

    side = torch.cuda.Stream(device=dev)
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        body()
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        body()
    for _ in range(args.warmup):
        g.replay()
    torch.cuda.synchronize()
    st = torch.cuda.current_stream()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    steps = max(2, min(args.steps, 5))
    e0.record(st)
    for _ in range(steps):
        g.replay()
    e1.record(st)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / steps
    s, _ = T.renderer.status()
    losses = T.losses()

    def timed(fn, reps=3):
        fn()
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(st)
        for _ in range(reps):
            fn()
        b.record(st)
        torch.cuda.synchronize()
        return a.elapsed_time(b) / reps

    adam_ms = timed(T.adam)
    loss_ms = timed(T.loss)
    adam_bytes = 0
    for name in tr.PARAMS:
        cnt = T.raw[name].numel()
        extra = 4 if name in ("log_scale", "logit_opacity") else (2 if name in ("sh", "sem") else 0)
        adam_bytes += cnt * (16 + 12 + extra)
    P = T.renderer.n_pixels
    C = T.scene.n_sem
    loss_bytes = P * (2 * 4 * (8 + C) + 2 * 4 * 8 + 4 * (8 + C))
    hbm = float(peaks.get("hbm_gbs", 6800.0))
    views = len(cams)
    res = {"workload": f"{args.train_gauss // 1_000_000}M-Gaussian synthetic room, 8 orbit views "
                       "at 1920x1080, 64 logits, BF16 feature copies, FP32 masters",
           "ms_per_step": ms, "steps_per_s": 1000.0 / ms, "views_per_s": views * 1000.0 / ms,
           "status": int(s), "loss": losses,
           "adam": {"ms": adam_ms, "bytes": adam_bytes, "achieved_gbs": adam_bytes / adam_ms / 1e6,
                    "frac_of_hbm": adam_bytes / adam_ms / 1e6 / hbm},
           "loss_kernels": {"ms": loss_ms, "bytes": loss_bytes,
                            "achieved_gbs": loss_bytes / loss_ms / 1e6,
                            "frac_of_hbm": loss_bytes / loss_ms / 1e6 / hbm},
           "steps": steps, "path": "one CUDA graph per step (prune every 3000 steps, outside)"}
    del g, T
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return res


class OracleSampler:
    """The FP64 oracle, as it stands, on view 0 of the benchmark workload, in
    bounded steps.  The per-view fixed work (the float32 binning recipe, the
    preprocess of all Gaussians and its backward) is timed once; one step is
    the forward + backward of the tile composite over a band of ``n_tiles``
    tiles around the image centre, back to the per-Gaussian quantities.  A
    whole view is extrapolated as fixed + step * tiles_per_view / n_tiles."""

    def __init__(self, n_tiles: int):
        import numpy as np
        import torch

        import oracle
        from oracle import raster as orr
        from paper_2510_12174_gb300 import scenes

        self.cores = os.cpu_count() or 1
        torch.set_num_threads(self.cores)
        sc, cams = scenes.config3_orbit(N_VIEWS, n=N_GAUSS, feat_bf16=True)
        self.cam = cams[0]
        up = scenes.upstream_grads([self.cam], sc.n_sem, seed=5)
        self.up = {k: torch.as_tensor(np.asarray(up[k][0], dtype=np.float64)) for k in up}
        TX = (self.cam.width + 15) // 16
        TY = (self.cam.height + 15) // 16
        self.tiles_per_view = TX * TY
        row = TY // 2
        self.tiles = [row * TX + (TX // 2 - n_tiles // 2) + j for j in range(n_tiles)]
        t0 = time.perf_counter()
        self.binning = oracle.bin_cameras_fast(sc, [self.cam])
        params = orr.Params.from_scene(sc, requires_grad=True)
        prep = orr.preprocess(params, self.cam)
        t1 = time.perf_counter()
        # backward of the preprocess: every per-Gaussian quantity gets an
        # upstream gradient, as after a full-view composite
        tot = sum((x * torch.ones_like(x)).sum() for x in prep.tensors() if x.requires_grad)
        tot.backward()
        t2 = time.perf_counter()
        self.fixed_s = t2 - t0
        self.fixed_detail = {"binning_and_preprocess_s": t1 - t0, "preprocess_backward_s": t2 - t1}
        self.prep = orr.Prep(*[x.detach().clone().requires_grad_(True) for x in prep.tensors()])
        self.orr = orr

    def step(self) -> float:
        """Forward + backward of the tile band; returns the wall seconds."""
        import torch
        t0 = time.perf_counter()
        pd = self.prep
        for x in pd.tensors():
            x.grad = None
        r = self.orr.render_camera(pd, self.cam, self.binning, 0, tiles=self.tiles)
        tot = torch.zeros((), dtype=torch.float64)
        for key, name in (("rgb", "rgb"), ("depth", "depth"), ("normal", "normal_g"),
                          ("kmap", "kmap"), ("logits", "logits")):
            tot = tot + (r[key] * self.up[name]).sum()
        tot.backward()
        return time.perf_counter() - t0

    def per_view_s(self, step_s: float) -> float:
        return self.fixed_s + step_s * self.tiles_per_view / len(self.tiles)

    def describe(self, step_s: float, steps: int) -> dict:
        return {"kind": "oracle", "cores": self.cores,
                "sample": f"FP64 oracle on view 0 (1280x720) of the workload: binning, "
                          f"preprocess and its backward once ({self.fixed_s:.1f} s), then "
                          f"{steps} step(s) of forward + backward over {len(self.tiles)} of "
                          f"{self.tiles_per_view} tiles ({step_s:.2f} s each); a view is "
                          f"extrapolated by tile count",
                "fixed_s": self.fixed_s, "fixed_detail": self.fixed_detail,
                "step_s": step_s, "tiles_per_step": len(self.tiles),
                "tiles_per_view": self.tiles_per_view, "extrapolated": True}


def cpu_baseline(n_tiles: int, steps: int = 3):
    """The oracle on a bounded sample of the workload (about 10-30 s of CPU)."""
    smp = OracleSampler(n_tiles)
    ts = sorted(smp.step() for _ in range(steps))
    step_s = ts[len(ts) // 2]
    d = smp.describe(step_s, steps)
    d.update({"value": 1.0 / smp.per_view_s(step_s), "unit": "views/s"})
    return d


def run_reference(args):
    """The reference arm: the FP64 oracle on the host cores.  Every step is
    one bounded sample (the tile band of OracleSampler); ms_per_step is its
    measured wall time, and ``value`` the views/s that the sampled rate
    extrapolates to."""
    world, rank = _dist()
    if rank != 0:
        return
    t_start = time.perf_counter()
    smp = OracleSampler(args.cpu_tiles)
    for _ in range(args.warmup):
        smp.step()
    ts = [smp.step() for _ in range(max(1, args.steps))]
    step_s = statistics.median(ts)
    v = 1.0 / smp.per_view_s(step_s)
    cb = smp.describe(step_s, len(ts))
    cb["value"] = v
    cb["unit"] = "views/s"
    line = {"impl": "reference", "metric": METRIC, "value": v, "unit": "views/s",
            "n_gpus": world, "steps": len(ts), "warmup": args.warmup,
            "ms_per_step": step_s * 1000.0, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": workload_config(),
            "cpu_baseline": cb,
            "e2e": {"value": v, "unit": "views/s", "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0},
            "views_per_step": v * step_s,
            "wall_s": time.perf_counter() - t_start}
    print(json.dumps(line), flush=True)


def run_profile_case(args):
    """A small case of the benchmark's kernels for ncu captures: the same
    room scene with --n-gauss Gaussians seen by --views orbit views at
    1280x720 (BF16 features, 64 logits), three warm-up steps and --steps
    steps of forward + normal from depth + backward, called directly (no
    graph), so that each kernel launches once per step.  Prints the work
    counters of the step (pairs evaluated / blended, instances), which turn
    the FP32 instruction counters of one launch into flops per pair."""
    import torch

    import __graft_entry__ as ge
    from paper_2510_12174_gb300 import rasterizer as rz
    from paper_2510_12174_gb300 import scenes

    ge.build()
    dev = torch.device("cuda", 0)
    torch.cuda.set_device(dev)
    sc, cams = scenes.config3_orbit(args.views, n=args.n_gauss, feat_bf16=True)
    r = rz.Renderer(rz.DeviceScene.from_scene(sc, device=dev, feat_bf16=True), cams)
    out = r.forward()
    torch.cuda.synchronize()
    up = _device_upstream(r, sc.n_sem, 5, dev)
    grads = r.alloc_grads()
    gbuf = torch.empty(r.n_pixels, device=dev)
    for _ in range(3 + args.steps):
        r.forward(out)
        r.backward(out, up, grads=grads, g_depth_buf=gbuf)
    torch.cuda.synchronize()
    n_eval, n_blend = r.stats()
    print(json.dumps({"profile_case": f"{args.n_gauss} Gaussians, {args.views} orbit views at "
                                      "1280x720, 64 logits, BF16 features",
                      "pairs_evaluated": n_eval, "pairs_blended": n_blend,
                      "instances": r.last_instances, "pixels": r.n_pixels,
                      "device_bytes": torch.cuda.max_memory_allocated()}), flush=True)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--n-gauss", type=int, default=N_GAUSS)
    ap.add_argument("--cpu-tiles", type=int, default=16,
                    help="tiles per oracle sample step (reference arm and cpu_baseline)")
    ap.add_argument("--skip-per-view", action="store_true")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--skip-train", action="store_true",
                    help="leave out the training-step measurement")
    ap.add_argument("--skip-configs", action="store_true",
                    help="leave out the configuration 1, 2 and 4 measurements")
    ap.add_argument("--profile-case", action="store_true",
                    help="run the small profiling case (--n-gauss, --views) and exit")
    ap.add_argument("--views", type=int, default=4, help="views of the profiling case")
    ap.add_argument("--train-gauss", type=int, default=6_000_000)
    ap.add_argument("--simt-logits", action="store_true",
                    help="blend the logits on the FP32 pipes instead of the tensor cores")
    ap.add_argument("--batch", type=int, default=0, choices=[0, 8, 16, 32, 64],
                    help="Gaussians staged per batch by the composites (0: library default)")
    ap.add_argument("--ctas", type=int, default=0,
                    help="persistent composite CTAs per SM (0: library default)")
    ap.add_argument("--batch-fwd", type=int, default=0, choices=[0, 16, 32, 64],
                    help="forward composite batch (0: library default)")
    ap.add_argument("--ctas-fwd", type=int, default=0,
                    help="forward composite CTAs per SM (0: library default)")
    ap.add_argument("--tile", default="16x16",
                    help="tile shape WxH of the binning and the composites "
                         "(16x16, 8x32, 32x8 or 64x4)")
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    if args.profile_case:
        run_profile_case(args)
    elif args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
