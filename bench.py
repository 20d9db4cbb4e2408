#!/usr/bin/env python
"""Frame-rate benchmark of the 4D-GS per-frame render path on GB300.

Workload (one step = one frame = one pass of the whole path): the D-NeRF-shaped
synthetic object -- N=100k Gaussians from a 32-component mixture in the unit
sphere, SH degree 3, HexPlane spatial {64,128} x temporal 25 x 32 features, MLP
width 64 -- rendered at 800x800 from 50 hemisphere cameras x 20 timestamps in
[0,1] (view i = camera i % 50, timestamp (i // 50) % 20).  The scene stays
resident in HBM; each timed frame uploads its camera and t, then replays one
captured CUDA graph of deform -> project -> depth sort -> tile binning (gather,
column and row bits, lists) -> composite.  L2 is flushed (a 256 MB device write) before every timed frame, and
the flush is outside the timed interval.

Prints ONE JSON line (rank 0).  --impl reference times the FP64 CPU oracle on
the host cores instead.  Under torchrun (N>1) every rank renders its own views
(independent replicas, weak scaling); the timing is the max over ranks.
"""
import argparse
import json
import os
import statistics
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "FPS at 800×800/100k Gaussians (BF16 vs FP32 MLP); serving p50/p99 ms"
WIDTH = HEIGHT = 800
N_CAMS, N_TIMES = 50, 20
WORKLOAD = ("D-NeRF-shaped synthetic object: N=100k Gaussians (32-component mixture in the unit sphere), "
            "SH degree 3, HexPlane spatial {64,128} x temporal 25 x 32 features, MLP width 64, "
            "800x800, 50 hemisphere cameras (radius 4, 50 deg FOV) x 20 timestamps in [0,1]")


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=2000)
    ap.add_argument("--warmup", type=int, default=50)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--prec", default="auto", choices=["auto", "fp32", "bf16"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-serving", action="store_true")
    ap.add_argument("--no-training", action="store_true")
    ap.add_argument("--no-stress", action="store_true")
    ap.add_argument("--no-extensions", action="store_true")
    ap.add_argument("--sort-pairs", type=int, default=0,
                    help="instead of the frame benchmark: time fs4d_sort_pairs on this many random pairs")
    ap.add_argument("--sort-bits", type=int, default=13)
    ap.add_argument("--e2e-steps", type=int, default=500)
    return ap.parse_args()


_VIEWS = None


def views(step: int, rank: int, world: int):
    """View `step` of this rank: camera (step*world+rank) % 50, timestamp index
    ((step*world+rank) // 50) % 20.  The camera list is built once."""
    global _VIEWS
    if _VIEWS is None:
        from paper_2310_08528_gb300 import scenegen as sg
        _VIEWS = (sg.hemisphere_cameras(N_CAMS, width=WIDTH, height=HEIGHT, seed=0), np.linspace(0.0, 1.0, N_TIMES))
    cams, ts = _VIEWS
    i = step * world + rank
    return cams[i % N_CAMS], float(ts[(i // N_CAMS) % N_TIMES])


def max_over_ranks(dist, value: float, device) -> float:
    """The slowest replica's time: every rank renders its own views (weak scaling)
    and the job ends when the last one does.  `dist` is None on one GPU; with a
    process group the value is all-reduced (MAX) and the ranks leave together."""
    if dist is None:
        return value
    import torch
    t = torch.tensor([value], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    dist.barrier()
    return float(t.item())


# ----------------------------------------------------------------- clocks

class ClockSampler:
    """nvidia-smi clocks and throttle reasons, sampled every 20 ms while running."""

    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
              "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
              "clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.lines = []

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "20"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except OSError:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def __exit__(self, *exc):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self):
        sm, mx, reasons = [], [], set()
        names = ("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap")
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 8:
                continue
            try:
                sm.append(float(parts[0]))
                mx.append(float(parts[1]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[4:8]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": [], "samples": 0}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
                "samples": len(sm)}


# ----------------------------------------------------------------- roofline

def load_peaks(sms: int = 152):
    """Roofline denominators: the measured copy bandwidth and bf16 GEMM rate of this
    pool's GB300s when present, else the fallback figures; sms = the device's SM count."""
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        d = json.load(open(p))
        return {"hbm_gbs": d["hbm_gbs"], "bf16_tflops": d["bf16_tflops"],
                "bf16_tflops_sustained": d.get("bf16_tflops_sustained"), "sm_max_mhz": d.get("sm_max_mhz", 2070.0),
                "sms": sms, "source": "measured"}
    return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0, "sm_max_mhz": 2070.0,
            "sms": sms, "source": "fallback"}


def stage_work(stage: str, n: int, K: int, pixels: int, passes: int, prec: str, evals: int = 0,
               bitmap: bool = True, visited: int = None, direct: bool = False):
    """Algorithmic bytes or FLOPs of one frame's launches of each stage (per-unit
    figures times the units processed).  Returns a list of (bound, work, unit);
    the first entry is the stage's primary bound; an empty list: the stage does
    no work of its own.  visited: tile pairs the compositing must read (each
    tile's list up to its last contributing Gaussian); direct: a frame composited
    straight from the depth order (its bands share one projection and one depth order)."""
    if stage == "deform":
        flops = 2 * (64 * 64 + 64 * 64 + 3 * 64 * 64 + 64 * 10) * n   # MLP contraction, 42,240 FLOP/Gaussian
        return [(("tensor" if prec == "bf16" else "alu"), flops, "FLOP"), ("hbm", 80 * n, "B")]
    if stage == "project":
        # read: mean, quaternion, log-scale, opacity logit, 48 SH floats; written: xy, conic + opacity,
        # rgb, depth, radius, tile rectangle, depth-sort key and index
        return [("hbm", n * (12 + 16 + 12 + 4 + 48 * 4) + n * (8 + 16 + 12 + 4 + 4 + 16 + 4 + 4), "B")]
    if stage == "depth_sort":
        # 4 passes over 32-bit keys, each reading and writing an 8 B key and a 4 B index per Gaussian
        return [("hbm", 4 * n * 24, "B")]
    if stage == "binning":
        if direct:
            # pairs per band: radius, rect, y parts per Gaussian
            return [("hbm", n * (4 + 16 + 8), "B")]
        if bitmap:
            # tile lists: order + rect + 36 B of projected data in, the same but the order out in rank
            # order per Gaussian; a 4 B rank out per pair
            return [("hbm", n * (4 + 52 + 52) + K * 4, "B")]
        # emission: order, rect, depth in + offset out per Gaussian; one 8 B (tile | index) word per pair
        # out (frames that keep no backward state sort these words without a value array)
        return [("hbm", n * (4 + 16 + 4 + 4) + K * 8, "B")]
    if stage == "sort":
        if direct:
            # column and row bits: order, radius, rect, y parts, xy, conic + opacity, rgb in and 40 B out in
            # rank order per Gaussian
            return [("hbm", n * (4 + 4 + 16 + 8 + 8 + 16 + 12 + 40), "B")]
        if bitmap:
            return []  # no pair sort: the column and row bits give each tile's Gaussians in depth order
        return [("hbm", passes * K * 16, "B")]                         # read + write 8 B per pair per pass
    if stage == "composite":
        # gather (idx + xy, conic/opacity, rgb) per visited pair and the rgb write per pixel; ~15 FLOP per
        # tested (pixel, Gaussian) up to each pixel's last contributor
        v = K if visited is None else visited
        return [("hbm", v * 40 + pixels * 12, "B"), ("alu", 15 * evals, "FLOP")]
    raise KeyError(stage)


def _frac(bound, work, sec, peaks):
    if bound == "hbm":
        ach, peak, u = work / sec / 1e9, peaks["hbm_gbs"], "GB/s"
    elif bound == "tensor":
        ach, peak, u = work / sec / 1e12, peaks["bf16_tflops"], "TFLOP/s"
    else:  # float32 FMA pipe: SMs x 128 lanes x 2 FLOP x max SM clock
        ach, peak, u = work / sec / 1e12, peaks["sms"] * 128 * 2 * peaks["sm_max_mhz"] * 1e6 / 1e12, "TFLOP/s"
    return {"bound": bound, "achieved": ach, "peak": peak, "unit": u, "frac": ach / peak}


SINGLE_KERNEL = {"deform": "deform_tc_kernel / deform_fp32_kernel", "project": "project_kernel",
                 "composite": "composite_kernel"}
FUSED = {"sort": "tile lists from column and row bits: no pair sort (the binning stage lists each tile in depth order)"}


def visited_pairs(torch, nc, tile: int = 16) -> int:
    """Tile pairs the compositing must read: per tile, its list up to the last
    contributing Gaussian of any of its pixels (nc = last contributor per pixel)."""
    H, W = nc.shape
    ty, tx = (H + tile - 1) // tile, (W + tile - 1) // tile
    pad = torch.zeros((ty * tile, tx * tile), dtype=nc.dtype, device=nc.device)
    pad[:H, :W] = nc
    return int(pad.view(ty, tile, tx, tile).amax(dim=(1, 3)).sum().item())


def roofline(stage_ms, n, K, pixels, passes, prec, peaks, evals, bitmap=True, visited=None, direct=False):
    out = {}
    for st, ms in stage_ms.items():
        work = stage_work(st, n, K, pixels, passes, prec, evals, bitmap, visited, direct)
        if not work:
            out[st] = {"ms": ms, "fused": FUSED[st]}
            continue
        items = [_frac(b, w, ms * 1e-3, peaks) for b, w, _ in work]
        best = max(items, key=lambda r: r["frac"]) if st == "composite" else items[0]
        out[st] = dict(best, ms=ms)
        if len(items) > 1:
            out[st]["also"] = [r for r in items if r is not best]
    return out


# ----------------------------------------------------------------- CPU oracle

def cpu_baseline(budget_s: float = 12.0, max_frames: int = 40):
    import oracle
    from paper_2310_08528_gb300 import scenegen as sg
    threads = os.cpu_count() or 1
    oracle.set_threads(threads)
    scene = sg.make_object(0)
    n = 0
    t0 = time.perf_counter()
    while n < max_frames:
        cam, t = views(n, 0, 1)
        oracle.render(scene, cam, t)
        n += 1
        if time.perf_counter() - t0 > budget_s:
            break
    dt = time.perf_counter() - t0
    return {"value": n / dt, "unit": "frames/s", "cores": threads, "kind": "oracle",
            "sample": f"{n} full 800x800 frames of the 100k-Gaussian object (FP64 C++ oracle, OpenMP over "
                      f"{threads} host threads), {dt:.1f} s"}


def run_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    import oracle
    from paper_2310_08528_gb300 import scenegen as sg
    threads = os.cpu_count() or 1
    oracle.set_threads(threads)
    scene = sg.make_object(0)
    for i in range(min(args.warmup, 3)):
        cam, t = views(i, 0, 1)
        oracle.render(scene, cam, t)
    budget = 60.0
    n, t0 = 0, time.perf_counter()
    while n < args.steps:
        cam, t = views(n, 0, 1)
        oracle.render(scene, cam, t)
        n += 1
        if time.perf_counter() - t0 > budget:
            break
    dt = time.perf_counter() - t0
    fps = n / dt
    sample = (f"{n} of {args.steps} requested frames (full 800x800 frames; capped at {budget:.0f} s), "
              f"FP64 C++ oracle on {threads} host threads")
    line = {"impl": "reference", "metric": METRIC, "value": fps, "unit": "frames/s", "n_gpus": args.gpus,
            "steps": n, "warmup": min(args.warmup, 3), "ms_per_step": 1e3 * dt / n, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": WORKLOAD, "l2": "n/a (host)"},
            "cpu_baseline": {"value": fps, "unit": "frames/s", "cores": threads, "kind": "oracle", "sample": sample},
            "e2e": {"value": fps, "unit": "frames/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


# ----------------------------------------------------------------- serving

SERVE_RES = ((400, 400), (800, 800), (1352, 1014), (1920, 1080))


def random_camera(rng, w, h):
    from paper_2310_08528_gb300 import scenegen as sg
    az = rng.uniform(0, 2 * np.pi)
    z = rng.uniform(0.05, 0.9)
    r = np.sqrt(1 - z * z)
    eye = (4 * r * np.cos(az), 4 * r * np.sin(az), 4 * z)
    return sg.look_at(eye, (0.0, 0.0, 0.0), (0.0, 0.0, 1.0), w, h, 50.0)


def training_bench(ctx, fs4d, torch, sid, scene, stream, steps=10, warmup=3):
    """The backward row: one training view at 800x800 / 100k = a forward that keeps its state
    (fs4d_render with a saved frame) + fs4d_render_backward of a dense dL/dI into every parameter
    group, timed with CUDA events on the context's stream (FP32 arithmetic in both)."""
    try:
        shapes = {"means": scene.means.shape, "log_scales": scene.log_scales.shape, "quats": scene.quats.shape,
                  "opacity_logits": scene.opacity_logits.shape, "sh": scene.sh.shape, "planes": scene.planes.shape,
                  "mlp": scene.mlp.shape}
        g = {k: torch.zeros(v, device="cuda") for k, v in shapes.items()}
        dl = torch.randn((HEIGHT, WIDTH, 3), device="cuda", generator=torch.Generator("cuda").manual_seed(0))
        fwd, bwd, parts = [], [], []
        with torch.cuda.stream(stream):
            for i in range(warmup + steps):
                cam, t = views(i, 0, 1)
                e0, e1, e2 = (torch.cuda.Event(enable_timing=True) for _ in range(3))
                e0.record(stream)
                _, frame = ctx.render_saved(sid, cam, t, fs4d.FP32)
                e1.record(stream)
                ctx.render_backward(frame, dl, g)
                e2.record(stream)
                ctx.frame_free(frame)
                stream.synchronize()
                if i >= warmup:
                    fwd.append(e0.elapsed_time(e1))
                    bwd.append(e1.elapsed_time(e2))
            # per-kernel times of the backward, from a separate timed pass
            ctx.set_stage_timing(True)
            for i in range(3):
                cam, t = views(i, 0, 1)
                _, frame = ctx.render_saved(sid, cam, t, fs4d.FP32)
                ctx.render_backward(frame, dl, g)
                parts.append(ctx.backward_times())
                ctx.frame_free(frame)
            ctx.set_stage_timing(False)
        f, b = float(np.median(fwd)), float(np.median(bwd))
        per = {k: float(np.median([p[k] for p in parts])) for k in parts[0]}
        return {"workload": "one view of the 800x800 / 100k object, dL/dI ~ N(0,1), gradients of every parameter "
                            "group", "steps": steps, "forward_saved_ms": f, "backward_ms": b, "step_ms": f + b,
                "views_per_s": 1e3 / (f + b), "backward_kernels_ms": per,
                "note": "the forward keeps the backward's state (tile lists cut to each ellipse's box, written into the frame's own buffers)"}
    except Exception as exc:  # the headline line must still be printed
        return {"error": f"{type(exc).__name__}: {exc}"}


def training_c2_bench(ctx, fs4d, torch, stream, steps=12, warmup=3):
    """Config 2's training step: the Neu3D-shaped room (300k Gaussians in a 6x4x6
    box, SH 3, HexPlane {64,128} x 150 x 32) at 1352x1014 from forward-facing
    cameras, L1 against targets rendered from the same scene with the planes
    perturbed by N(0, 0.01), BF16 forward, float32 backward, TV loss and Adam
    (fs4d_train_step), timed with CUDA events per step."""
    from paper_2310_08528_gb300 import scenegen as sg
    try:
        scene = sg.make_room(0)
        sid = ctx.load_scene(scene)
        sid_t = ctx.load_scene(sg.perturb_planes(scene, 0))
        cams = sg.forward_cameras(8, seed=0)
        ts = [float(k) / 149.0 for k in range(0, 150, 19)]
        with torch.cuda.stream(stream):
            targets = [ctx.render(sid_t, cams[i % 8], ts[i % len(ts)], fs4d.FP32) for i in range(8)]
        ctx.unload_scene(sid_t)
        tr = fs4d.Trainer(ctx, sid, warmup + steps)
        ms, l1s = [], []
        losses = torch.zeros(2, device="cuda")
        with torch.cuda.stream(stream):
            for i in range(warmup + steps):
                e0, e1 = _events(torch)
                e0.record(stream)
                tr.step(cams[i % 8], ts[i % len(ts)], targets[i % 8], fs4d.BF16, losses)
                e1.record(stream)
                stream.synchronize()
                l1s.append(float(losses[0].item()))
                if i >= warmup:
                    ms.append(e0.elapsed_time(e1))
            ctx.set_stage_timing(True)
            tr.step(cams[0], ts[0], targets[0], fs4d.BF16, losses)
            fwd = ctx.stage_times()
            bwd = ctx.backward_times()
            ctx.set_stage_timing(False)
        tr.close()
        ctx.unload_scene(sid)
        t = float(np.median(ms))
        return {"workload": "room: N=300k (64-cluster mixture in a 6x4x6 box), SH 3, HexPlane {64,128} x 150 x 32, "
                            "1352x1014 forward-facing cameras, L1 to targets rendered with planes + N(0,0.01), "
                            "TV weight 1e-4, Adam (App. A rates)",
                "steps": steps, "step_ms": t, "steps_per_s": 1e3 / t, "forward": "bf16", "backward": "fp32",
                "l1_first": l1s[0], "l1_last": l1s[-1], "forward_stages_ms": fwd, "backward_kernels_ms": bwd}
    except Exception as exc:  # the headline line must still be printed
        return {"error": f"{type(exc).__name__}: {exc}"}


def serving_bench(ctx, fs4d, torch, rates=(500.0, 2000.0), seconds=1.5, precs=("bf16", "fp32")):
    """Continuous batching under Poisson arrivals: 8 resident scenes of 100k-500k
    Gaussians, (scene, random hemisphere camera, t ~ U[0,1]), resolution uniform
    over 400x400, 800x800, 1352x1014, 1920x1080; device-resident outputs."""
    from paper_2310_08528_gb300 import scenegen as sg
    sizes = [int(100_000 + i * 400_000 / 7) for i in range(8)]
    sids = [ctx.load_scene(sg.make_object(i, n=n)) for i, n in enumerate(sizes)]
    srv = fs4d.Server(ctx, max_inflight=8, max_batch=8, hbm_budget_bytes=24 << 30, pairs_per_gaussian=12.0)
    pool = [torch.empty(1080 * 1920 * 3, device="cuda") for _ in range(96)]
    free = list(range(len(pool)))
    busy = {}

    def reap():
        out = srv.poll(4096)
        for c in out:
            free.append(busy.pop(c["ticket"]))
        return out

    rng = np.random.default_rng(123)
    # warm-up: every (scene, resolution, precision) once, so graphs are captured
    for p in precs:
        pc = fs4d.BF16 if p == "bf16" else fs4d.FP32
        items = []
        for s in sids:
            for (w, h) in SERVE_RES:
                while not free:
                    reap()
                b = free.pop()
                items.append((s, random_camera(rng, w, h), float(rng.uniform()), pool[b][: w * h * 3], pc, b))
        for it in items:
            tk = srv.submit(*it[:5])
            busy[tk] = it[5]
            while not free:
                reap()
        srv.drain()
        reap()
    results = {}
    for p in precs:
        pc = fs4d.BF16 if p == "bf16" else fs4d.FP32
        for rate in rates:
            lat, done_all = [], []
            n_req = int(rate * seconds)
            gaps = rng.exponential(1.0 / rate, n_req)
            t0 = time.perf_counter()
            due = t0
            for i in range(n_req):
                due += gaps[i]
                s = sids[int(rng.integers(0, len(sids)))]
                w, h = SERVE_RES[int(rng.integers(0, 4))]
                cam = random_camera(rng, w, h)
                while time.perf_counter() < due:
                    done_all += reap()
                while not free:
                    done_all += reap()
                b = free.pop()
                tk = srv.submit(s, cam, float(rng.uniform()), pool[b][: w * h * 3], pc)
                busy[tk] = b
            srv.drain()
            done_all += reap()
            wall = time.perf_counter() - t0
            ok = [c for c in done_all if c["status"] == 0]
            lat = np.array([c["done_ms"] - c["submit_ms"] for c in ok])
            span_ms = max(c["done_ms"] for c in ok) - min(c["submit_ms"] for c in ok)
            results[f"{p}@{int(rate)}"] = {
                "offered_req_s": rate, "requests": n_req, "completed": len(ok),
                "failed": len(done_all) - len(ok), "throughput_req_s": len(ok) / (span_ms * 1e-3),
                "p50_ms": float(np.percentile(lat, 50)), "p99_ms": float(np.percentile(lat, 99)),
                "mean_ms": float(lat.mean()), "wall_s": wall}
    st = srv.stats()
    srv.close()
    for s in sids:
        ctx.unload_scene(s)
    return {"workload": "8 resident scenes (object generator, seeds 0-7, N=100k..500k), Poisson arrivals, "
                        "random hemisphere camera, t~U[0,1], resolution uniform over 400x400/800x800/1352x1014/"
                        "1920x1080; latency = host submit -> completion observed by the scheduler",
            "config": {"max_inflight": 8, "max_batch": 8, "hbm_budget_gb": 24},
            "results": results,
            "server_stats": {k: int(v) for k, v in st.items()}}


# ----------------------------------------------------------------- stress workload

STRESS_RES = ((1920, 1080), (3840, 2160))
STRESS_WORKLOAD = ("stress: N=2M Gaussians (32-component mixture in the unit sphere) with log-scales N(-2.5,0.5), "
                   "SH degree 3, HexPlane spatial {64,128,256} x temporal 300 x 32 features, MLP width 64; 16 "
                   "timestamps deformed in one launch; frames at 1920x1080 and 3840x2160 from a hemisphere camera")


def _events(torch):
    return torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)


def _sort_passes(width, height, bands):
    tx, ty = (width + 15) // 16, (height + 15) // 16
    tiles = tx * ((ty + bands - 1) // bands)
    return (int(np.ceil(np.log2(max(tiles, 2)))) + 7) // 8


def stress_bench(ctx, fs4d, torch, stream, peaks, frames=3):
    """The stress workload: the batched deformation of 16 timestamps (both
    precisions) and frames at 1080p and 4K.  Every input is far larger than L2
    (2M Gaussians; 1.3e9 and 5e9 tile pairs per frame), so no flush is needed.
    Frames with more pairs than one pair-sort pass counts render in bands of
    tile rows, which share one projection and one depth order."""
    from paper_2310_08528_gb300 import scenegen as sg
    try:
        scene = sg.make_stress(0)
        sid = ctx.load_scene(scene)
        n = scene.n
        ts = [float(v) for v in np.linspace(0.0, 1.0, 16)]
        dev = torch.device("cuda", torch.cuda.current_device())
        out = {"workload": STRESS_WORKLOAD, "n_gaussians": n,
               "l2": "inputs larger than L2 (no flush)", "timing": "CUDA events on the context's stream"}
        bufs = (torch.empty((16, n, 3), device=dev), torch.empty((16, n, 4), device=dev),
                torch.empty((16, n, 3), device=dev))
        deform = {}
        with torch.cuda.stream(stream):
            for p in ("bf16", "fp32"):
                pc = fs4d.BF16 if p == "bf16" else fs4d.FP32
                ctx.deform(sid, ts, pc, out=bufs)
                ms = []
                for _ in range(frames):
                    e0, e1 = _events(torch)
                    e0.record(stream)
                    ctx.deform(sid, ts, pc, out=bufs)
                    e1.record(stream)
                    stream.synchronize()
                    ms.append(e0.elapsed_time(e1))
                t = float(np.median(ms))
                work = stage_work("deform", 16 * n, 0, 0, 0, p)
                deform[p] = {"ms": t, "gaussian_timesteps_per_s": 16 * n / (t * 1e-3),
                             "roofline": _frac(work[0][0], work[0][1], t * 1e-3, peaks),
                             "streamed": _frac("hbm", work[1][1], t * 1e-3, peaks)}
        out["deform_16t"] = deform
        del bufs
        res = {}
        for (w, h) in STRESS_RES:
            cam = sg.hemisphere_cameras(4, width=w, height=h, seed=7)[1]
            image = torch.empty((h, w, 3), device=dev)
            r = {}
            with torch.cuda.stream(stream):
                for p in ("bf16", "fp32"):
                    pc = fs4d.BF16 if p == "bf16" else fs4d.FP32
                    ctx.render(sid, cam, 0.5, pc, image=image)  # finds the bands, sizes the buffers
                    ms = []
                    for i in range(frames):
                        e0, e1 = _events(torch)
                        e0.record(stream)
                        ctx.render(sid, cam, ts[(5 * i) % 16], pc, image=image)
                        e1.record(stream)
                        stream.synchronize()
                        ms.append(e0.elapsed_time(e1))
                    t = float(np.median(ms))
                    r[p] = {"ms": t, "fps": 1e3 / t, "gaussians_per_s": n / (t * 1e-3),
                            "tile_pairs": ctx.last_pairs(), "bands": ctx.last_bands()}
                ctx.set_stage_timing(True)
                _, _, nc = ctx.render(sid, cam, 0.5, fs4d.BF16, with_aux=True)
                st = ctx.stage_times()
                ctx.set_stage_timing(False)
                K, bands = ctx.last_pairs(), ctx.last_bands()
                direct = ctx.last_binning() == fs4d.BINNING_SORT  # (no lists: of AUTO's frames, these)
                vis, evals = visited_pairs(torch, nc), int(nc.sum().item())
            r["stages"] = roofline(st, n, K, w * h, _sort_passes(w, h, bands), "bf16", peaks, evals, bitmap=False,
                                   visited=vis, direct=direct)
            r["tile_pairs"], r["tile_pairs_visited"], r["bands"] = K, vis, bands
            res[f"{w}x{h}"] = r
            del image, nc
        out["frames"] = res
        ctx.unload_scene(sid)
        return out
    except Exception as exc:  # the headline line must still be printed
        return {"error": f"{type(exc).__name__}: {exc}"}


def bf16_vs_fp32(ctx, fs4d, torch, sid, scene, stream):
    """The BF16 path against the FP32 path (itself within 2e-5 of the FP64 oracle) on
    the benchmark scene: max |dX|, |dr|, |ds| of the deformation at 5 timestamps,
    and the image PSNR over 5 views."""
    ts = [0.0, 0.25, 0.5, 0.75, 1.0]
    with torch.cuda.stream(stream):
        a = ctx.deform(sid, ts, fs4d.BF16)
        b = ctx.deform(sid, ts, fs4d.FP32)
        errs = [float((x - y).abs().max().item()) for x, y in zip(a, b)]
        mse = []
        for i in range(5):
            cam, t = views(97 * i, 0, 1)
            x = ctx.render(sid, cam, t, fs4d.BF16)
            y = ctx.render(sid, cam, t, fs4d.FP32)
            mse.append(float(((x - y) ** 2).mean().item()))
    stream.synchronize()
    psnr = [float(10 * np.log10(1.0 / m)) if m > 0 else float("inf") for m in mse]
    return {"max_abs_dx": errs[0], "max_abs_dr": errs[1], "max_abs_ds": errs[2], "psnr_db_min": min(psnr),
            "psnr_db_mean": float(np.mean(psnr)), "views": 5, "timestamps": ts,
            "reference": "the FP32 path (within 2e-5 of the FP64 oracle in the parity tests)"}


# ----------------------------------------------------------------- GPU arm

def measure(ctx, fs4d, torch, sid, prec, steps, warmup, rank, world, stream, cap):
    """Graph-captured frames; returns (per-frame ms list, mean stage ms).  The
    frame rate comes from a graph captured WITHOUT the stage-timing events; the
    stage breakdown from a second graph captured with them, replayed separately."""
    dev = torch.device("cuda", torch.cuda.current_device())
    shape_cam, _ = views(0, rank, world)
    d_cam = torch.empty(23, dtype=torch.float32, device=dev)
    d_t = torch.empty(1, dtype=torch.float32, device=dev)
    image = torch.empty((HEIGHT, WIDTH, 3), device=dev)
    n_views = N_CAMS * N_TIMES
    host_cams = torch.empty((n_views, 23), dtype=torch.float32).pin_memory()
    host_ts = torch.empty((n_views, 1), dtype=torch.float32).pin_memory()
    for i in range(n_views):
        cam, t = views(i, 0, 1)
        host_cams[i] = torch.from_numpy(np.frombuffer(bytes(fs4d.camera_struct(cam)), dtype=np.float32).copy())
        host_ts[i, 0] = t
    flush = torch.empty(64 * 1024 * 1024, dtype=torch.int32, device=dev)  # 256 MB > 129 MB L2
    graphs = {}
    with torch.cuda.stream(stream):
        ctx.render_async(sid, shape_cam, d_cam, d_t, image, prec)  # warm the kernels outside the capture
        stream.synchronize()
        for timed in (False, True):
            ctx.set_stage_timing(timed)
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=stream):
                ctx.render_async(sid, shape_cam, d_cam, d_t, image, prec)
            graphs[timed] = g
        ctx.set_stage_timing(False)
    starts = [torch.cuda.Event(enable_timing=True) for _ in range(steps)]
    ends = [torch.cuda.Event(enable_timing=True) for _ in range(steps)]
    with torch.cuda.stream(stream):
        for i in range(warmup + steps):
            v = (i * world + rank) % n_views
            flush.fill_(i)
            j = i - warmup
            if j >= 0:
                starts[j].record(stream)
            d_cam.copy_(host_cams[v], non_blocking=True)
            d_t.copy_(host_ts[v], non_blocking=True)
            graphs[False].replay()
            if j >= 0:
                ends[j].record(stream)
    stream.synchronize()
    ctx.check_device_status()  # no capacity overflow and no timed-out wait in any frame
    frame_ms = [s.elapsed_time(e) for s, e in zip(starts, ends)]
    # stage breakdown on the same views, from the graph with the stage events
    stages = []
    with torch.cuda.stream(stream):
        for i in range(min(steps, 50)):
            v = (i * world + rank) % n_views
            flush.fill_(i)
            d_cam.copy_(host_cams[v], non_blocking=True)
            d_t.copy_(host_ts[v], non_blocking=True)
            graphs[True].replay()
            stages.append(ctx.stage_times())  # waits for this frame
    stream.synchronize()
    ctx.check_device_status()
    mean_st = {k: float(np.mean([s[k] for s in stages])) for k in stages[0]}
    return frame_ms, mean_st


def extensions_bench(ctx, fs4d, torch, sg, sid, scene, stream, cap, steps=300, warmup=10):
    """The rows beyond the headline frame, on the same 800x800 / 100k object:
    the colour and opacity heads (App. B) in graph-replayed frames, composition of
    two objects in one frame, a tracking batch of 16 timestamps, and one
    densification."""
    out = {}
    try:
        cid = ctx.load_scene(sg.with_color_heads(scene, 5))
        ctx.reserve(cid, WIDTH, HEIGHT, cap)
        ch = {}
        for p, pc in (("bf16", fs4d.BF16), ("fp32", fs4d.FP32)):
            ms, st = measure(ctx, fs4d, torch, cid, pc, steps, warmup, 0, 1, stream, cap)
            ch[p] = {"fps": 1e3 / float(np.mean(ms)), "p50_ms": float(np.percentile(ms, 50)),
                     "stages_ms": st}
        ch["note"] = "graph-replayed frames as in the headline; the deform stage includes the heads (FP32 SIMT)"
        out["color_heads"] = ch
        ctx.unload_scene(cid)
    except Exception as exc:
        out["color_heads"] = {"error": f"{type(exc).__name__}: {exc}"}
    try:
        oid = ctx.load_scene(sg.make_object(1))
        shifts = np.array([[-0.6, 0.0, 0.0], [0.6, 0.0, 0.0]], np.float32)
        comp = {}
        with torch.cuda.stream(stream):
            for p, pc in (("bf16", fs4d.BF16), ("fp32", fs4d.FP32)):
                for i in range(3):
                    cam, t = views(i, 0, 1)
                    ctx.render_composed([sid, oid], cam, t, pc, shifts=shifts)
                stream.synchronize()
                k = 40
                t0 = time.perf_counter()
                for i in range(k):
                    cam, t = views(i, 0, 1)
                    ctx.render_composed([sid, oid], cam, t, pc, shifts=shifts)
                stream.synchronize()
                comp[p] = {"ms_per_frame": (time.perf_counter() - t0) * 1e3 / k}
        comp["workload"] = "two 100k objects (200k Gaussians) in one 800x800 frame, eager host-synchronised calls"
        out["composition"] = comp
        trk = {}
        ts = np.linspace(0.0, 1.0, 16).astype(np.float32)
        outs = (torch.empty((16, scene.n, 3), device="cuda"), torch.empty((16, scene.n, 4), device="cuda"),
                torch.empty((16, scene.n, 3), device="cuda"))
        with torch.cuda.stream(stream):
            for p, pc in (("bf16", fs4d.BF16), ("fp32", fs4d.FP32)):
                ctx.deform(sid, ts, pc, outs)
                ms = []
                for _ in range(10):
                    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                    e0.record(stream)
                    ctx.deform(sid, ts, pc, outs)
                    e1.record(stream)
                    stream.synchronize()
                    ms.append(e0.elapsed_time(e1))
                m = float(np.median(ms))
                trk[p] = {"ms": m, "gaussian_timestamps_per_s": 16 * scene.n / (m * 1e-3)}
        trk["workload"] = "fs4d_deform of the 100k object at 16 timestamps in one call (trajectories)"
        out["tracking"] = trk
        ctx.unload_scene(oid)
    except Exception as exc:
        out["composition_tracking"] = {"error": f"{type(exc).__name__}: {exc}"}
    try:
        did = ctx.load_scene(scene)
        n = scene.n
        gen = torch.Generator("cuda").manual_seed(7)
        vis = torch.full((n,), 20.0, device="cuda")
        gsum = torch.rand(n, device="cuda", generator=gen) * 4e-3  # mean norm ~2e-4 per view
        normals = torch.randn((n, 2, 3), device="cuda", generator=gen)
        thr = float(np.quantile(np.linspace(0.0, 2e-4, 1001), 0.9))  # ~10% of the Gaussians densify
        split = float(np.quantile(scene.log_scales.max(1), 0.5))
        prune = float(np.quantile(scene.opacity_logits, 0.05))
        stream.synchronize()
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        m = ctx.densify_raw(did, (gsum, vis), normals, thr, split, prune)
        ms = (time.perf_counter() - t0) * 1e3
        out["densify"] = {"ms": ms, "n_before": n, "n_after": m,
                          "workload": "fs4d_densify of a copy of the 100k object: ~10% over the gradient "
                                      "threshold (half copied, half split), ~5% pruned; wall time of the "
                                      "call (its result size is read back once)"}
        ctx.unload_scene(did)
    except Exception as exc:
        out["densify"] = {"error": f"{type(exc).__name__}: {exc}"}
    return out


def sort_only(args):
    """Standalone radix sort of random (key, value) pairs on the low sort_bits bits
    (the pair sort of a frame sorts tile bits only: 12-15 bits).  Prints one JSON
    line with the sort's time and HBM bandwidth (24 B per pair per pass plus the
    8 B per pair histogram pass)."""
    import torch
    from paper_2310_08528_gb300 import fs4d
    n, bits = args.sort_pairs, args.sort_bits
    ctx = fs4d.Context(0)
    gen = torch.Generator("cuda").manual_seed(0)
    v = torch.arange(n, dtype=torch.int32, device="cuda")
    ms = []
    for i in range(args.warmup + args.steps):
        k = torch.randint(0, 1 << bits, (n,), dtype=torch.int64, device="cuda", generator=gen)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        ctx.sort_pairs(k, v, bits)
        e1.record()
        torch.cuda.synchronize()
        if i >= args.warmup:
            ms.append(e0.elapsed_time(e1))
    t = float(np.median(ms))
    passes = (bits + 7) // 8
    byt = passes * 24 * n + 8 * n
    peaks = load_peaks(torch.cuda.get_device_properties(0).multi_processor_count)
    print(json.dumps({"metric": "radix sort of (64-bit key, 32-bit value) pairs", "pairs": n, "key_bits": bits,
                      "ms": t, "pairs_per_s": n / (t * 1e-3), "hbm_gbs": byt / (t * 1e-3) / 1e9,
                      "hbm_frac": byt / (t * 1e-3) / 1e9 / peaks["hbm_gbs"], "steps": args.steps}), flush=True)
    ctx.close()
    return 0


def main():
    args = parse()
    if args.impl == "reference":
        return run_reference(args)
    if args.sort_pairs > 0:
        return sort_only(args)
    import torch
    from paper_2310_08528_gb300 import fs4d, scenegen as sg

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))

    scene = sg.make_object(0)
    stream = torch.cuda.Stream()
    ctx = fs4d.Context(local, stream)
    sid = ctx.load_scene(scene)
    # size the tile-pair buffers from the largest frame of the view set
    kmax = 0
    with torch.cuda.stream(stream):
        for c in range(N_CAMS):
            cam, t = views(c, 0, 1)
            ctx.render(sid, cam, t)
            kmax = max(kmax, ctx.last_pairs())
    stream.synchronize()
    cap = int(kmax * 1.25) + 4096
    ctx.reserve(sid, WIDTH, HEIGHT, cap)
    tiles = ((WIDTH + 15) // 16) * ((HEIGHT + 15) // 16)
    passes = (int(np.ceil(np.log2(tiles))) + 7) // 8   # the pair sort keys on the tile bits only
    bitmap = ctx.last_binning() == fs4d.BINNING_BITMAP
    # (pixel, Gaussian) tests the compositing must make: each pixel walks its tile's list up to its
    # last contributor (summed over the frames of the view set)
    evals, pairs, visited = [], [], []
    with torch.cuda.stream(stream):
        for c in range(0, N_CAMS * N_TIMES, 97):
            cam, t = views(c, 0, 1)
            _, _, nc = ctx.render(sid, cam, t, with_aux=True)
            evals.append(int(nc.sum().item()))
            visited.append(visited_pairs(torch, nc))
            pairs.append(ctx.last_pairs())
    evals, mean_pairs, visited = int(np.mean(evals)), int(np.mean(pairs)), int(np.mean(visited))

    bf16_ok = True
    try:
        with torch.cuda.stream(stream):
            ctx.render(sid, views(0, 0, 1)[0], 0.5, fs4d.BF16)
        stream.synchronize()
    except fs4d.Fs4dError:
        bf16_ok = False
    precs = ["fp32"] + (["bf16"] if bf16_ok else [])
    head = args.prec if args.prec != "auto" else ("bf16" if bf16_ok else "fp32")
    if head == "bf16" and not bf16_ok:
        raise SystemExit("bf16 requested but the BF16 path is not available for this scene")

    # kernels of one graph-replayed frame, as the library counts them for the same call
    # (deform, project, the depth sort, then lists: gather, bits, lists, or sort: emission,
    # tile scan, pair-sort passes; then composite)
    launches = {}
    with torch.cuda.stream(stream):
        dev = torch.device("cuda", torch.cuda.current_device())
        shape_cam, t0 = views(0, 0, 1)
        d_cam = torch.from_numpy(np.frombuffer(bytes(fs4d.camera_struct(shape_cam)), dtype=np.float32).copy()).to(dev)
        d_t = torch.full((1,), t0, dtype=torch.float32, device=dev)
        img = torch.empty((HEIGHT, WIDTH, 3), device=dev)
        for p in precs:
            ctx.render_async(sid, shape_cam, d_cam, d_t, img, fs4d.BF16 if p == "bf16" else fs4d.FP32)
            launches[p] = ctx.last_launches()
    stream.synchronize()

    results = {}
    clocks = None
    for p in precs:
        pc = fs4d.BF16 if p == "bf16" else fs4d.FP32
        if dist:
            dist.barrier()
        torch.cuda.synchronize()
        if p == head:
            with ClockSampler(local) as cs:
                frame_ms, st = measure(ctx, fs4d, torch, sid, pc, args.steps, args.warmup, rank, world, stream, cap)
            clocks = cs.summary()
        else:
            frame_ms, st = measure(ctx, fs4d, torch, sid, pc, args.steps, args.warmup, rank, world, stream, cap)
        torch.cuda.synchronize()
        total = max_over_ranks(dist, float(np.sum(frame_ms)), "cuda")
        results[p] = {"fps": world * args.steps / (total * 1e-3), "ms_per_step": total / args.steps,
                      "gaussians_per_s": scene.n * world * args.steps / (total * 1e-3),
                      "p50_ms": float(np.percentile(frame_ms, 50)), "p99_ms": float(np.percentile(frame_ms, 99)),
                      "stages_ms": st}

    # end-to-end through the batched host-buffer C call (cameras in, every frame's image out to host
    # memory, copies inside the timed region, each overlapped with the next frame's render)
    e2e_steps = min(args.e2e_steps, args.steps)
    pc = fs4d.BF16 if head == "bf16" else fs4d.FP32
    host_imgs = [torch.empty((HEIGHT, WIDTH, 3), dtype=torch.float32).pin_memory().numpy() for _ in range(2)]
    e2e_views = [views(i, rank, world) for i in range(e2e_steps)]
    e2e_cams, e2e_ts = [v[0] for v in e2e_views], [v[1] for v in e2e_views]
    e2e_outs = [host_imgs[i & 1] for i in range(e2e_steps)]
    with torch.cuda.stream(stream):
        ctx.render_host_batch(sid, e2e_cams[:3], e2e_ts[:3], pc, e2e_outs[:3])
        if dist:
            dist.barrier()
        t0 = time.perf_counter()
        ctx.render_host_batch(sid, e2e_cams, e2e_ts, pc, e2e_outs)
        e2e_s = time.perf_counter() - t0
    e2e_s = max_over_ranks(dist, e2e_s, "cuda")

    if rank != 0:
        if dist:
            dist.destroy_process_group()
        return 0

    peaks = load_peaks(torch.cuda.get_device_properties(local).multi_processor_count)
    K = mean_pairs
    rf = roofline(results[head]["stages_ms"], scene.n, K, WIDTH * HEIGHT, passes, head, peaks, evals, bitmap,
                  visited)
    # the dominant KERNEL: the longest single-kernel stage (the binning stage is a chain of
    # depth-sort passes and binning kernels, reported under "stages")
    dom = max((k for k in rf if "frac" in rf[k] and k in SINGLE_KERNEL), key=lambda k: rf[k]["ms"])
    traffic = None
    tf = os.path.join(ROOT, "profiles", "traffic.json")
    if os.path.exists(tf):
        tr = json.load(open(tf)).get(head, {}).get(dom)
        if tr:
            traffic = tr.get("bytes_per_launch")
    line = {
        "metric": METRIC, "value": results[head]["fps"], "unit": "frames/s", "n_gpus": world, "steps": args.steps,
        "gaussians_per_s": results[head]["gaussians_per_s"],
        "warmup": args.warmup, "ms_per_step": results[head]["ms_per_step"], "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "bf16" if head == "bf16" else "f32", "data": "synthetic",
        "config": {"workload": WORKLOAD, "n_gaussians": scene.n, "resolution": [WIDTH, HEIGHT],
                   "binning": "tile lists from column and row bits" if bitmap else "radix sort",
                   "tile_pairs_mean": K, "tile_pairs_visited_mean": visited, "pixel_gaussian_tests_mean": evals, "pair_capacity": cap, "parallelism": f"replicas x{world}",
                   "l2": "flushed before every timed frame (256 MB device write, outside the timed interval)",
                   "timing": "CUDA events around camera upload + CUDA-graph replay of one frame (graph without "
                             "the stage-timing events; stages from a second graph replayed separately)"},
        "roofline": {"kernel": SINGLE_KERNEL[dom], "stage": dom, "bound": rf[dom]["bound"], "achieved": rf[dom]["achieved"], "peak": rf[dom]["peak"],
                     "unit": rf[dom]["unit"], "frac": rf[dom]["frac"], "traffic": traffic,
                     "peak_source": peaks["source"]},
        "stages": rf,
        "fp32_fps": results.get("fp32", {}).get("fps"),
        "precisions": results,
        "e2e": {"value": e2e_steps * world / e2e_s, "unit": "frames/s", "h2d_bytes_per_step": 96,
                "d2h_bytes_per_step": WIDTH * HEIGHT * 12 + 8,
                "call": "fs4d_render_host_batch (host cameras in, every frame's image out to pinned host "
                        "memory, copies overlapped with the next frame's render; one call for all steps)"},
        "gpu_launches": launches[head] * args.steps,  # the timed region of `value`
        "launches_per_frame": launches,
        "clocks": clocks,
    }
    if bf16_ok:
        line["bf16_vs_fp32"] = bf16_vs_fp32(ctx, fs4d, torch, sid, scene, stream)
    if not args.no_training:
        line["training"] = training_bench(ctx, fs4d, torch, sid, scene, stream)
        line["training_c2"] = training_c2_bench(ctx, fs4d, torch, stream)
    if not args.no_serving:
        line["serving"] = serving_bench(ctx, fs4d, torch)
    if not args.no_stress:
        line["stress"] = stress_bench(ctx, fs4d, torch, stream, peaks)
    if not args.no_extensions:
        line["extensions"] = extensions_bench(ctx, fs4d, torch, sg, sid, scene, stream, cap)
    if world == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline()
    print(json.dumps(line), flush=True)
    if dist:
        dist.destroy_process_group()
    return 0


if __name__ == "__main__":
    sys.exit(main())
