#!/usr/bin/env python
"""Throughput of the compositional sparse-voxel rasterizer on one GB300.

A step is one pass of the whole hot path over one frame of the compositional
workload (500k-leaf LiDAR-shaped background + 3 actors of 20k leaves, SH degree
3, one 1920x1080 camera): forward render through the C ABI, then the backward
replay for a fixed upstream gradient.  The metric is rendered megapixels per
second, fwd+bwd (``value``); the forward alone is reported beside it.

Timing: W untimed warm-up steps, then K steps, each bracketed by CUDA events on
the rendering stream with an L2 flush (a 512 MB write) between steps outside
the events; barrier + synchronize around the timed loop; max over ranks.
Inside the timed loop the library brackets only the dominant stage with
events (its live duration gives the roofline); the per-stage table comes from
a separate run before it with every stage bracketed, so that the headline
carries no instrumentation of the other stages.
``e2e`` repeats the step through the public API with the upstream gradient
copied from pinned host memory and every result (images and gradients) copied
back each step.  ``cpu_baseline`` times the FP64 oracle on a bounded pixel
sample of the same frame on the host cores.

``--impl reference`` runs the oracle as the reference arm (no GPU work).
Under torchrun every rank renders its own frame (weak scaling, no collective).
"""
import argparse
import hashlib
import json
import math
import os
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

MEASURED_PEAKS = os.path.join(ROOT, "MEASURED_PEAKS.json")
TRAFFIC = os.path.join(ROOT, "profiles", "traffic.json")
METRIC = "Mpix/s fwd & fwd+bwd; served p50/p99 latency vs plain path, 1 GB300"
WORKLOAD = ("compositional fwd+bwd: LiDAR-shaped background 500k leaves (levels 6-12, 200 m root) + 3 actors x "
            "20k leaves on straight lanes, SH degree 3, one 1920x1080 camera, K=1, eps_stop=1e-4")

# Algorithmic FP32 operations per unit of the method (FMA = 2, exponential = 1), not counted from the
# kernels: a ray-box slab test 20 (per pixel x listed voxel, and per pixel x actor clip box); per
# composited segment K samples of 31 (position, trilinear interpolation of 8 corners, activation)
# plus 16 (alpha, transmittance, the colour and depth accumulation).  The backward replays the
# forward's arithmetic (it needs every segment's transmittance and prefix sums) and adds, per sample,
# 35 (the 8 trilinear weights, the activation's derivative, d tau / d corner) and per segment 43
# (dL/d tau from the upstream gradients and the suffix sums, the chain to the 8 corners and the 3
# colour channels, and the 11 additions into the per-voxel gradient sums).
F_TEST = 20
F_BOX = 20
F_SAMPLE = 31
F_SEG = 16
F_SAMPLE_BWD = F_SAMPLE + 35
F_SEG_BWD = F_SEG + 43


def log(*a):
    print(*a, file=sys.stderr, flush=True)


def parse():
    p = argparse.ArgumentParser()
    p.add_argument("--gpus", type=int, default=1)
    p.add_argument("--steps", type=int, default=200)
    p.add_argument("--warmup", type=int, default=10)
    p.add_argument("--impl", choices=("ours", "reference"), default="ours")
    p.add_argument("--no-e2e", action="store_true")
    p.add_argument("--core-only", action="store_true",
                   help="time only the rendering path: skip the normals, sky, feature-field and initialisation sections")
    p.add_argument("--no-cpu-baseline", action="store_true")
    p.add_argument("--cpu-seconds", type=float, default=12.0, help="target CPU work of the oracle sample")
    p.add_argument("--seed", type=int, default=0)
    p.add_argument("--no-serving", action="store_true")
    p.add_argument("--serve-seconds", type=float, default=2.0, help="arrival window per rate and path")
    p.add_argument("--serve-min-requests", type=int, default=1000,
                   help="requests per rate at least (the window grows for low rates), so p99 rests on >= 10 tail samples")
    p.add_argument("--serve-rates", default="200,500,1000,2000")
    p.add_argument("--profile-pass", action="store_true",
                   help="no timing: one warm-up and one profiled pass of every row on the 1080p frame, for a "
                        "counter capture (prints the library's launch counts of both passes)")
    p.add_argument("--traffic-from", default=None,
                   help="build profiles/traffic.json and a table from an ncu --csv capture of --profile-pass")
    p.add_argument("--large", default="cfg3,cfg5",
                   help="larger scenes timed after the headline (comma list of cfg3, cfg5; empty: none)")
    return p.parse_args()


def dist_env():
    return int(os.environ.get("RANK", 0)), int(os.environ.get("WORLD_SIZE", 1)), int(os.environ.get("LOCAL_RANK", 0))


def max_over_ranks(values, world, device="cpu"):
    """Per-rank timings -> their maximum over all ranks (the job is as slow as its slowest rank)."""
    import torch
    t = torch.tensor([float(v) for v in values], dtype=torch.float64, device=device)
    if world > 1:
        import torch.distributed as dist
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return [float(x) for x in t]


def whole_job_mpix_s(world, pixels_per_rank, ms_per_step):
    """Weak scaling: every rank renders its own frame; the job processes world x pixels per step."""
    return world * pixels_per_rank / (ms_per_step * 1e-3) / 1e6


# ---------------------------------------------------------------------------
# clocks during the timed region
# ---------------------------------------------------------------------------

class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index, interval_ms=25):
        self.gpu = gpu_index
        self.interval_ms = int(interval_ms)
        self.proc = None
        self.path = None

    def start(self):
        try:
            fd, self.path = tempfile.mkstemp(suffix=".csv")
            os.close(fd)
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", str(self.interval_ms)],
                                         stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except Exception as e:
            log("clock sampler unavailable:", e)
            self.proc = None

    def has_samples(self):
        try:
            return self.proc is not None and os.path.getsize(self.path) > 0
        except OSError:
            return False

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        rows = []
        for line in open(self.path):
            parts = [x.strip() for x in line.split(",")]
            if len(parts) >= 9:
                rows.append(parts)
        os.unlink(self.path)
        if not rows:
            return None
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4) if r[5 + i].lower() == "active"})
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(rows)}


# ---------------------------------------------------------------------------
# the workload
# ---------------------------------------------------------------------------

def workload(seed):
    import synth
    return synth.config2(seed)


def upstream(cam, seed, device):
    import torch
    g = torch.Generator(device="cpu").manual_seed(seed + 17)
    P = cam.W * cam.H
    return (torch.randn((P, 3), generator=g).to(device), (0.01 * torch.randn((P,), generator=g)).to(device),
            torch.randn((P,), generator=g).to(device))


def stage_models(stats, work, n_vox_total, n_pix, K, sh_bytes_per_vox, key_bits):
    """Algorithmic bytes (HBM stages) or FP32 ops (compositing) per launch of each stage."""
    V, nv, P, T = n_vox_total, stats["n_visible"], stats["n_pairs"], stats["n_tiles"]
    vb = max(1, math.ceil(key_bits / 8))       # radix passes of the depth-key sort
    tb = max(1, math.ceil(math.log2(max(T, 2)) / 8))
    tests, boxes, segs = work["tests"], work["box_tests"], work["segments"]
    return {
        "project": ("hbm", V * 8 + nv * 24),  # each voxel's 8-byte key; per visible voxel key, index, count, rectangle
        "records": ("hbm", nv * (4 + 8 + 4 + 8 + 32 + sh_bytes_per_vox + 64 + 8) + P * 8),
        "sort_vox": ("hbm", vb * nv * 24),
        "sort_pairs": ("hbm", tb * P * 16),
        "ranges": ("hbm", P * (4 + 4 + 8 + 1) + T * 12),
        "composite_fwd": ("alu", tests * F_TEST + boxes * F_BOX + segs * (K * F_SAMPLE + F_SEG)),
        "composite_bwd": ("alu", tests * F_TEST + boxes * F_BOX + segs * (K * F_SAMPLE_BWD + F_SEG_BWD)),
        # the same kernels' algorithmic DRAM bytes: per pair the voxel payload (densities 32, colour 12,
        # key 8) read once per tile, per pixel 20 B of images and 8 B of saved state; the backward also
        # reads the 20 B of upstream gradients per pixel and adds into 44 B of gradient per visible voxel
        "composite_fwd_bytes": ("hbm", P * 52 + n_pix * 28),
        "composite_bwd_bytes": ("hbm", P * 52 + n_pix * 48 + nv * 88),
        "sh_bwd": ("hbm", nv * (48 + 16 + sh_bytes_per_vox + 64 + 2 * sh_bytes_per_vox + 4)),
    }


# Stages (the library's profiler names) and the other rows, with the kernels that make them up and the
# sources that decide their DRAM traffic; a stage's traffic figure is kept only while those sources are
# unchanged.
STAGE_KERNELS = {
    "project": (("k_project",), ("dv_project.cu", "dv_internal.cuh")),
    "sort_vox": (("k_os_pass<unsigned long", "k_ol_count<unsigned long", "k_ol_scatter<unsigned long"),
                 ("dv_scan_sort.cu", "dv_internal.cuh")),
    "records": (("k_records_emit",), ("dv_project.cu", "dv_internal.cuh")),
    "sort_pairs": (("k_os_pass<unsigned int", "k_ol_count<unsigned int", "k_ol_scatter<unsigned int"),
                   ("dv_scan_sort.cu", "dv_internal.cuh")),
    "ranges": (("k_pair_mask", "k_tile_count", "k_tile_scatter"), ("dv_project.cu", "dv_internal.cuh")),
    "composite_fwd": (("k_composite<0", "k_composite_act<0"),
                      ("dv_composite.cu", "dv_composite_act.cu", "dv_composite.cuh", "dv_internal.cuh", "dv_project.cu")),
    "composite_bwd": (("k_composite<1", "k_composite_act<1"),
                      ("dv_composite.cu", "dv_composite_act.cu", "dv_composite.cuh", "dv_internal.cuh", "dv_project.cu")),
    "sh_bwd": (("k_sh_bwd",), ("dv_composite.cu", "dv_internal.cuh")),
}


def sources_hash(files):
    h = hashlib.sha256()
    for f in files:
        h.update(open(os.path.join(ROOT, "paper_2606_23031_gb300", "csrc", f), "rb").read())
    return h.hexdigest()[:16]


def load_traffic(stage):
    """DRAM bytes per launch of a stage from the committed ncu capture, or None once its sources changed."""
    try:
        t = json.load(open(TRAFFIC))
        e = t["stages"][stage]
    except Exception:
        return None
    if e.get("source_hash") != sources_hash(STAGE_KERNELS[stage][1]):
        return None
    return e.get("bytes_per_launch")


def peaks():
    try:
        m = json.load(open(MEASURED_PEAKS))
        return {"hbm_gbs": float(m["hbm_gbs"]), "src": "measured", "sm_max_mhz": float(m.get("sm_max_mhz", 2070.0))}
    except Exception:
        return {"hbm_gbs": 6800.0, "src": "fallback", "sm_max_mhz": 2070.0}


# ---------------------------------------------------------------------------
# CPU baseline / reference arm (the FP64 oracle on host cores)
# ---------------------------------------------------------------------------

def oracle_sample(sc, cam, n_px, seed):
    import numpy as np
    import oracle
    rng = np.random.default_rng(seed)
    pix = np.sort(rng.choice(cam.W * cam.H, size=n_px, replace=False))
    g = np.random.default_rng(seed + 1)
    g_rgb, g_d, g_a = g.normal(size=(n_px, 3)), 0.01 * g.normal(size=n_px), g.normal(size=n_px)
    t0 = time.perf_counter()
    oracle.render(sc.octrees, sc.poses, cam, oracle.Opts(1, 1e-4), pixels=pix)
    oracle.backward(sc.octrees, sc.poses, cam, g_rgb, g_d, g_a, oracle.Opts(1, 1e-4), pixels=pix)
    return time.perf_counter() - t0


def calibrate_oracle(sc, cam, seconds, seed):
    t = oracle_sample(sc, cam, 16, seed)
    per_px = t / 16
    n = int(min(max(seconds / max(per_px, 1e-6), 16), cam.W * cam.H, 8192))
    return n, per_px


def cpu_baseline(sc, cam, seconds, seed):
    n, _ = calibrate_oracle(sc, cam, seconds, seed)
    t = oracle_sample(sc, cam, n, seed + 5)
    return {"value": n / t / 1e6, "unit": "Mpix/s", "cores": os.cpu_count(), "kind": "oracle",
            "sample": f"{n} uniformly sampled pixels of the 1920x1080 frame, forward + backward, FP64 brute force "
                      f"over every voxel, {os.cpu_count()} threads ({t:.1f} s)"}


def run_reference(args):
    rank, world, _ = dist_env()
    if rank != 0:
        return 0
    sc, cams, _ = workload(args.seed)
    cam = cams[0]
    n, per_px = calibrate_oracle(sc, cam, max(1.0, min(args.cpu_seconds, 60.0 / max(args.steps + args.warmup, 1))),
                                 args.seed)
    for w in range(args.warmup):
        oracle_sample(sc, cam, max(8, n // 8), args.seed + 100 + w)
    times = [oracle_sample(sc, cam, n, args.seed + 200 + s) for s in range(args.steps)]
    tot = sum(times)
    value = n * args.steps / tot / 1e6
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": "Mpix/s", "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * tot / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": WORKLOAD, "sample_pixels_per_step": n},
            "cpu_baseline": {"value": value, "unit": "Mpix/s", "cores": os.cpu_count(), "kind": "oracle",
                             "sample": f"{n} sampled pixels per step, fwd+bwd, FP64 brute force"},
            "e2e": {"value": value, "unit": "Mpix/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0



# ---------------------------------------------------------------------------
# serving: continuous batching vs one request per launch (cfg 4 workload)
# ---------------------------------------------------------------------------

SERVE_WORKLOAD = ("config-2 background (500k leaves) + 20 actors x 20k leaves resident; Poisson requests, camera at "
                  "u ~ U(0,1) on a 100 m straight track, timestamp ~ U(0,10) s setting all 20 actor poses, "
                  "resolution uniform over {480x270, 960x540, 1920x1080}")


def serve_once(dv, ds, scene, reqs, mode, opts):
    import numpy as np
    import torch
    import synth
    if mode == "plain":
        cfg = dict(max_views=1, n_workers=1)
    else:
        cfg = dict(max_views=16, n_workers=2)
    srv = dv.Server(ds, max_batch_pixels=16 * 1920 * 1080, max_inflight_pixels=24 * 1920 * 1080, opts=opts, **cfg)
    pools = {}
    users = {}

    def out_for(cam, k):
        key = (cam.W, cam.H)
        pool = pools.setdefault(key, [])
        slot = k % 48
        while len(pool) <= slot:
            n = cam.W * cam.H
            pool.append((torch.empty((n, 3), device="cuda"), torch.empty((n,), device="cuda"),
                         torch.empty((n,), device="cuda")))
        prev = users.get((key, slot))
        if prev is not None:
            srv.wait(prev, 600000.0)          # the buffer's previous request must be done
        return pool[slot], (key, slot)

    # warm-up (contexts, pools, first launches)
    warm = [srv.submit(c.camera, synth.request_poses(scene, c.t), out_for(c.camera, i)[0])
            for i, c in enumerate(reqs[:8])]
    for t in warm:
        srv.wait(t, 600000.0)
        srv.release(t)
    users.clear()
    tickets, lags, pixels = [], [], 0
    t0 = time.perf_counter()
    for k, r in enumerate(reqs):
        now = time.perf_counter() - t0
        if r.arrival_s > now:
            time.sleep(r.arrival_s - now)
        buf, key = out_for(r.camera, k)
        lag = time.perf_counter() - t0 - r.arrival_s
        t = srv.submit(r.camera, synth.request_poses(scene, r.t), buf)
        users[key] = t
        tickets.append(t)
        lags.append(lag)
        pixels += r.camera.W * r.camera.H
    lat = []
    for t, lag in zip(tickets, lags):
        lat.append(srv.wait(t, 600000.0) + 1e3 * lag)
    t_end = time.perf_counter() - t0
    st = srv.stats()
    srv.close()
    lat = np.array(lat)
    return {"p50_ms": float(np.percentile(lat, 50)), "p99_ms": float(np.percentile(lat, 99)),
            "mean_ms": float(lat.mean()), "mpix_s": pixels / t_end / 1e6, "requests": len(reqs),
            "batches": st["batches"], "max_batch": st["max_batch"]}


def serving_bench(args, dv, opts):
    import synth
    scene = synth.config4(args.seed)
    ds = [dv.DeviceOctree.from_host(o) for o in scene.octrees]
    rows = []
    for rate in [float(x) for x in args.serve_rates.split(",") if x]:
        n = max(args.serve_min_requests, int(rate * args.serve_seconds))
        reqs = synth.request_stream(n, rate, args.seed + int(rate))
        row = {"rate_hz": rate}
        for mode in ("plain", "batched"):
            row[mode] = serve_once(dv, ds, scene, reqs, mode, opts)
        rows.append(row)
        log("serving", rate, row)
    return {"workload": SERVE_WORKLOAD, "plain": "max_views=1, 1 worker (one request per launch)",
            "batched": "max_views=16, 2 workers, continuous batching", "latency": "arrival -> outputs written",
            "rates": rows}

# ---------------------------------------------------------------------------
# the larger scenes: 8M-leaf background + 20 actors and 32M + 64 actors, six surround cameras in one call
# ---------------------------------------------------------------------------

LARGE = {
    "cfg3": ("full frame: LiDAR-shaped background 8M leaves (levels 6-14, 200 x 200 x 30 m) + 20 actors of 20k-60k "
             "leaves, 6 surround cameras 1920x1080 in one call, K=1, eps_stop=1e-4"),
    "cfg5": ("stress: LiDAR-shaped background 32M leaves (levels 6-16, 500 x 500 x 40 m) + 64 actors of 40k leaves, "
             "6 surround cameras 3840x2160 in one call, K=1, eps_stop=1e-4"),
}


def large_scene_bench(args, dv, dev, which, alu_peak, pk, flush):
    """Forward and forward+backward Mpix/s of one render call over all six cameras of a large scene, with
    the compositing kernels' roofline (CUDA events around each stage, separate runs)."""
    import torch
    import synth
    t0 = time.perf_counter()
    sc, cams = synth.config3(args.seed) if which == "cfg3" else synth.config5(args.seed)
    t_gen = time.perf_counter() - t0
    ds = [dv.DeviceOctree.from_host(o, dev) for o in sc.octrees]
    opts = dv.make_opts(1, 1e-4)
    ctx = dv.default_context(dev.index)
    stream = torch.cuda.current_stream()
    n_pix = sum(c.W * c.H for c in cams)
    g = torch.Generator(device=dev).manual_seed(args.seed + 23)
    g_rgb = torch.randn((n_pix, 3), generator=g, device=dev)
    g_d = 0.01 * torch.randn((n_pix,), generator=g, device=dev)
    g_a = torch.randn((n_pix,), generator=g, device=dev)
    d_dens = [torch.zeros_like(o.dens) for o in ds]
    d_sh = [torch.zeros_like(o.sh) for o in ds]

    def step(bwd):
        out = dv.dv_render(ds, sc.poses, cams, opts, ctx=ctx, save_state=bwd)
        if bwd:
            dv.dv_render_backward(out[-1], g_rgb, g_d, g_a, d_dens, d_sh)
            out[-1].free()

    step(True)
    torch.cuda.synchronize()
    _, _, _, st = dv.dv_render(ds, sc.poses, cams, opts, ctx=ctx, save_state=True)
    stats, work = st.stats(-1), st.work(-1)
    st.free()
    n = 3 if which == "cfg3" else 2
    res = {"workload": LARGE[which], "pixels_per_step": n_pix, "visible_voxels": stats["n_visible"],
           "pairs": stats["n_pairs"], "work": work, "generate_s": t_gen, "steps": n}
    for bwd, key in ((False, "fwd"), (True, "fwd_bwd")):
        ms = 0.0
        for _ in range(n):
            flush.zero_()
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(stream)
            step(bwd)
            b.record(stream)
            b.synchronize()
            ms += a.elapsed_time(b)
        res[key] = {"value": n_pix / (ms / n * 1e-3) / 1e6, "unit": "Mpix/s", "ms_per_step": ms / n}
    ctx.profile(True, stages=["composite_fwd", "composite_bwd"])
    ctx.profile_read()
    for _ in range(n):
        flush.zero_()
        step(True)
    torch.cuda.synchronize()
    pr = ctx.profile_read()
    ctx.profile(False)
    K = 1
    tests, boxes, segs = work["tests"], work["box_tests"], work["segments"]
    for kname, per_seg in (("composite_fwd", K * F_SAMPLE + F_SEG), ("composite_bwd", K * F_SAMPLE_BWD + F_SEG_BWD)):
        ms_k = pr[kname][0] / max(pr[kname][1], 1)
        flops = tests * F_TEST + boxes * F_BOX + segs * per_seg
        res[kname] = {"ms_per_run": ms_k, "algorithmic_flops": flops,
                      "achieved_tflops": flops / (ms_k * 1e-3) / 1e12,
                      "frac": flops / (ms_k * 1e-3) / 1e12 / alu_peak, "bound": "alu"}
    del ds, d_dens, d_sh
    torch.cuda.empty_cache()
    return res


# ---------------------------------------------------------------------------
# our arm
# ---------------------------------------------------------------------------

def run_ours(args):
    import numpy as np
    import torch
    import torch.distributed as dist

    import paper_2606_23031_gb300 as dv

    rank, world, local = dist_env()
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if world > 1:
        dist.init_process_group("nccl", device_id=dev)

    dv.load()
    sc, cams, _ = workload(args.seed + rank)
    cam = cams[0]
    ds = [dv.DeviceOctree.from_host(o, dev) for o in sc.octrees]
    opts = dv.make_opts(1, 1e-4)
    g_rgb, g_d, g_a = upstream(cam, args.seed, dev)
    d_dens = [torch.zeros_like(o.dens) for o in ds]
    d_sh = [torch.zeros_like(o.sh) for o in ds]
    flush = torch.empty(512 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
    ctx = dv.default_context(local)
    stream = torch.cuda.current_stream()
    n_pix = cam.W * cam.H

    def step():
        rgb, depth, alpha, st = dv.dv_render(ds, sc.poses, cams, opts, ctx=ctx, save_state=True)
        dv.dv_render_backward(st, g_rgb, g_d, g_a, d_dens, d_sh)
        return st

    def fwd_only():
        dv.dv_render(ds, sc.poses, cams, opts, ctx=ctx)

    def sync_all():
        torch.cuda.synchronize()
        if world > 1:
            dist.barrier()

    for _ in range(args.warmup):
        st = step()
        st.free()
    sync_all()
    # one extra (untimed) step for the work counters and sizes of this frame
    st = step()
    stats = st.stats(0)
    work = st.work(0)
    st.free()

    # ---- per-stage split, outside the timed region: every stage bracketed by events ----
    pk = peaks()
    # the FP32 FMA peak, measured here on this device (dv_measure_fp32_fma: dependent-FMA chains on every SM),
    # with the SM clock sampled while it runs
    n_sm = torch.cuda.get_device_properties(dev).multi_processor_count
    clk_p = ClockSampler(local)
    clk_p.start()
    time.sleep(0.3)
    f_peak, ms_peak = 0.0, 0.0
    for _ in range(3):
        f, m_ = dv.dv_measure_fp32_fma(local, 8192, 20)
        f_peak, ms_peak = f_peak + f, ms_peak + m_
    clk_peak = clk_p.stop()
    alu_peak = f_peak / (ms_peak * 1e-3) / 1e12   # TFLOP/s
    alu_peak_src = (f"measured: dv_measure_fp32_fma on {n_sm} SMs ({f_peak:.3g} FP32 ops in {ms_peak:.1f} ms, "
                    f"8 dependent-FMA chains per thread, full occupancy), SM clock median "
                    f"{(clk_peak or {}).get('sm_mhz')} MHz; nominal {n_sm} SMs x 128 lanes x 2 x "
                    f"{pk['sm_max_mhz']:.0f} MHz = {n_sm * 256 * pk['sm_max_mhz'] * 1e-6:.1f} TFLOP/s")
    sh_bytes = sum(o.n * (o.sh_degree + 1) ** 2 * 12 for o in sc.octrees) / max(sum(o.n for o in sc.octrees), 1)
    max_level = max(int((np.asarray(o.key, np.uint64) >> np.uint64(57)).max()) for o in sc.octrees if o.n)
    key_bits = 3 * max_level + max(1, math.ceil(math.log2(len(sc.octrees))))
    models = stage_models(stats, work, sum(o.n for o in sc.octrees), n_pix, 1, sh_bytes, key_bits)
    n_split = max(3, min(args.steps, 20))
    ctx.profile(True)
    ctx.profile_read()
    for _ in range(n_split):
        flush.zero_()
        step().free()
    sync_all()
    prof_split = ctx.profile_read()
    ctx.profile(False)
    dom = max((k for k in prof_split if k in models and prof_split[k][1]), key=lambda k: prof_split[k][0])

    # ---- timed fwd+bwd: events around the dominant stage only (its live duration for the roofline) ----
    clk = ClockSampler(local)
    clk.start()
    # untimed steps until nvidia-smi has taken its first sample, so that its samples cover the timed loops
    t_wait = time.perf_counter()
    while not clk.has_samples() and time.perf_counter() - t_wait < 3.0:
        step().free()
        torch.cuda.synchronize()
    launches0 = dv.dv_launch_count()
    ctx.profile(True, stages=[dom])
    ctx.profile_read()
    sync_all()
    wall0 = time.perf_counter()
    ms = 0.0
    for _ in range(args.steps):
        flush.zero_()
        a = torch.cuda.Event(enable_timing=True)
        b = torch.cuda.Event(enable_timing=True)
        a.record(stream)
        st = step()
        b.record(stream)
        b.synchronize()
        ms += a.elapsed_time(b)
        st.free()
    sync_all()
    wall = time.perf_counter() - wall0
    prof_timed = ctx.profile_read()
    ctx.profile(False)
    launches = dv.dv_launch_count() - launches0

    # ---- timed forward only ----
    for _ in range(2):
        fwd_only()
    sync_all()
    ms_f = 0.0
    for _ in range(args.steps):
        flush.zero_()
        a = torch.cuda.Event(enable_timing=True)
        b = torch.cuda.Event(enable_timing=True)
        a.record(stream)
        fwd_only()
        b.record(stream)
        b.synchronize()
        ms_f += a.elapsed_time(b)
    sync_all()
    clocks = clk.stop()  # sampled every 25 ms over both timed loops (fwd+bwd, then fwd)

    # ---- timed fwd+bwd with the normal state N (rendered and differentiated as well) ----
    g_n = None
    ms_n = 0.0
    if not args.core_only:
        g_n = torch.randn((n_pix, 3), generator=torch.Generator(dev).manual_seed(args.seed + 7), device=dev)

        def step_n():
            out = dv.dv_render(ds, sc.poses, cams, opts, ctx=ctx, save_state=True, normals=True)
            dv.dv_render_backward(out[-1], g_rgb, g_d, g_a, d_dens, d_sh, d_normal=g_n)
            return out[-1]

        for _ in range(3):
            step_n().free()
        sync_all()
        for _ in range(args.steps):
            flush.zero_()
            a = torch.cuda.Event(enable_timing=True)
            b = torch.cuda.Event(enable_timing=True)
            a.record(stream)
            st = step_n()
            b.record(stream)
            b.synchronize()
            ms_n += a.elapsed_time(b)
            st.free()
        sync_all()

    # ---- sky composite of Eq. 2 on the frame (1024 x 2048 equirectangular map): forward and backward ----
    ms_sky_f = ms_sky_b = 0.0
    if not args.core_only:
        env = torch.rand((1024, 2048, 3), generator=torch.Generator(dev).manual_seed(args.seed + 9), device=dev)
        rgb0, _, alpha0, _ = dv.dv_render(ds, sc.poses, cams, opts, ctx=ctx)
        sky_out = torch.empty_like(rgb0)
        d_env = torch.zeros_like(env)
        d_alpha = torch.zeros_like(alpha0)
        for _ in range(3):
            dv.dv_sky_composite(cams, env, rgb0, alpha0, ctx=ctx, out=sky_out)
            dv.dv_sky_backward(cams, env, alpha0, g_rgb, d_env, d_alpha, ctx=ctx)
        sync_all()
        for _ in range(args.steps):
            flush.zero_()
            a, b, c = (torch.cuda.Event(enable_timing=True) for _ in range(3))
            a.record(stream)
            dv.dv_sky_composite(cams, env, rgb0, alpha0, ctx=ctx, out=sky_out)
            b.record(stream)
            dv.dv_sky_backward(cams, env, alpha0, g_rgb, d_env, d_alpha, ctx=ctx)
            c.record(stream)
            c.synchronize()
            ms_sky_f += a.elapsed_time(b)
            ms_sky_b += b.elapsed_time(c)
        sync_all()

    # ---- feature fields: weights export of the frame, 64-channel feature render and fusion ----
    feats = None
    if not args.core_only:
        rgb0, _, alpha0, st0 = dv.dv_render(ds, sc.poses, cams, opts, ctx=ctx, save_state=True)
        nv = sum(o.n for o in sc.octrees)
        fe = torch.randn((nv, 64), generator=torch.Generator(dev).manual_seed(args.seed + 11), device=dev)
        f2 = torch.randn((n_pix, 64), generator=torch.Generator(dev).manual_seed(args.seed + 12), device=dev)
        acc = torch.zeros((nv, 64), device=dev)
        Wt = dv.dv_state_weights(st0)
        reps = max(3, args.steps // 10)
        t_ex = t_r = t_fu = 0.0
        for it in range(reps + 2):
            a, b, c, d_ = (torch.cuda.Event(enable_timing=True) for _ in range(4))
            flush.zero_()
            a.record(stream)
            dv.dv_state_weights(st0, out=Wt)
            b.record(stream)
            dv.dv_features_render(Wt, fe, ctx=ctx)
            c.record(stream)
            dv.dv_features_fuse(Wt, f2, acc, ctx=ctx)
            d_.record(stream)
            d_.synchronize()
            if it >= 2:
                t_ex += a.elapsed_time(b)
                t_r += b.elapsed_time(c)
                t_fu += c.elapsed_time(d_)
        st0.free()
        slots = int(Wt.voxel.numel())
        feats = {"what": "weights export of the frame, then a 64-channel feature render and 2-D feature fusion",
                 "slots": slots, "export_us": 1e3 * t_ex / reps, "render64_us": 1e3 * t_r / reps,
                 "fuse64_us": 1e3 * t_fu / reps,
                 # unique bytes: the slots once, one 64-float row per pixel once, and one 64-float row per
                 # visible voxel (read for the render; read and written by the fusion's additions)
                 "render64_gbs": (slots * 8 + n_pix * 64 * 4 + stats["n_visible"] * 64 * 4) / (t_r / reps * 1e-3) / 1e9,
                 "fuse64_gbs": (slots * 8 + n_pix * 64 * 4 + 2 * stats["n_visible"] * 64 * 4) / (t_fu / reps * 1e-3) / 1e9,
                 "bytes_model": ("unique bytes: per slot its (voxel, weight) once, one 64-float row per pixel "
                                 "(written by the render, read by the fusion) and one 64-float row per visible voxel "
                                 "(read by the render, read and written by the fusion)")}
        feats["render64_hbm_frac"] = feats["render64_gbs"] / pk["hbm_gbs"]
        feats["fuse64_hbm_frac"] = feats["fuse64_gbs"] / pk["hbm_gbs"]

    # ---- LiDAR-guided initialisation (Sec. 3.3) of the frame's background: shared corners, Eq. 1
    # prior from a 1.4M-point synthetic sweep, one proximity-subdivision round ----
    init = None
    if not args.core_only:
        import synth as _sy
        rng_i = np.random.default_rng(args.seed + 13)
        lay = _sy.city_layout(rng_i, 100.0, 30.0, 20)
        cloud = torch.as_tensor(np.float32(_sy.lidar_points(rng_i, lay, 1_000_000, 400_000)), device=dev)
        bg = sc.octrees[0]
        kt = torch.as_tensor(np.asarray(bg.key, np.uint64).view(np.int64), device=dev)
        L = int((np.asarray(bg.key, np.uint64) >> np.uint64(57)).max())
        s_min = float(bg.root_size) / 2 ** L
        dv.dv_shared_corners(kt, L, ctx=ctx)   # warm-up
        sync_all()
        t0 = time.perf_counter()
        grid_c, index_c = dv.dv_shared_corners(kt, L, ctx=ctx)
        t1 = time.perf_counter()
        dens_c = dv.dv_soft_prior(grid_c, bg.center, bg.root_size, L, cloud, s_min, ctx=ctx)
        torch.cuda.synchronize()
        t2 = time.perf_counter()
        new_keys = dv.dv_subdivide_round(kt, L, bg.center, bg.root_size, cloud, s_min, ctx=ctx)
        t3 = time.perf_counter()
        init = {"what": "background of the frame: shared corners, Eq. 1 prior from a 1.4M-point synthetic LiDAR "
                        "sweep, one subdivision round (threshold = finest voxel size); host wall time per call",
                "leaves": int(kt.numel()), "corners": int(grid_c.numel()), "points": int(cloud.shape[0]),
                "leaves_after_round": int(new_keys.numel()),
                "corners_ms": 1e3 * (t1 - t0), "prior_ms": 1e3 * (t2 - t1), "subdivide_ms": 1e3 * (t3 - t2)}
        del dens_c

    ms_step, ms_fwd, ms_nrm = max_over_ranks([ms / args.steps, ms_f / args.steps, ms_n / args.steps], world, dev)
    value = whole_job_mpix_s(world, n_pix, ms_step)
    value_fwd = whole_job_mpix_s(world, n_pix, ms_fwd)

    # ---- end to end through the public API with host buffers ----
    e2e = None
    if not args.no_e2e:
        h_g = [x.cpu().pin_memory() for x in (g_rgb, g_d, g_a)]
        d_g = [torch.empty_like(x) for x in (g_rgb, g_d, g_a)]
        h_out = [torch.empty((n_pix, 3), pin_memory=True), torch.empty((n_pix,), pin_memory=True),
                 torch.empty((n_pix,), pin_memory=True)]
        h_grad = [torch.empty(t.shape, pin_memory=True) for t in d_dens + d_sh]
        h2d = sum(x.numel() * 4 for x in h_g)
        d2h = sum(x.numel() * 4 for x in h_out) + sum(x.numel() * 4 for x in h_grad)

        # Frames are pipelined as a training or serving loop would run them: frame i's upstream
        # gradient is uploaded while frame i's forward runs (upload stream), its images go back
        # while its backward runs and its parameter gradients go back while frame i+1 computes
        # (download stream).  Device-side upstream and gradient buffers alternate between two sets,
        # each reused only after its previous copies have finished.
        up_stream, down_stream = torch.cuda.Stream(), torch.cuda.Stream()
        d_gs = [[torch.empty_like(x) for x in (g_rgb, g_d, g_a)] for _ in range(2)]
        grads = [[torch.zeros_like(t) for t in d_dens + d_sh] for _ in range(2)]
        ev_bwd = [torch.cuda.Event(), torch.cuda.Event()]
        ev_down = [torch.cuda.Event(), torch.cuda.Event()]
        for e in ev_bwd + ev_down:
            e.record(stream)
        n_oct = len(d_dens)

        def e2e_step(i):
            k = i % 2
            dg, gs = d_gs[k], grads[k]
            ev_in, ev_fwd = torch.cuda.Event(), torch.cuda.Event()
            with torch.cuda.stream(up_stream):
                up_stream.wait_event(ev_bwd[k])        # frame i-2's backward has read these buffers
                for hd, dd in zip(h_g, dg):
                    dd.copy_(hd, non_blocking=True)
                ev_in.record(up_stream)
            stream.wait_event(ev_down[k])              # frame i-2's gradients have left these buffers
            for t in gs:
                t.zero_()
            rgb, depth, alpha, st = dv.dv_render(ds, sc.poses, cams, opts, ctx=ctx, save_state=True)
            ev_fwd.record(stream)
            stream.wait_event(ev_in)
            dv.dv_render_backward(st, dg[0], dg[1], dg[2], gs[:n_oct], gs[n_oct:])
            ev_bwd[k].record(stream)
            with torch.cuda.stream(down_stream):
                down_stream.wait_event(ev_fwd)
                for ho, do in zip(h_out, (rgb, depth, alpha)):
                    do.record_stream(down_stream)
                    ho.copy_(do, non_blocking=True)
                down_stream.wait_event(ev_bwd[k])
                for hg, g_ in zip(h_grad, gs):
                    hg.copy_(g_, non_blocking=True)
                ev_down[k].record(down_stream)
            return st

        for i in range(4):
            e2e_step(i).free()
        sync_all()
        # the L2 flush between frames runs on the compute stream inside the pipeline; its own time,
        # measured alone, is taken out of the total
        fa, fb = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        fa.record(stream)
        for _ in range(args.steps):
            flush.zero_()
        fb.record(stream)
        fb.synchronize()
        ms_flush = fa.elapsed_time(fb)
        sync_all()
        a = torch.cuda.Event(enable_timing=True)
        b = torch.cuda.Event(enable_timing=True)
        a.record(stream)
        for i in range(args.steps):
            flush.zero_()
            e2e_step(i).free()   # stream-ordered: released once the frame's backward has run
        stream.wait_stream(down_stream)
        stream.wait_stream(up_stream)
        b.record(stream)
        b.synchronize()
        ms_e = a.elapsed_time(b) - ms_flush
        (ms_e2e,) = max_over_ranks([ms_e / args.steps], world, dev)
        e2e = {"value": whole_job_mpix_s(world, n_pix, ms_e2e), "unit": "Mpix/s",
               "ms_per_step": ms_e2e, "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h}

    # ---- per-stage figures (the split run) and the roofline of the dominant stage (the timed run) ----
    kernels = {}
    for name, (tot_ms, cnt) in prof_split.items():
        if name == dom:
            tot_ms, cnt = prof_timed[name]
        if cnt == 0:
            continue
        avg = tot_ms / cnt
        ent = {"ms_total": tot_ms, "runs": cnt, "ms_per_run": avg}
        if name in models:
            bound, amount = models[name]
            if bound == "hbm":
                ach = amount / (avg * 1e-3) / 1e9
                ent.update({"bound": "hbm", "algorithmic_bytes": amount, "achieved_gbs": ach,
                            "frac": ach / pk["hbm_gbs"]})
            else:
                ach = amount / (avg * 1e-3) / 1e12
                ent.update({"bound": "alu", "algorithmic_flops": amount, "achieved_tflops": ach,
                            "frac": ach / alu_peak})
                if name + "_bytes" in models:
                    # the compositing kernels also move DRAM bytes: their fraction of the copy bandwidth
                    b = models[name + "_bytes"][1]
                    ent.update({"algorithmic_bytes": b, "achieved_gbs": b / (avg * 1e-3) / 1e9,
                                "hbm_frac": b / (avg * 1e-3) / 1e9 / pk["hbm_gbs"]})
        tr = load_traffic(name)
        if tr is not None:
            ent["traffic"] = tr
        kernels[name] = ent
    d = kernels[dom]
    if d["bound"] == "hbm":
        roof = {"bound": "hbm", "achieved": d["achieved_gbs"], "peak": pk["hbm_gbs"], "unit": "GB/s",
                "frac": d["frac"], "traffic": load_traffic(dom), "kernel": dom,
                "peak_source": pk["src"] + " (MEASURED_PEAKS.json hbm_gbs)" if pk["src"] == "measured" else "fallback"}
    else:
        roof = {"bound": "alu", "achieved": d["achieved_tflops"], "peak": alu_peak, "unit": "TFLOP/s",
                "frac": d["frac"], "traffic": load_traffic(dom), "kernel": dom, "peak_source": alu_peak_src,
                "hbm_frac": d.get("hbm_frac"), "hbm_peak_gbs": pk["hbm_gbs"]}

    serving = None
    if rank == 0 and not args.no_serving:
        serving = serving_bench(args, dv, opts)

    large = {}
    if not args.core_only:
        for which in [x for x in args.large.split(",") if x]:
            large[which] = large_scene_bench(args, dv, dev, which, alu_peak, pk, flush)
            log(which, json.dumps(large[which]))

    cpu = None
    if rank == 0 and not args.no_cpu_baseline:
        cpu = cpu_baseline(sc, cam, args.cpu_seconds, args.seed)

    if rank == 0:
        line = {"metric": METRIC, "value": value, "unit": "Mpix/s", "n_gpus": world, "steps": args.steps,
                "warmup": args.warmup, "ms_per_step": ms_step, "higher_is_better": True, "scaling": "weak",
                "vs_baseline": None, "dtype": "f32", "data": "synthetic",
                "config": {"workload": WORKLOAD, "pixels_per_step": n_pix, "per_rank": "one frame per rank",
                           "l2": "flushed between timed steps (512 MB write outside the step events)",
                           "visible_voxels": stats["n_visible"], "pairs": stats["n_pairs"]},
                "fwd": {"value": value_fwd, "unit": "Mpix/s", "ms_per_step": ms_fwd},
                "features": feats,
                "init": init,
                "sky": None if args.core_only else {
                    "what": "sky composite of Eq. 2 on the frame, 1024x2048 equirectangular map",
                    "fwd_us": 1e3 * ms_sky_f / args.steps, "bwd_us": 1e3 * ms_sky_b / args.steps,
                    "fwd_gbs": 28.0 * n_pix / (ms_sky_f / args.steps * 1e-3) / 1e9,
                    "fwd_frac": 28.0 * n_pix / (ms_sky_f / args.steps * 1e-3) / 1e9 / pk["hbm_gbs"],
                    "bytes_per_pixel": {"fwd": 28, "bwd": 24}},
                "normals": None if args.core_only else {
                    "value": whole_job_mpix_s(world, n_pix, ms_nrm), "unit": "Mpix/s", "ms_per_step": ms_nrm,
                    "what": "fwd+bwd also rendering the normal state N and back-propagating a gradient on it"},
                "e2e": e2e, "roofline": roof, "cpu_baseline": cpu, "clocks": clocks, "gpu_launches": launches,
                "serving": serving, "large": large or None,
                "gpu_launches_per_step": launches / max(args.steps, 1), "wall_s_timed": wall,
                "work": work, "kernels": kernels,
                "kernels_source": (f"{dom}: CUDA events around it in every timed step; the other stages: "
                                   f"{n_split} steps outside the timed region with every stage bracketed by events")}
        print(json.dumps(line), flush=True)
    if world > 1:
        dist.barrier()
        dist.destroy_process_group()
    return 0


# ---------------------------------------------------------------------------
# counter capture: one profiled pass of every row, and the table built from it
# ---------------------------------------------------------------------------

def run_profile_pass(args):
    """No timing.  One warm-up pass and one profiled pass over every row on the 1080p frame (fwd+bwd,
    fwd+bwd with normals, the sky composite and its backward, the weights export with a 64-channel feature
    render and fusion, the initialisation calls, an asset grid), so that a counter capture of the library's
    kernels can skip the first pass by count.  Prints the library's launches of each pass."""
    import numpy as np
    import torch
    import paper_2606_23031_gb300 as dv
    import synth
    torch.cuda.set_device(0)
    dev = torch.device("cuda", 0)
    dv.load()
    sc, cams, _ = workload(args.seed)
    cam = cams[0]
    ds = [dv.DeviceOctree.from_host(o, dev) for o in sc.octrees]
    opts = dv.make_opts(1, 1e-4)
    ctx = dv.default_context(0)
    g_rgb, g_d, g_a = upstream(cam, args.seed, dev)
    n_pix = cam.W * cam.H
    g_n = torch.randn((n_pix, 3), generator=torch.Generator(dev).manual_seed(args.seed + 7), device=dev)
    d_dens = [torch.zeros_like(o.dens) for o in ds]
    d_sh = [torch.zeros_like(o.sh) for o in ds]
    env = torch.rand((1024, 2048, 3), generator=torch.Generator(dev).manual_seed(args.seed + 9), device=dev)
    nv = sum(o.n for o in sc.octrees)
    fe = torch.randn((nv, 64), generator=torch.Generator(dev).manual_seed(args.seed + 11), device=dev)
    f2 = torch.randn((n_pix, 64), generator=torch.Generator(dev).manual_seed(args.seed + 12), device=dev)
    acc = torch.zeros((nv, 64), device=dev)
    rng_i = np.random.default_rng(args.seed + 13)
    lay = synth.city_layout(rng_i, 100.0, 30.0, 20)
    cloud = torch.as_tensor(np.float32(synth.lidar_points(rng_i, lay, 1_000_000, 400_000)), device=dev)
    bg = sc.octrees[0]
    kt = torch.as_tensor(np.asarray(bg.key, np.uint64).view(np.int64), device=dev)
    L = int((np.asarray(bg.key, np.uint64) >> np.uint64(57)).max())
    s_min = float(bg.root_size) / 2 ** L
    sky_out = torch.empty((n_pix, 3), device=dev)
    d_env = torch.zeros_like(env)
    d_alpha = torch.zeros((n_pix,), device=dev)

    def one_pass():
        rgb, depth, alpha, st = dv.dv_render(ds, sc.poses, cams, opts, ctx=ctx, save_state=True)
        dv.dv_render_backward(st, g_rgb, g_d, g_a, d_dens, d_sh)
        out = dv.dv_render(ds, sc.poses, cams, opts, ctx=ctx, save_state=True, normals=True)
        dv.dv_render_backward(out[-1], g_rgb, g_d, g_a, d_dens, d_sh, d_normal=g_n)
        dv.dv_sky_composite(cams, env, rgb, alpha, ctx=ctx, out=sky_out)
        dv.dv_sky_backward(cams, env, alpha, g_rgb, d_env, d_alpha, ctx=ctx)
        w = dv.dv_state_weights(st)
        dv.dv_features_render(w, fe, ctx=ctx)
        dv.dv_features_fuse(w, f2, acc, ctx=ctx)
        grid_c, index_c = dv.dv_shared_corners(kt, L, ctx=ctx)
        dv.dv_soft_prior(grid_c, bg.center, bg.root_size, L, cloud, s_min, ctx=ctx)
        dv.dv_subdivide_round(kt, L, bg.center, bg.root_size, cloud, s_min, ctx=ctx)
        dv.dv_visibility_prune(kt, L, bg.center, bg.root_size, cams, 0.0, ctx=ctx)
        dv.dv_asset_init((4.5, 1.9, 1.6), 6, ctx=ctx)
        torch.cuda.synchronize()
        st.free()
        out[-1].free()

    dv.dv_launch_count(True)
    one_pass()
    warm = dv.dv_launch_count(True)
    one_pass()
    prof = dv.dv_launch_count(True)
    print(f"LAUNCHES {warm} {prof}", flush=True)
    return 0


def build_traffic(csv_path, out_path=TRAFFIC):
    """profiles/traffic.json and a markdown table (stdout) from an ncu --csv capture of one profiled pass
    (metrics dram__bytes_read.sum, dram__bytes_write.sum, gpu__time_duration.sum)."""
    import csv
    rows = {}
    with open(csv_path) as f:
        lines = [ln for ln in f if ln.startswith('"')]
    for r in csv.DictReader(lines):
        k = r["ID"]
        e = rows.setdefault(k, {"id": int(k), "name": r["Kernel Name"], "m": {}})
        v = r["Metric Value"].replace(",", "")
        unit = r.get("Metric Unit", "")
        scale = {"byte": 1, "Kbyte": 1e3, "Mbyte": 1e6, "Gbyte": 1e9, "ns": 1e-3, "nsecond": 1e-3, "us": 1.0,
                 "usecond": 1.0, "ms": 1e3, "msecond": 1e3}.get(unit, 1.0)
        try:
            e["m"][r["Metric Name"]] = float(v) * scale
        except ValueError:
            pass
    launches = sorted(rows.values(), key=lambda e: e["id"])
    # stage of every launch
    stage_of = []
    for e in launches:
        st = None
        for sname, (kernels, _) in STAGE_KERNELS.items():
            if any(kn in e["name"] for kn in kernels):
                st = sname
        # a large sort scans its digit counts between counting and scattering
        if "k_scan_" in e["name"] and stage_of and stage_of[-1] in ("sort_vox", "sort_pairs"):
            st = stage_of[-1]
        stage_of.append(st)
    # the profiled pass renders the frame twice (plain, then with normals): the stages of the plain
    # frame are its first occurrence of each stage until the first composite_bwd and sh_bwd
    stages = {}
    seen_sh = False
    for e, st in zip(launches, stage_of):
        if st is None or seen_sh:
            continue
        rec = stages.setdefault(st, {"bytes": 0.0, "us": 0.0, "kernels": []})
        rec["bytes"] += e["m"].get("dram__bytes_read.sum", 0.0) + e["m"].get("dram__bytes_write.sum", 0.0)
        rec["us"] += e["m"].get("gpu__time_duration.sum", 0.0)
        rec["kernels"].append(e["name"].split("(")[0])
        if st == "sh_bwd":
            seen_sh = True
    per_kernel = {}
    for e in launches:
        nm = e["name"].split("(")[0]
        d = per_kernel.setdefault(nm, {"launches": 0, "bytes": 0.0, "us": 0.0})
        d["launches"] += 1
        d["bytes"] += e["m"].get("dram__bytes_read.sum", 0.0) + e["m"].get("dram__bytes_write.sum", 0.0)
        d["us"] += e["m"].get("gpu__time_duration.sum", 0.0)
    out = {"source": "ncu --metrics dram__bytes_read.sum,dram__bytes_write.sum,gpu__time_duration.sum "
                     "--clock-control none -k regex:k_ -s <warm-up launches> -c <pass launches> --csv "
                     "python bench.py --profile-pass (one pass of every row on the 1920x1080 frame)",
           "stages": {st: {"bytes_per_launch": int(r["bytes"]), "us_ncu": r["us"],
                           "source_hash": sources_hash(STAGE_KERNELS[st][1]), "kernels": r["kernels"]}
                      for st, r in stages.items()},
           "kernels": per_kernel}
    with open(out_path, "w") as f:
        json.dump(out, f, indent=1)
    print("| kernel | launches | DRAM bytes (read + write) | ncu time (us, serialised) |")
    print("|---|---|---|---|")
    for nm, d in sorted(per_kernel.items(), key=lambda kv: -kv[1]["us"]):
        print(f"| `{nm}` | {d['launches']} | {d['bytes'] / 1e6:.2f} MB | {d['us']:.1f} |")
    return 0


def main():
    args = parse()
    if args.traffic_from:
        return build_traffic(args.traffic_from)
    if args.profile_pass:
        return run_profile_pass(args)
    if args.impl == "reference":
        return run_reference(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
