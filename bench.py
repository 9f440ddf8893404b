"""Benchmark: keyframe densification at 1920x960 with 6 source views.

One step = one keyframe through the whole hot path: random initialisation,
8 red-black iterations of propagation + refinement (11x11 window sampled at
stride 2, bilateral weights, best-3 of 6 views), then the geometric
consistency filter of that keyframe against 4 neighbouring depth maps.
Inputs are seeded synthetic panoramas (scenes/) already resident in HBM;
the L2 is flushed between timed steps and each step is timed with CUDA
events on the launching stream.

At N = 1 the line also carries the batched form (32 keyframes of mixed sizes in
one batch, fp16 images, against the plain per-keyframe path with fp32 images),
the served form (300 Poisson requests over a 64-frame fp16 ring against a FIFO
of the plain fp32 path) and the precision forms (one 3840x1920 keyframe with 8
sources stored as fp32, fp16 and uint8), each with its own config (--no-extras
skips them).

--impl reference times the CPU oracle on the same workload (bounded sample
per step: random initialisation plus one half-sweep of the 1920x960 frame,
scaled to a keyframe, plus the consistency filter).
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import tempfile
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

W, H, N_SRC, ITERS = 1920, 960, 6, 8
N_NEIGHBOURS = 4
METRIC = "keyframes/s (1920x960, 6 views, 11x11/2 window, 8 iterations, best-3, + consistency filter)"
WORKLOAD = "equirect PatchMatch densify 1920x960 u8, 6 sources, 11x11 stride 2, 8 iters, best-3, filter vs 4 maps"
# FP32-pipe instructions of one view-sample by the algorithm's own count:
# transform 9, two four-quadrant arctangents 2 x 12, hypot 3, scale to pixel
# coordinates 2, bilinear (floor, fraction, footprint, 3 lerps) 12, centred
# moments 5  ->  55.
OPS_PER_VIEW_SAMPLE = 55
FP32_LANES_PER_SM = 128
# DRAM bytes of one 6-view half-sweep launch at 1920x960 (dram__bytes_read.sum +
# dram__bytes_write.sum from one ncu capture of the current kernel build:
# 49,884,160 read + 848,640 written). Set to None whenever the kernel changes
# until it is captured again.
SWEEP_DRAM_BYTES = 49_884_160 + 848_640


def _dist():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled during the timed region."""

    def __init__(self, index):
        self.index = str(index)
        self.proc = None
        self.path = None

    def __enter__(self):
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={q}", "--format=csv,noheader,nounits",
                                          "-i", self.index, "-lms", "200"],
                                         stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
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

    def summary(self):
        if not self.path or not os.path.exists(self.path):
            return None
        rows = []
        for line in open(self.path):
            f = [x.strip() for x in line.split(",")]
            if len(f) < 9:
                continue
            try:
                rows.append((float(f[1]), float(f[2]), f[5], f[6], f[7], f[8]))
            except ValueError:
                continue
        os.unlink(self.path)
        if not rows:
            return None
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4) if r[2 + i].lower() == "active"})
        return {"sm_mhz": statistics.median(r[0] for r in rows), "sm_max_mhz": max(r[1] for r in rows),
                "samples": len(rows), "reasons": reasons}


def max_over_ranks(x: float) -> float:
    """Largest value of x over the ranks of the (gloo) process group; every rank
    gets it. Replicas run independent keyframes, so this timing reduction is the
    only exchange between them."""
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(x)], dtype=torch.float64)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    dist.barrier()
    return float(t.item())


def replica_throughput(world_size: int, steps: int, max_total_ms: float) -> float:
    """Whole-job keyframes/s of N replicas: every rank densifies `steps` keyframes,
    the job takes as long as the slowest rank."""
    return world_size * steps / (max_total_ms / 1e3)


def make_workload(seed_scene=1001):
    """Trajectory of 7 + 4 frames: keyframe = frame 5, sources = frames 2..4, 6..8,
    filter neighbours = keyframes 3, 4, 6, 7 (their maps are densified in warm-up)."""
    import scenes
    traj = scenes.trajectory(11, seed=2000)
    scene = scenes.Scene(seed=seed_scene)
    scene.objects = scenes.place_objects(seed_scene + 77, [c for _, _, c in traj], n=20)
    frames = []
    for (R, t, C) in traj:
        img, rg = scene.render(R, t, W, H, with_range=True)
        frames.append(scenes.Frame(R, t, C, scenes.quantise_u8(img), rg))
    params = dict(d_min=0.3, d_max=10.0, patch_w=11, patch_stride=2, iterations=ITERS, best_k=3,
                  sigma_color=0.2, sigma_space=3.0, n_refine=6, neighbor_table=0, seed=42, keyframe_id=5)
    return frames, params


def problem_of(frames, k):
    srcs = [frames[j] for j in (k - 3, k - 2, k - 1, k + 1, k + 2, k + 3)]
    return frames[k], srcs


def keyframe_config(world_size: int) -> dict:
    """The keyframe workload's description, the same for both arms."""
    return dict(workload=WORKLOAD, image_storage="u8", width=W, height=H, sources=N_SRC, iterations=ITERS,
                window="11x11/2", best_k=3, filter_neighbours=N_NEIGHBOURS,
                l2="flushed (256 MiB write) between steps",
                parallelism="replicas" if world_size > 1 else "single")


def algorithmic_counts():
    evals = W * H * (1 + ITERS * (8 + 6))
    view_samples = evals * N_SRC * 36
    return evals, view_samples


def run_gpu(args):
    import torch
    import paper_2211_16266_gb300 as pm

    ws, rank, local = _dist()
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if ws > 1:
        import torch.distributed as dist
        dist.init_process_group("gloo")
    frames, params = make_workload()
    stream = torch.cuda.Stream(device=dev)
    ctx = pm.Context(local, stream=stream)
    to_dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)
    dimg = {k: to_dev(frames[k].image) for k in range(len(frames))}
    poses = {k: (frames[k].R, frames[k].t) for k in range(len(frames))}

    def args_for(k):
        _, srcs = problem_of(frames, k)
        idx = (k - 3, k - 2, k - 1, k + 1, k + 2, k + 3)
        return dimg[k], poses[k], [dimg[j] for j in idx], [poses[j] for j in idx]

    KF, NB = 5, (3, 4, 6, 7)
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        nb_maps = {k: pm.pmsp_densify(ctx, *args_for(k), dict(params, keyframe_id=k)) for k in NB}
        out = pm.Maps.empty(W, H, device=dev)
        filt = torch.empty((H, W), dtype=torch.float32, device=dev)
        agree = torch.empty((H, W), dtype=torch.int32, device=dev)
        flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)
    kf_args = args_for(KF)

    def step():
        pm.pmsp_densify(ctx, *kf_args, params, out=out)
        pm.pmsp_consistency_filter(ctx, out.depth, poses[KF], [nb_maps[k].depth for k in NB],
                                   [poses[k] for k in NB], 1.0, 2, out=filt, agree=agree)

    with torch.cuda.stream(stream):
        for _ in range(args.warmup):
            step()
    stream.synchronize()

    # per-kernel timing of one half-sweep launch set (the dominant kernel)
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    times = []
    if ws > 1:
        import torch.distributed as dist
        dist.barrier()
    torch.cuda.synchronize()
    uuid = getattr(torch.cuda.get_device_properties(dev), "uuid", None)
    smi_id = f"GPU-{uuid}" if uuid is not None and not str(uuid).startswith("GPU-") else (str(uuid) if uuid else local)
    with ClockSampler(smi_id) as clk:
        with torch.cuda.stream(stream):
            for i in range(args.steps):
                flush.zero_()
                ev[i][0].record(stream)
                step()
                ev[i][1].record(stream)
        stream.synchronize()
    times = [a.elapsed_time(b) for a, b in ev]
    total_ms = sum(times)
    if ws > 1:
        total_ms = max_over_ranks(total_ms)

    # dominant kernel: time the 16 half-sweeps of one keyframe alone (same stream)
    sweep_ms = time_sweeps(pm, ctx, stream, kf_args, params, out, flush)

    # end to end through the C ABI with host buffers (pinned), copies inside the timed region
    e2e = None if args.no_e2e else run_e2e(pm, ctx, stream, frames, KF, NB, nb_maps, params, args)

    evals, vs = algorithmic_counts()
    clocks = clk.summary() or {}
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    res = dict(
        metric=METRIC, value=replica_throughput(ws, args.steps, total_ms), unit="keyframes/s", n_gpus=ws,
        steps=args.steps, warmup=args.warmup, ms_per_step=total_ms / args.steps, higher_is_better=True,
        scaling="weak", vs_baseline=None, dtype="f32", data="synthetic",
        config=keyframe_config(ws),
        latency_ms=dict(p50=float(np.percentile(times, 50)), p99=float(np.percentile(times, 99))),
        hypothesis_evals_per_s=ws * evals * args.steps / (total_ms / 1e3),
        # initialisation, every half-sweep's pooled kernel, the bounded one beside all but the first, the filter
        gpu_launches=args.steps * (1 + 2 * ITERS + (2 * ITERS - 1) + 1),
        clocks=clocks,
    )
    if rank == 0:
        peak_mhz = clocks.get("sm_max_mhz") or 2070.0
        nominal = sms * FP32_LANES_PER_SM * peak_mhz * 1e6 / OPS_PER_VIEW_SAMPLE
        with torch.cuda.stream(stream):
            peaks = pm.pmsp_measure_peaks(ctx)
        fma_rate = max(peaks["fp32_fma_per_s"], peaks["fp32x2_fma_per_s"])
        peak = fma_rate / OPS_PER_VIEW_SAMPLE
        vs_per_sweep = W * H / 2 * 14 * N_SRC * 36
        achieved = vs_per_sweep / (sweep_ms / 1e3)
        res["roofline"] = dict(bound="alu", achieved=achieved, peak=peak, unit="view-samples/s",
                               frac=achieved / peak, traffic=SWEEP_DRAM_BYTES, traffic_unit="bytes per launch",
                               kernel="pixel_kernel<6, SWEEP, 11x11/2 window> (one half-sweep)",
                               ms_per_launch=sweep_ms,
                               peak_basis=f"measured FP32 FMA rate {fma_rate:.4g}/s (pmsp_measure_peaks: "
                                          f"max of scalar and packed f32x2 FMA chains over all SMs) / "
                                          f"{OPS_PER_VIEW_SAMPLE} FP32 operations per view-sample",
                               peak_nominal=nominal,
                               units_basis="the method's 8 neighbour + 6 refinement candidates per pixel, 6 views, "
                                           "36 samples; the kernel skips neighbour candidates bit-identical to the "
                                           "incumbent or an earlier one (about 4.4 % of the evaluation rounds on "
                                           "this workload), whose cost is known; timed as half-sweeps called on their own, "
                                           "while those of a run also leave out neighbours they know and refinement "
                                           "tests that cannot win",
                               units=dict(
                                   # one gather and four special-function results per view-sample
                                   gather_frac_of_l1_peak=achieved / peaks["gather_l1_per_s"],
                                   sfu_frac=4 * achieved / peaks["sfu_per_s"],
                                   hbm=hbm_fraction(SWEEP_DRAM_BYTES, sweep_ms)),
                               measured_peaks=peaks)
        res["e2e"] = e2e
        gt = frames[KF].range
        dk = out.depth.cpu().numpy()
        res["ground_truth"] = dict(within_5pct=float(np.mean(np.abs(dk - gt) < 0.05 * gt)),
                                   within_1pct=float(np.mean(np.abs(dk - gt) < 0.01 * gt)),
                                   of="the keyframe's range map before the filter, against the rendered range")
        if not args.no_cpu_baseline and ws == 1:
            nb_np = [nb_maps[k].depth.cpu().numpy() for k in NB]
            res["cpu_baseline"] = cpu_baseline(frames, KF, params, out.depth.cpu().numpy(), nb_np, NB)
        if ws == 1 and not args.no_extras:
            res.update(extra_forms(args))
        print(json.dumps(res))
    ctx.close()
    if ws > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


def precision_forms(reps=3, n_sample=300):
    """The 3840x1920 precision workload (8 sources, 8-bit texture + N(0, 2 DN) noise,
    11x11/2, 8 iterations, best-3) rendered once and stored as fp32 (render / 255), fp16
    (the same minus 0.5, centred) and uint8 (the render quantised): per form the
    keyframe time (median of `reps`, CUDA events), the share of pixels within 5 % and 1 %
    of the rendered range, and the share of `n_sample` seeded pixels whose stored cost is
    within 1e-4 of the FP64 oracle's cost of the stored plane."""
    import torch
    import oracle
    import scenes
    import paper_2211_16266_gb300 as pm
    base = scenes.config2(fmt="f32")
    params = base.params
    dev = torch.device("cuda", 0)
    stream = torch.cuda.Stream(device=dev)
    ctx = pm.Context(0, stream=stream)
    conv = {"f32": lambda im: im,
            "f16": lambda im: (im - 0.5).astype(np.float16),
            "u8": lambda im: np.clip(np.rint(im * 255.0), 0, 255).astype(np.uint8)}
    gt = base.ref.range
    H, W = gt.shape
    rng = np.random.default_rng(6)
    us, vs = rng.integers(0, W, n_sample), rng.integers(0, H, n_sample)
    out = {}
    for fmt, f in conv.items():
        ref, srcs = f(base.ref.image), [f(fr.image) for fr in base.srcs]
        d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)
        args = (d(ref), (base.ref.R, base.ref.t), [d(x) for x in srcs], [(fr.R, fr.t) for fr in base.srcs])
        with torch.cuda.stream(stream):
            maps = pm.Maps.empty(W, H, device=dev)
            pm.pmsp_densify(ctx, *args, params, out=maps)
            ts = []
            for _ in range(reps):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record(stream)
                pm.pmsp_densify(ctx, *args, params, out=maps)
                b.record(stream)
                ts.append((a, b))
        stream.synchronize()
        ms = float(np.median([a.elapsed_time(b) for a, b in ts]))
        dep, nrm, cst = (x.astype(np.float64) for x in maps.numpy())
        pb = oracle.Problem(ref, (base.ref.R, base.ref.t), srcs, [(fr.R, fr.t) for fr in base.srcs], **params)
        errs = np.array([abs(pb.cost(u, v, dep[v, u], nrm[:, v, u]) - cst[v, u]) for u, v in zip(us, vs)])
        out[fmt] = dict(ms=ms, keyframes_per_s=1e3 / ms,
                        within_5pct_of_gt=float(np.mean(np.abs(dep - gt) < 0.05 * gt)),
                        within_1pct_of_gt=float(np.mean(np.abs(dep - gt) < 0.01 * gt)),
                        stored_cost_within_1e4_of_fp64_oracle=float(np.mean(errs <= 1e-4)))
    ctx.close()
    return out


# The autotuner's pick on the 32-keyframe fp16 batch (bench.py --workload batched):
# pmsp_tuning(blocks_per_sm, order, patch_stride, strategy, tile, tpp, lanes).
BATCH_TUNING = (0, 0, 0, 1, 0, 1)


def extra_forms(args):
    """The batched, served and precision forms beside the keyframe line (N = 1 only): the
    32-keyframe batch in fp16 against the plain per-keyframe path with fp32 images, the
    served fp16 ring (lanes) against the plain fp32 FIFO on the Poisson trace, and one
    3840x1920 keyframe stored three ways, with ground-truth accuracy and latency. A form
    that fails reports its error in its own key; the keyframe line is printed either way."""
    import traceback
    import paper_2211_16266_gb300 as pm

    def guarded(fn):
        try:
            return fn()
        except Exception as e:  # keep the headline line: report the failure in the extra's key
            traceback.print_exc(file=sys.stderr)
            return dict(error=f"{type(e).__name__}: {e}")

    def batched():
        forms, used = batched_forms(formats=("f16", "f32"), reps=3, tuning=BATCH_TUNING)
        return dict(metric=BATCHED_METRIC, unit="keyframes/s", value=forms["batched_f16"]["keyframes_per_s"],
                    config=dict(workload="32 mixed keyframes in one batch, CUDA graph, fp16 images", tuning=used),
                    forms=forms)

    def serving():
        runs = serving_runs(args.requests, [("served", "f16", pm.PMSP_SCHED_LANES), ("plain", "f32", None)])
        return dict(metric=SERVING_METRIC, unit="keyframes/s", value=runs["served_f16_lanes"]["keyframes_per_s"],
                    latency_ms=dict(p50=runs["served_f16_lanes"]["p50_ms"], p99=runs["served_f16_lanes"]["p99_ms"]),
                    config=dict(workload=f"{args.requests} Poisson requests over a 64-frame fp16 ring, lanes "
                                         "scheduler, 40 GB admission cap"),
                    runs=runs)

    def precision():
        prec = precision_forms()
        return dict(metric="keyframes/s, 3840x1920, 8 views, 11x11/2, 8 iterations, best-3", unit="keyframes/s",
                    value=prec["f16"]["keyframes_per_s"],
                    config=dict(workload="one 3840x1920 keyframe, 8-bit texture + 2 DN noise, stored as fp32, "
                                         "fp16 (centred) and uint8; FP32 arithmetic, FP64 poses"),
                    forms=prec)

    return dict(batched=guarded(batched), serving=guarded(serving), precision=guarded(precision))


def hbm_fraction(bytes_per_launch, ms_per_launch):
    """DRAM bytes of one half-sweep launch (ncu) over its duration, against the measured
    copy bandwidth in MEASURED_PEAKS.json when it is there, else the 6.8 TB/s fallback."""
    peak, basis = 6800.0, "fallback 6.8 TB/s"
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            peak, basis = float(json.load(f)["hbm_gbs"]), "measured copy bandwidth"
    except (OSError, KeyError, ValueError):
        pass
    if bytes_per_launch is None:
        return None
    gbs = bytes_per_launch / (ms_per_launch / 1e3) / 1e9
    return dict(achieved_gbs=gbs, peak_gbs=peak, frac=gbs / peak, peak_basis=basis)


def time_sweeps(pm, ctx, stream, kf_args, params, out, flush):
    """Mean duration of one half-sweep launch (dominant kernel), CUDA events on its stream."""
    import torch
    state = pm.Maps(out.depth.clone(), out.normal.clone(), out.cost.clone())
    reps = 6
    durs = []
    with torch.cuda.stream(stream):
        for r in range(reps):
            flush.zero_()
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(stream)
            pm.pmsp_halfsweep(ctx, *kf_args, params, r & 1, 9 + r // 2, state)
            b.record(stream)
            durs.append((a, b))
    stream.synchronize()
    # the half-sweep call also uploads 6 textures (device copies); subtract nothing: they are ~10 us
    return float(np.mean([a.elapsed_time(b) for a, b in durs]))


def run_e2e(pm, ctx, stream, frames, KF, NB, nb_maps, params, args):
    import torch
    pin = lambda a: torch.from_numpy(np.ascontiguousarray(a)).pin_memory().numpy()
    idx = (KF - 3, KF - 2, KF - 1, KF + 1, KF + 2, KF + 3)
    ref = pin(frames[KF].image)
    srcs = [pin(frames[j].image) for j in idx]
    nbd = [pin(nb_maps[k].depth.cpu().numpy()) for k in NB]
    out = pm.Maps(pin(np.zeros((H, W), np.float32)), pin(np.zeros((3, H, W), np.float32)),
                  pin(np.zeros((H, W), np.float32)))
    filt = pin(np.zeros((H, W), np.float32))
    agree = pin(np.zeros((H, W), np.int32))
    poses = lambda ks: [(frames[k].R, frames[k].t) for k in ks]

    def step():
        pm.pmsp_densify(ctx, ref, (frames[KF].R, frames[KF].t), srcs, poses(idx), params, out=out)
        pm.pmsp_consistency_filter(ctx, out.depth, (frames[KF].R, frames[KF].t), nbd, poses(NB), 1.0, 2,
                                   out=filt, agree=agree)

    for _ in range(args.warmup):
        step()
    n = args.steps
    t0 = time.perf_counter()
    for _ in range(n):
        step()
    dt = (time.perf_counter() - t0) / n
    h2d = ref.nbytes + sum(s.nbytes for s in srcs) + out.depth.nbytes + sum(d.nbytes for d in nbd)
    d2h = out.depth.nbytes + out.normal.nbytes + out.cost.nbytes + filt.nbytes + agree.nbytes
    return dict(value=1.0 / dt, unit="keyframes/s", h2d_bytes_per_step=int(h2d), d2h_bytes_per_step=int(d2h),
                steps=n, timer="host wall clock around the C-ABI calls")


def cpu_baseline(frames, KF, params, depth=None, nb_depths=None, NB=()):
    """The oracle as it stands on the host cores, on a bounded sample of the keyframe:
    random initialisation, one red half-sweep (scaled to the 2 x iterations half-sweeps)
    and, when the keyframe's and its neighbours' depth maps are given, the consistency
    filter against them. Beside it, one core: 400 sampled pixel initialisations and
    updates (orc_random_plane + orc_cost, orc_update_pixel, serial code), scaled to the
    keyframe's pixels."""
    import oracle
    ref, srcs = problem_of(frames, KF)
    pb = oracle.Problem(ref.image, (ref.R, ref.t), [f.image for f in srcs], [(f.R, f.t) for f in srcs], **params)
    t0 = time.perf_counter()
    d, n, c = pb.init()
    t1 = time.perf_counter()
    pb.halfsweep(d, n, c, 0, 0)
    t2 = time.perf_counter()
    t_filter = 0.0
    if depth is not None and nb_depths:
        oracle.consistency_filter(depth, (ref.R, ref.t), nb_depths, [(frames[k].R, frames[k].t) for k in NB], 1.0, 2)
        t_filter = time.perf_counter() - t2
    t_kf = (t1 - t0) + 2 * ITERS * (t2 - t1) + t_filter
    cores = len(os.sched_getaffinity(0)) if hasattr(os, "sched_getaffinity") else os.cpu_count()
    cores = int(os.environ.get("OMP_NUM_THREADS", cores))
    # one core: serial per-pixel calls on a seeded sample of pixels
    Hk, Wk = ref.image.shape
    rng = np.random.default_rng(11)
    us, vs = rng.integers(0, Wk, 400), rng.integers(0, Hk, 400)
    t3 = time.perf_counter()
    for u, v in zip(us, vs):
        dd, nn = pb.random_plane(u, v)
        pb.cost(u, v, dd, nn)
    t4 = time.perf_counter()
    for u, v in zip(us, vs):
        pb.update_pixel(d, n, c, u, v, 1)
    t5 = time.perf_counter()
    t_kf1 = Wk * Hk * (t4 - t3) / len(us) + 2 * ITERS * (Wk * Hk / 2) * (t5 - t4) / len(us)
    return dict(value=1.0 / t_kf, unit="keyframes/s", cores=cores, kind="oracle",
                sample=f"FP64 oracle on {cores} cores: random init ({t1 - t0:.1f} s) + one red half-sweep "
                       f"({t2 - t1:.1f} s) of the 1920x960 keyframe, scaled to init + {2 * ITERS} half-sweeps, "
                       f"+ consistency filter vs {len(NB)} maps ({t_filter:.2f} s)",
                single_core=dict(value=1.0 / t_kf1, unit="keyframes/s", cores=1,
                                 sample=f"400 seeded pixels: random plane + cost, then one pixel update, "
                                        f"serial, scaled to {Wk}x{Hk} init + {2 * ITERS} half-sweeps "
                                        f"(filter not included)"))


def run_reference(args):
    ws, rank, _ = _dist()
    if rank != 0:
        return
    frames, params = make_workload()
    KF, NB = 5, (3, 4, 6, 7)
    per, wall = [], []
    for _ in range(args.steps):
        t0 = time.perf_counter()
        # the filter's inputs: rendered ranges stand in for the neighbours' maps (same work)
        cb = cpu_baseline(frames, KF, params, frames[KF].range, [frames[k].range for k in NB], NB)
        wall.append(time.perf_counter() - t0)
        per.append(1.0 / cb["value"])
    val = args.steps / sum(per)
    cb["value"] = val
    # each step times a bounded sample and scales it to a keyframe: ms_per_step is the
    # wall time a sampled step took (the timed region is steps x that), and the value
    # in keyframes/s comes from the scaled keyframe time, reported beside it
    cb["sample_s_per_step"] = float(np.mean(wall))
    cb["keyframe_s_scaled"] = float(sum(per) / args.steps)
    print(json.dumps(dict(impl="reference", metric=METRIC, value=val, unit="keyframes/s", n_gpus=ws,
                          steps=args.steps, warmup=args.warmup, ms_per_step=1e3 * float(np.mean(wall)),
                          higher_is_better=True, scaling="weak", vs_baseline=None, dtype="f64",
                          data="synthetic", config=keyframe_config(ws), cpu_baseline=cb,
                          e2e=dict(value=val, unit="keyframes/s", h2d_bytes_per_step=0, d2h_bytes_per_step=0))))


BATCH_CLASSES = ((960, 480, 12), (1920, 960, 14), (3840, 1920, 6))


class ClassFrames:
    """Frames of one resolution class rendered along one trajectory (ss=1). uint8 images are
    quantised DN; fp32 images hold the unquantised render / 255, fp16 images the same
    minus 0.5."""

    def __init__(self, W, H, n, seed, fmt, with_range=False):
        import scenes
        self.W, self.H = W, H
        traj = scenes.trajectory(n, seed=seed)
        scene = scenes.Scene(seed=1003)
        scene.objects = scenes.place_objects(1080, [c for _, _, c in traj], n=20)
        self.frames, self.ranges = [], []
        for (R, t, C) in traj:
            img, rg = scene.render(R, t, W, H, ss=1, with_range=with_range)
            if fmt == "u8":
                im = scenes.quantise_u8(img)
            elif fmt == "f16":
                # centred on 0: fp16 rounding is finer near 0, and the cost depends on
                # intensity differences and correlations only
                im = (img / 255.0 - 0.5).astype(np.float16)
            else:
                im = (img / 255.0).astype(np.float32)
            self.frames.append((im, (R, t)))
            self.ranges.append(rg)


def batched_problems(fmt, seed=3000, with_range=False):
    """32 keyframes: 12 at 960x480, 14 at 1920x960, 6 at 3840x1920, 4-10 sources each.
    Items are (reference, sources, params, ground-truth range or None)."""
    rng = np.random.default_rng(seed)
    out = []
    for ci, (W, H, count) in enumerate(BATCH_CLASSES):
        cf = ClassFrames(W, H, 2 * count + 11, 2000 + ci, fmt, with_range)
        for k in range(count):
            centre = 5 + 2 * k
            S = int(rng.integers(4, 11))
            offs = [o for o in (-1, 1, -2, 2, -3, 3, -4, 4, -5, 5)][:S]
            params = dict(d_min=0.3, d_max=10.0, patch_w=11, patch_stride=2, iterations=ITERS, best_k=3,
                          sigma_color=0.2, sigma_space=3.0, n_refine=6, neighbor_table=0, seed=42,
                          keyframe_id=1000 * ci + k)
            out.append((cf.frames[centre], [cf.frames[centre + o] for o in offs], params, cf.ranges[centre]))
    return out


def batched_forms(formats=("f16", "u8", "f32"), reps=3, tuning=None):
    """The 32-keyframe mix in one batch (CUDA graph; autotuned when `tuning` is None),
    fp16 storage, and the plain per-keyframe path on the same keyframes with each image
    format in `formats`; per form its median time, keyframes/s and share of pixels within
    1 % of the rendered range. Returns (forms, tuning used)."""
    import torch
    import paper_2211_16266_gb300 as pm
    dev = torch.device("cuda", 0)
    stream = torch.cuda.Stream(device=dev)
    ctx = pm.Context(0, stream=stream)
    res, acc = {}, {}
    used = None

    def accuracy(outs, gts):
        good = total = 0
        for o, gt in zip(outs, gts):
            d = o.depth.cpu().numpy()
            good += int(np.sum(np.abs(d - gt) < 0.01 * gt))
            total += gt.size
        return good / total

    for fmt in formats:
        probs = batched_problems(fmt, with_range=True)
        gts = [p[3] for p in probs]
        to_dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)
        cache = {}

        def d(im):
            key = id(im)
            if key not in cache:
                cache[key] = to_dev(im)
            return cache[key]
        items = [(d(ref[0]), ref[1], [d(s[0]) for s in srcs], [s[1] for s in srcs], p) for ref, srcs, p, _ in probs]
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            outs = [pm.Maps.empty(it[0].shape[1], it[0].shape[0], device=dev) for it in items]

            def timed(fn, n):
                fn()
                stream.synchronize()
                ts = []
                for _ in range(n):
                    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                    a.record(stream)
                    fn()
                    b.record(stream)
                    stream.synchronize()
                    ts.append(a.elapsed_time(b))
                return float(np.median(ts))

            def plain():
                for it, o in zip(items, outs):
                    pm.pmsp_densify(ctx, *it, out=o)
            if fmt == "f16":
                batch = pm.Batch([(*it, o) for it, o in zip(items, outs)])
                t = pm.pmsp_autotune(ctx, batch, 0.0) if tuning is None else pm.pmsp_tuning(*tuning)
                res["batched_f16"] = timed(lambda: pm.pmsp_densify_batch(ctx, batch, pm.PMSP_BATCH_GRAPH, t), reps)
                stream.synchronize()
                acc["batched_f16"] = accuracy(outs, gts)
                used = dict(blocks_per_sm=t.blocks_per_sm, order=t.order, patch_stride=t.patch_stride,
                            strategy=t.strategy, tile=t.tile, tpp=t.tpp, lanes=t.lanes)
            res[f"plain_{fmt}"] = timed(plain, reps)
            stream.synchronize()
            acc[f"plain_{fmt}"] = accuracy(outs, gts)
    ctx.close()
    n = sum(c for _, _, c in BATCH_CLASSES)
    forms = {k: dict(ms=res[k], keyframes_per_s=n / (res[k] / 1e3), within_1pct_of_gt=acc[k]) for k in res}
    return forms, used


BATCHED_METRIC = "keyframes/s, 32 mixed keyframes (12x960x480, 14x1920x960, 6x3840x1920), 4-10 views"


def run_batched(args):
    """Config: 32 mixed keyframes in one batch (persistent/concurrent launches, CUDA graph,
    autotuned), FP16 storage, against the plain per-keyframe path on the same keyframes with
    uint8, fp16 and fp32 images; ground-truth accuracy of each (share of pixels within 1 %)."""
    forms, used = batched_forms(reps=max(2, args.steps))
    print(json.dumps(dict(
        metric=BATCHED_METRIC, value=forms["batched_f16"]["keyframes_per_s"], unit="keyframes/s", n_gpus=1,
        steps=args.steps, warmup=1, ms_per_step=forms["batched_f16"]["ms"], higher_is_better=True, scaling="weak",
        vs_baseline=None, dtype="f32", data="synthetic",
        config=dict(workload="batched form: one batch of 32 keyframes, CUDA graph, autotuned", image_storage="f16",
                    tuning=used, forms=forms))))


def run_batched_uniform(args):
    """Config: 4 keyframes at 960x480 with 6 sources each (921,600 pixels, as many as one
    1920x960 keyframe), 11x11/2, best-3, 2 iterations, uint8: the persistent strategy (one
    launch per phase over every keyframe's tiles) against per-keyframe chains, best of 5."""
    import torch
    import scenes
    import paper_2211_16266_gb300 as pm
    dev = torch.device("cuda", 0)
    stream = torch.cuda.Stream(device=dev)
    ctx = pm.Context(0, stream=stream)
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)
    items = []
    for k in range(4):
        p = scenes.trajectory_problem(960, 480, 6, offset=k, with_range=False)
        prm = dict(d_min=0.3, d_max=10.0, patch_w=11, patch_stride=2, iterations=2, best_k=3, sigma_color=0.2,
                   sigma_space=3.0, n_refine=6, neighbor_table=0, seed=42, keyframe_id=k)
        with torch.cuda.stream(stream):
            out = pm.Maps.empty(960, 480, device=dev)
        items.append((d(p.ref.image), (p.ref.R, p.ref.t), [d(f.image) for f in p.srcs],
                      [(f.R, f.t) for f in p.srcs], prm, out))
    batch = pm.Batch(items)
    res = {}
    for name, t in [("persistent", pm.pmsp_tuning(0, 0, 0, 0, 0, 1)), ("chains", pm.pmsp_tuning(0, 0, 0, 1, 0, 1))]:
        with torch.cuda.stream(stream):
            pm.pmsp_densify_batch(ctx, batch, 0, t)
            stream.synchronize()
            ts = []
            for _ in range(5):
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record(stream)
                pm.pmsp_densify_batch(ctx, batch, 0, t)
                e1.record(stream)
                stream.synchronize()
                ts.append(e0.elapsed_time(e1))
        res[name] = min(ts)
    ctx.close()
    print(json.dumps(dict(metric="ms per batch, 4 keyframes 960x480, 6 views, 2 iterations", unit="ms",
                          higher_is_better=False, value=res["persistent"], data="synthetic",
                          config=dict(workload="uniform batch: persistent strategy vs per-keyframe chains",
                                      image_storage="u8"),
                          ms=res)))


def serving_runs(n_req, runs):
    """Poisson requests (4/s, 1-s bursts at 12/s every 20 s, seed 3000) of the batched mix's
    sizes and 4-10 views; each run is ("served", format, scheduler) over a 64-frame ring or
    ("plain", format, None), a FIFO of the plain per-keyframe path on the same arrivals.
    Returns p50/p99 latency (arrival to maps on the host) and keyframes/s per run."""
    import threading
    import torch
    import paper_2211_16266_gb300 as pm
    rng = np.random.default_rng(3000)
    t, arrivals = 0.0, []
    while len(arrivals) < n_req:
        rate = 12.0 if (t % 20.0) < 1.0 else 4.0
        t += rng.exponential(1.0 / rate)
        arrivals.append(t)
    weights = np.array([c for _, _, c in BATCH_CLASSES], float)
    classes = rng.choice(3, size=n_req, p=weights / weights.sum())
    views = rng.integers(4, 11, size=n_req)
    out = {}
    frames_of = {}
    for mode, fmt, sched in runs:
        if fmt not in frames_of:
            frames_of[fmt] = [ClassFrames(W, H, 24, 2000 + ci, fmt) for ci, (W, H, _) in enumerate(BATCH_CLASSES)]
        cfs = frames_of[fmt]
        lat = []
        if mode == "served":
            ctx = pm.Context(0, stream=None, ring_capacity=64, scheduler=sched)
            counters = [0, 0, 0]
            ids = [[], [], []]
            next_id = [0]
            maps = {ci: pm.Maps.empty(W, H) for ci, (W, H, _) in enumerate(BATCH_CLASSES)}
            tickets = []
            lock = threading.Lock()
            stop = threading.Event()

            def retriever():
                # results are read back as they finish (polled every 0.5 ms), so a
                # latency ends when the maps are on the host, as in the plain path
                while not stop.is_set() or tickets:
                    with lock:
                        pending = list(tickets)
                    for entry in pending:
                        if pm.pmsp_poll(ctx, entry[0], maps[entry[1]]) is not None:
                            lat.append(time.perf_counter() - entry[2])
                            with lock:
                                tickets.remove(entry)
                    time.sleep(0.0005)

            def push(ci):
                cf = cfs[ci]
                im, pose = cf.frames[counters[ci] % len(cf.frames)]
                counters[ci] += 1
                fid = next_id[0]
                next_id[0] += 1
                while True:
                    try:
                        pm.pmsp_ring_push(ctx, fid, im, pose)
                        break
                    except pm.PmspError as e:
                        # back-pressure: every ring frame is held by queued or running
                        # requests; wait for results to release some
                        if e.code != pm.PMSP_EBUSY:
                            raise
                        time.sleep(0.001)
                ids[ci].append(fid)
                return fid
            for ci in range(3):           # warm the ring: 10 frames per class
                for _ in range(10):
                    push(ci)
            th = threading.Thread(target=retriever, daemon=True)
            t0 = time.perf_counter()
            th.start()
            for k in range(n_req):
                now = time.perf_counter() - t0
                if arrivals[k] > now:
                    time.sleep(arrivals[k] - now)
                ci = int(classes[k])
                ref = push(ci)
                S = int(views[k])
                srcs = ids[ci][-(S + 1):-1]
                p = dict(d_min=0.3, d_max=10.0, patch_w=11, patch_stride=2, iterations=ITERS, best_k=3,
                         sigma_color=0.2, sigma_space=3.0, n_refine=6, neighbor_table=0, seed=42, keyframe_id=k)
                tk = pm.pmsp_submit(ctx, ref, srcs, p)
                with lock:
                    tickets.append((tk, ci, t0 + arrivals[k]))  # latency counts from the arrival
            stop.set()
            th.join()
            wall = time.perf_counter() - t0
            ctx.close()
        else:
            # the plain path has no ring: every request uploads its reference and sources
            # from the host and reads its maps back, like the served requests
            ctx = pm.Context(0)
            dframes = [[im for im, _ in cf.frames] for cf in cfs]
            outs = {ci: pm.Maps.empty(W, H) for ci, (W, H, _) in enumerate(BATCH_CLASSES)}
            counters = [10, 10, 10]
            t0 = time.perf_counter()
            busy_until = 0.0
            for k in range(n_req):
                now = time.perf_counter() - t0
                if arrivals[k] > now:
                    time.sleep(arrivals[k] - now)
                ci = int(classes[k])
                n_f = len(cfs[ci].frames)
                r = counters[ci]
                counters[ci] += 1
                S = int(views[k])
                ref_i = r % n_f
                src_i = [(r - j) % n_f for j in range(1, S + 1)]
                p = dict(d_min=0.3, d_max=10.0, patch_w=11, patch_stride=2, iterations=ITERS, best_k=3,
                         sigma_color=0.2, sigma_space=3.0, n_refine=6, neighbor_table=0, seed=42, keyframe_id=k)
                # FIFO: the request waits for the previous ones (single worker), then runs alone
                pm.pmsp_densify(ctx, dframes[ci][ref_i], cfs[ci].frames[ref_i][1], [dframes[ci][j] for j in src_i],
                                [cfs[ci].frames[j][1] for j in src_i], p, out=outs[ci])
                lat.append(time.perf_counter() - t0 - arrivals[k])  # host maps: the call returned with them
            wall = time.perf_counter() - t0
            ctx.close()
        lat = np.array(lat) * 1e3
        name = f"{mode}_{fmt}" + ("" if sched is None else ("_lanes" if sched == pm.PMSP_SCHED_LANES else "_steps"))
        out[name] = dict(p50_ms=float(np.percentile(lat, 50)), p99_ms=float(np.percentile(lat, 99)),
                         keyframes_per_s=n_req / wall, wall_s=wall)
        print(name, out[name], file=sys.stderr, flush=True)
    return out


SERVING_METRIC = "p50/p99 latency and keyframes/s, Poisson 4/s + 12/s bursts, mixed sizes"


def run_serving(args):
    """Config: Poisson requests (4/s, 1-s bursts at 12/s every 20 s) of mixed sizes served by
    continuous batching over a 64-frame ring (FP16), with either scheduler, against a FIFO
    of the plain per-keyframe path (fp32, and with --serving-all uint8, images) on the same
    arrival trace."""
    import paper_2211_16266_gb300 as pm
    n_req = args.requests
    runs = [("served", "f16", pm.PMSP_SCHED_LANES), ("served", "f16", pm.PMSP_SCHED_STEPS), ("plain", "f32", None)]
    if args.serving_all:
        runs.append(("plain", "u8", None))
    out = serving_runs(n_req, runs)
    best = min(("served_f16_lanes", "served_f16_steps"), key=lambda k: out[k]["p99_ms"])
    print(json.dumps(dict(
        metric=SERVING_METRIC,
        value=out[best]["keyframes_per_s"], unit="keyframes/s", n_gpus=1, steps=n_req, warmup=0,
        ms_per_step=1e3 * out[best]["wall_s"] / n_req, higher_is_better=True, scaling="weak",
        vs_baseline=None, dtype="f32", data="synthetic",
        latency_ms=dict(p50=out[best]["p50_ms"], p99=out[best]["p99_ms"]),
        config=dict(workload=f"serving form: {n_req} requests over a 64-frame ring, continuous batching",
                    image_storage="f16", scheduler=best.rsplit("_", 1)[1], runs=out))))


def run_pipeline(args):
    """Online-mode pipeline on a 16-frame synthetic walk at 1920x960 (uint8): for each of
    10 keyframes, densify against 6 neighbouring frames (with plane-map warping from the
    previous keyframe, or from random planes), then the consistency filter against up
    to 4 neighbouring keyframes' maps, the median post-filter, fusion of all filtered
    keyframes into one voxel-deduplicated cloud and the completeness at every keyframe
    position at 720x360 (the paper's measure). Reports keyframes/s of the whole chain,
    per-stage device times, completeness, cloud size and accuracy against ground truth."""
    import torch
    import scenes
    import paper_2211_16266_gb300 as pm
    n_frames, first, last = 16, 3, 13
    traj = scenes.trajectory(n_frames, seed=2000)
    scene = scenes.Scene(seed=1001)
    scene.objects = scenes.place_objects(1078, [c for _, _, c in traj], n=20)
    frames = []
    for (R, t, C) in traj:
        img, rg = scene.render(R, t, W, H, with_range=True)
        frames.append(scenes.Frame(R, t, C, scenes.quantise_u8(img), rg))
    dev = torch.device("cuda", 0)
    dimg = [torch.from_numpy(np.ascontiguousarray(f.image)).to(dev) for f in frames]
    pose = [(f.R, f.t) for f in frames]
    keys = list(range(first, last))
    stream = torch.cuda.Stream(device=dev)
    ctx = pm.Context(0, stream=stream)
    out = {}
    for iters in (8, 3):
        for mode in ("warped", "random"):
            params = dict(d_min=0.3, d_max=10.0, patch_w=11, patch_stride=2, iterations=iters, best_k=3,
                          sigma_color=0.2, sigma_space=3.0, n_refine=6, neighbor_table=0, seed=42)
            ev = {s: [] for s in ("densify", "filter", "median", "fuse", "completeness")}

            def timed(stage, fn):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record(stream)
                r = fn()
                b.record(stream)
                ev[stage].append((a, b))
                return r

            maps = {}
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            with torch.cuda.stream(stream):
                for k in keys:
                    idx = (k - 3, k - 2, k - 1, k + 1, k + 2, k + 3)
                    a = (dimg[k], pose[k], [dimg[j] for j in idx], [pose[j] for j in idx], dict(params, keyframe_id=k))
                    if mode == "warped" and k - 1 in maps:
                        maps[k] = timed("densify", lambda: pm.pmsp_densify_warped(ctx, *a, maps[k - 1], pose[k - 1]))
                    else:
                        maps[k] = timed("densify", lambda: pm.pmsp_densify(ctx, *a))
                filt = {}
                for k in keys:
                    nb = [j for j in (k - 2, k - 1, k + 1, k + 2) if j in maps]
                    f, _ = timed("filter", lambda: pm.pmsp_consistency_filter(
                        ctx, maps[k].depth, pose[k], [maps[j].depth for j in nb], [pose[j] for j in nb], 1.0, 2))
                    filt[k] = timed("median", lambda: pm.pmsp_median_filter(ctx, f, 2, 0.05))
                pts, _, n_pts = timed("fuse", lambda: pm.pmsp_fuse(ctx, [filt[k] for k in keys], [pose[k] for k in keys],
                                                                   0.01, cap=len(keys) * W * H))
                comp = [timed("completeness", lambda: pm.pmsp_completeness(ctx, pts, pose[k], 720, 360)[0])
                        for k in keys]
            stream.synchronize()
            wall = time.perf_counter() - t0
            ms = {s: float(sum(a.elapsed_time(b) for a, b in v)) for s, v in ev.items()}
            valid, good = 0.0, 0.0
            for k in keys:
                d = filt[k].cpu().numpy()
                gt = frames[k].range
                valid += np.mean(d > 0)
                good += np.mean((d > 0) & (np.abs(d - gt) < 0.01 * gt))
            out[f"{mode}_{iters}it"] = dict(
                keyframes_per_s=len(keys) / (sum(ms.values()) / 1e3), wall_s=wall, stage_ms=ms,
                completeness_720x360=float(np.mean(comp)), points=int(n_pts),
                valid_share=valid / len(keys), within_1pct_of_gt=good / len(keys))
    ctx.close()
    main_r = out["warped_8it"]
    print(json.dumps(dict(
        metric="keyframes/s of the online pipeline (densify + consistency + median + fusion + completeness)",
        value=main_r["keyframes_per_s"], unit="keyframes/s", n_gpus=1, steps=len(keys), warmup=0,
        ms_per_step=1e3 / main_r["keyframes_per_s"], higher_is_better=True, scaling="weak", vs_baseline=None,
        dtype="f32", data="synthetic",
        config=dict(image_storage="u8", workload="online pipeline: 10 keyframes 1920x960 along a 16-frame walk, 6 views, 11x11/2, "
                             "best-3, filter vs 4 keyframes, median 5x5/5 %, 1 cm voxels, 720x360 completeness"),
        runs=out)))


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--workload", default="keyframe",
                    choices=["keyframe", "batched", "batched-uniform", "serving", "pipeline"])
    ap.add_argument("--requests", type=int, default=300)
    ap.add_argument("--serving-all", action="store_true", help="serving workload: also the uint8 FIFO")
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="gb300", choices=["gb300", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-e2e", action="store_true", help="skip the host-buffer end-to-end leg")
    ap.add_argument("--no-extras", action="store_true",
                    help="keyframe workload: skip the batched and served forms run after it at N = 1")
    args = ap.parse_args()
    if args.impl == "reference":
        run_reference(args)
        return
    import __graft_entry__
    __graft_entry__.build()
    if args.workload == "batched":
        run_batched(args)
    elif args.workload == "batched-uniform":
        run_batched_uniform(args)
    elif args.workload == "serving":
        run_serving(args)
    elif args.workload == "pipeline":
        run_pipeline(args)
    else:
        run_gpu(args)


if __name__ == "__main__":
    main()
