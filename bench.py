#!/usr/bin/env python3
"""Benchmark: whitened injections per second of the on-the-fly simulation path.

One step is one batch of the method's per-batch pass (Sec. 3.2) on the long-window
three-detector workload (H1+L1+V1, 2048 Hz, 8 s windows, N = 16384, 8192 draws per
step): prior draws and the FP64 per-draw set-up (prepared one batch ahead on a side
stream), and ``simulate_prepared`` (TaylorF2 waveforms, projection, crops, injection,
whitening) for B draws, through the libgwx C ABI.  The background (a fresh
coloured-noise stretch and its Welch PSD) is regenerated inside the timed loop every
``--background-every`` steps (default 16; the paper keeps one background chunk for
many batches); the line also reports the rate with a fresh background every step.
Further legs: end to end through pinned host memory, the same step on the 4 s
geometry (``hl3``), the log-likelihood with importance weights on ragged events, the
learned part, and the FFT kernels against cuFFT.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl gwx|reference]

Timing: W untimed steps, then K steps, each bracketed by CUDA events on the
launching stream, with a 256 MiB buffer written between steps (outside the events;
the 1.6 GB output of a step exceeds L2 anyway); barrier + synchronize before and
after; max over ranks.  Under torchrun each rank is an independent replica on its
own GPU with its own step counters (weak scaling, no data-path collective).  Rank 0
prints one JSON line: the headline with its configuration and bounds, and the main figure of
every further leg; ``--record PATH`` writes all of the legs' figures to a file.
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

import workloads  # noqa: E402

WORKLOAD = "sweep"
STEP_STRIDE = 1 << 20            # per-rank offset of the step counters
FP32_LANES_PER_SM = 128          # FP32 FMA lanes per Blackwell SM
SM_MAX_MHZ_FALLBACK = 2070.0
# ncu DRAM traffic (read + write bytes) per k_simulate launch, in steady state (the
# launch after another, caches not flushed, so the write-back of the previous launch's
# dirty lines is counted and this launch's own L2-resident tail is not), keyed by
# workload, with the hash of the kernel sources it was measured on.  A workload whose
# capture does not match the current sources reports null.
TRAFFIC = {"sweep": {"bytes_per_launch": 8 * 199703808, "B": 8192, "sources_sha1": "673a2fe948b01e62dd6b1520886d0f38acf32f76",
                    "note": "ncu DRAM read + write of the second of two back-to-back 1024-draw launches of the same "
                            "geometry (caches not flushed: it pays the first launch's write-back, 199.70 MB), scaled "
                            "by the draws per launch"}}


def _measured_peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as fh:
            return json.load(fh)
    except (OSError, ValueError):
        return {}


MEASURED_PEAKS = _measured_peaks()


def describe(wl):
    return ("%s: TaylorF2 3.5PN (IMRPhenomD tables unavailable), %s, fs=%d Hz, %g s windows (N=%d), "
            "B=%d draws/step, %g s background (L=%d), Welch %g s Hann segments 50%% overlap, f_lo=%g Hz"
            % (wl["name"], "+".join(wl["dets"]), wl["fs"], wl["T"], wl["N"], wl["B"], wl["L"] / wl["fs"], wl["L"],
               wl["seg_len"] / wl["fs"], wl["f_lo"]))


def flops_per_injection(wl):
    """Algorithmic FP32 flops of one whitened injection in the fused kernel:
    per detector a forward and an inverse real FFT of N points (2.5 N log2 N each)
    and ~20 flops per bin of frequency-domain work, plus ~150 flops per bin for the
    waveform shared by the detectors."""
    N, D = wl["N"], len(wl["dets"])
    F = N // 2 + 1
    return D * (2 * 2.5 * N * math.log2(N) + 20 * F) + 150 * F


def kernel_sources_sha1():
    h = hashlib.sha1()
    for f in ("k_fused.cu", "fft16.cuh", "fft16r.cuh", "common.cuh", "waveform.cuh", "tc05.cuh"):
        with open(os.path.join(ROOT, "paper_2407_19048_gb300", "csrc", f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()


def fp32_peak(torch, sm_mhz):
    """FP32 peak of this GPU in TFLOP/s at the given SM clock: the SM count reported by
    the device (cudaGetDeviceProperties) x 128 FMA lanes per SM x 2 flops."""
    props = torch.cuda.get_device_properties(torch.cuda.current_device())
    n_sm = int(props.multi_processor_count)
    return n_sm, n_sm * FP32_LANES_PER_SM * 2 * float(sm_mhz) * 1e6 / 1e12


def sm_max_mhz(clk):
    """Maximum SM clock: nvidia-smi's clocks.max.sm sampled during the run, else the
    measured figure, else the part's nominal maximum."""
    if clk and clk.get("sm_max_mhz"):
        return float(clk["sm_max_mhz"]), "nvidia-smi clocks.max.sm"
    if MEASURED_PEAKS.get("sm_max_mhz"):
        return float(MEASURED_PEAKS["sm_max_mhz"]), "MEASURED_PEAKS.json sm_max_mhz"
    return SM_MAX_MHZ_FALLBACK, "nominal maximum"


def traffic_per_launch(wl):
    t = TRAFFIC.get(wl["name"])
    if t and t["sources_sha1"] == kernel_sources_sha1() and t["B"] == wl["B"]:
        return t["bytes_per_launch"]
    return None


def bench_config(wl, args, world):
    """The `config` object of the JSON line; both arms print the same one."""
    return {"workload": describe(wl), "global_batch": wl["B"] * world, "seq_len": wl["N"],
            "parallelism": "replicas: one per GPU with disjoint Philox counters, no data-path collective",
            "l2": "outputs (%.2f GB per step) exceed L2; a 256 MiB buffer is also written between timed steps, "
                  "outside the events" % (wl["B"] * len(wl["dets"]) * wl["N"] * 4 / 1e9),
            "step": "prior draws + FP64 per-draw set-up of the next batch, and the fused pass (waveforms, "
                    "projection, crops, injection, whitening) of this batch; background (coloured noise + Welch "
                    "PSD) regenerated every %d steps" % args.background_every,
            "background_every": args.background_every}


def step_counter(rank, i):
    """Counter of step i on a rank: ranks draw disjoint Philox streams."""
    return (rank * STEP_STRIDE + i) & 0xFFFFFFFF


def max_over_ranks(value, dist=None):
    if dist is None or not dist.is_initialized() or dist.get_world_size() == 1:
        return value
    import torch
    t = torch.tensor([float(value)], dtype=torch.float64,
                     device="cuda" if dist.get_backend() == "nccl" else "cpu")
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


# ----------------------------------------------------------------- clocks
class ClockSampler:
    QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.gpu = gpu_index
        self.proc = None
        self.path = None

    def start(self):
        try:
            out_dir = os.environ.get("GWX_CLOCKS_DIR") or tempfile.gettempdir()
            os.makedirs(out_dir, exist_ok=True)
            self.path = os.path.join(out_dir, "clocks_bench_%d.csv" % os.getpid())
            self.fh = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.gpu), "--query-gpu=" + self.QUERY,
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=self.fh, stderr=subprocess.DEVNULL)
        except (OSError, FileNotFoundError):
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.fh.close()
        rows = [l.split(",") for l in open(self.path) if l.count(",") >= 8]
        if not rows:
            return None
        sm = [float(r[1]) for r in rows if r[1].strip().replace(".", "").isdigit()]
        sm_max = max(float(r[2]) for r in rows if r[2].strip().replace(".", "").isdigit())
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[j] for r in rows for j in range(4) if r[5 + j].strip() == "Active"})
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": sm_max, "reasons": reasons,
                "samples": len(rows)}


# ----------------------------------------------------------------- oracle timing
_BG_CACHE = {}


def _oracle_slice(task):
    """One oracle work item in a pool process: (workload, background step, step, first
    draw, draws) -> seconds spent (the background is regenerated when its step changes,
    as the GPU arm regenerates it every few steps)."""
    wl, bg_step, step, d0, n = task
    from oracle import pipeline
    t0 = time.perf_counter()
    if _BG_CACHE.get("step") != (wl["name"], bg_step):
        _BG_CACHE["bg"] = pipeline.background(wl, bg_step)
        _BG_CACHE["step"] = (wl["name"], bg_step)
    pipeline.simulate_batch(wl, step, draws=range(d0, d0 + n), bg=_BG_CACHE["bg"])
    return time.perf_counter() - t0


def _oracle_pool(cores):
    import concurrent.futures as cf
    import multiprocessing as mp
    return cf.ProcessPoolExecutor(max_workers=cores, mp_context=mp.get_context("spawn"))


def oracle_rate(wl, min_seconds=10.0, draws_per_worker=8, background_every=1, cores=None):
    """Injections/s of the FP64 oracle on all host cores: a pool of spawned processes (one
    per core) runs waveform, projection, injection and whitening for slices of draws
    against one background for at least ``min_seconds``; the background (noise + Welch)
    and the prior are timed on their own and charged per step (the background 1 /
    background_every of it)."""
    from oracle import pipeline, prior
    cores = cores or os.cpu_count() or 1
    t0 = time.perf_counter()
    pipeline.background(wl, 0)
    t_bg = time.perf_counter() - t0
    t0 = time.perf_counter()
    prior.sample_prior(wl["prior"], wl["param_seed"], 0, wl["B"], wl["L"], wl["N"])
    t_prior = time.perf_counter() - t0
    with _oracle_pool(cores) as ex:
        list(ex.map(_oracle_slice, [(wl, 0, 0, 0, 1)] * cores))          # start-up and background cache
        done, t0 = 0, time.perf_counter()
        while time.perf_counter() - t0 < min_seconds:
            d0 = (done * draws_per_worker) % wl["B"]
            list(ex.map(_oracle_slice, [(wl, 0, 0, (d0 + i * draws_per_worker) % (wl["B"] - draws_per_worker + 1),
                                         draws_per_worker) for i in range(cores)]))
            done += cores
        wall = time.perf_counter() - t0
    rate_draws = done * draws_per_worker / wall
    t_step = t_bg / background_every + t_prior + wl["B"] / rate_draws
    sample = ("oracle (numpy FP64) on %s, %d spawned processes (one per host core): slices of %d draws for %.1f s "
              "(%d draws), plus one background (%.2f s, charged 1/%d per step) and the prior (%.2f s); a %d-draw "
              "step extrapolated as t_bg/%d + t_prior + B / (draws per second)" %
              (wl["name"], cores, draws_per_worker, wall, done * draws_per_worker, t_bg, background_every, t_prior,
               wl["B"], background_every))
    return wl["B"] / t_step, t_step, sample, cores


def run_reference(args, wl):
    """The oracle arm: each step is a bounded sample of the workload, timed whole.  A
    step is b = draws_per_core x cores draws of the batch: the oracle's prior for them
    (on the main process), then waveform, projection, injection and whitening spread
    over one spawned process per host core, with a fresh background (noise + Welch)
    in every process every --background-every steps, as in the GPU arm.  value = draws
    timed / seconds timed; ms_per_step is the measured time of the b-draw step."""
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    cores = os.cpu_count() or 1
    per = max(1, args.reference_draws_per_core)
    b = per * cores
    R = max(1, args.background_every)
    from oracle import prior
    times = []
    with _oracle_pool(cores) as ex:
        list(ex.map(_oracle_slice, [(wl, 0, 0, 0, 1)] * cores))          # start-up
        for i in range(args.warmup + args.steps):
            t0 = time.perf_counter()
            prior.sample_prior(wl["prior"], wl["param_seed"], i, b, wl["L"], wl["N"])
            list(ex.map(_oracle_slice, [(wl, (i // R) * R, i, (k * per) % (wl["B"] - per + 1), per)
                                        for k in range(cores)]))
            dt = time.perf_counter() - t0
            if i >= args.warmup:
                times.append(dt)
    value = len(times) * b / sum(times)
    sample = ("each step: %d of the %d draws of a batch, all timed: the oracle prior for them on the main process, "
              "then waveform, projection, injection and whitening in %d spawned processes (one per host core, %d "
              "draws each), with a fresh background and its Welch PSD in every process every %d steps (those steps "
              "include it)" % (b, wl["B"], cores, per, R))
    line = {"impl": "reference", "metric": "whitened injections/sec", "value": value, "unit": "injections/s",
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * sum(times) / len(times), "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic (seeded coloured aLIGO-fit noise, Philox prior draws)",
            "config": bench_config(wl, args, 1),
            "cpu_baseline": {"value": value, "unit": "injections/s", "cores": cores, "kind": "oracle",
                             "sample": sample},
            "e2e": {"value": value, "unit": "injections/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


# ----------------------------------------------------------------- GPU arm
def loglike_leg(gwx, torch, wl, rank, lo=2000, hi=50000):
    """ln L of ragged events at the importance-weighting scale: E=64 events with
    U{lo..hi} samples each (by default 2000..50000, about 1.7 million samples) drawn
    from the prior."""
    import numpy as np
    E = 64
    counts = workloads.ragged_counts(41 + rank, E, lo, hi)
    offs = np.concatenate([[0], np.cumsum(counts)])
    S = int(offs[-1])
    sim = gwx.simulator.Simulator(dict(wl, B=E))
    y, th, _ = sim.step(step_counter(rank, 999))
    y_data = y.clone()
    theta, _ = gwx.sample_prior(wl["prior"], 77, step_counter(rank, 1), S, wl["L"], wl["N"])
    offs_d = torch.from_numpy(offs).cuda()
    out = torch.empty(S, dtype=torch.float64, device="cuda")
    for _ in range(2):
        gwx.log_likelihood(y_data, sim.psd, wl["seg_len"], wl["fs"], wl["f_lo"], wl["dets"], 0.0, theta, offs_d,
                           out=out)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    reps = 3
    e0.record()
    for _ in range(reps):
        gwx.log_likelihood(y_data, sim.psd, wl["seg_len"], wl["fs"], wl["f_lo"], wl["dets"], 0.0, theta, offs_d,
                           out=out)
    e1.record()
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / reps

    # the plain importance-sampling path: prior samples scored, then weighted per event
    def chain():
        gwx.log_likelihood(y_data, sim.psd, wl["seg_len"], wl["fs"], wl["f_lo"], wl["dets"], 0.0, theta, offs_d,
                           out=out)
        return gwx.importance_weights(out, offs_d)

    chain()
    torch.cuda.synchronize()
    e0.record()
    for _ in range(reps):
        w, ess, eff, lnz = chain()
    e1.record()
    torch.cuda.synchronize()
    chain_ms = e0.elapsed_time(e1) / reps
    ess_total = float(ess.sum().item())
    return {"value": S / (ms * 1e-3), "unit": "samples/s", "ms_per_call": ms, "samples": S, "events": E,
            "note": "plain batched-likelihood path: TaylorF2 template + projection + whitened residual per sample, "
                    "FP32 products, FP64 sums",
            "importance": {"metric": "importance-weighted posterior samples/sec (prior as proposal)",
                           "value": ess_total / (chain_ms * 1e-3), "unit": "effective samples/s",
                           "ms_per_chain": chain_ms, "ess_total": ess_total,
                           "median_efficiency": float(eff.median().item()),
                           "chain": "log_likelihood + importance_weights over all events"}}


def serving_leg(gwx, torch, rank, n_events=1000):
    """Streaming loop of the plain importance-sampling path on the 8 s, three-detector
    geometry (N = 16384): 1000 events with U{2000..50000} samples each arrive one at a
    time; per event the samples are drawn from the prior, scored by the likelihood and
    weighted (`scorer.Scorer`: preallocated buffers, C-ABI calls on one stream), and the
    event's effective sample size is read back to the host.  Latency is host time from
    the start of the event to that read."""
    import numpy as np
    from paper_2407_19048_gb300.scorer import Scorer
    wl = workloads.workload("sweep", B=n_events)
    counts = workloads.ragged_counts(5 + rank, n_events, 2000, 50000)
    sim = gwx.simulator.Simulator(wl)
    y, _, _ = sim.step(step_counter(rank, 5000))
    scorer = Scorer(wl, int(counts.max()), sim.psd)
    for e in range(5):
        scorer.score(y[e], int(counts[e]), step_counter(rank, e))
    torch.cuda.synchronize()
    lat = []
    t0 = time.perf_counter()
    for e in range(n_events):
        a = time.perf_counter()
        scorer.score(y[e], int(counts[e]), step_counter(rank, e))
        lat.append(time.perf_counter() - a)
    wall = time.perf_counter() - t0
    lat_ms = np.array(lat) * 1e3
    del sim, y, scorer
    return {"events": n_events, "samples": int(counts.sum()), "events_per_s": n_events / wall,
            "samples_per_s": float(counts.sum()) / wall, "latency_ms_p50": float(np.percentile(lat_ms, 50)),
            "latency_ms_p99": float(np.percentile(lat_ms, 99)), "latency_ms_max": float(lat_ms.max()),
            "workload": "8 s windows at 2048 Hz (N = 16384), H1+L1+V1, U{2000..50000} prior samples per event",
            "per_event": "sample_prior + log_likelihood + importance_weights + host read of ESS, efficiency, ln Z "
                         "(preallocated, one stream)"}


def gemm_leg(gwx, torch, shape=(8192, 8192, 8192)):
    """The learned part's dense product C = A B^T (bfloat16 in, FP32 accumulation,
    bfloat16 out) on the tensor cores, against cuBLAS (torch.matmul) on the same GPU."""
    M, N, K = shape
    g = torch.Generator(device="cuda")
    g.manual_seed(7)
    A = torch.randn(M, K, device="cuda", generator=g).to(torch.bfloat16)
    B = torch.randn(N, K, device="cuda", generator=g).to(torch.bfloat16)
    C = torch.empty(M, N, device="cuda", dtype=torch.bfloat16)

    def timed(fn, reps=20):
        for _ in range(3):
            fn()
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(reps):
            fn()
        b.record()
        torch.cuda.synchronize()
        return a.elapsed_time(b) / reps

    group = gwx.gemm_autotune(A, B, C)
    ms = timed(lambda: gwx.gemm_bf16(A, B, out=C))
    bias = torch.zeros(N, device="cuda", dtype=torch.float32)
    ms_dense = timed(lambda: gwx.dense_bf16(A, B, bias, act=gwx.ACT_GELU, out=C))
    gwx.device_status()
    ms_cublas = timed(lambda: torch.matmul(A, B.t(), out=C))
    flops = 2.0 * M * N * K
    peak = MEASURED_PEAKS.get("bf16_tflops")
    achieved = flops / ms / 1e9
    del A, B, C
    return {"shape": [M, N, K], "ms": ms, "tflops": achieved, "autotuned_band": group,
            "dense_bias_gelu_ms": ms_dense,
            "cublas_ms": ms_cublas,
            "cublas_tflops": flops / ms_cublas / 1e9,
            "roofline": {"bound": "tensor", "achieved": achieved, "peak": peak, "unit": "TFLOP/s",
                         "frac": achieved / peak if peak else None,
                         "peak_basis": "measured bf16 burst (MEASURED_PEAKS.json)"}}


def padded_leg(gwx, torch, rank, B=2048, N_pad=8192, reps=20):
    """Definition B (padded-grid waveforms: generate and project on an N_pad-point grid,
    inverse-transform the padded segment, inject its first N samples, whiten; five libgwx
    calls) against the fused Definition A pass, on the two-detector geometry (1024 Hz, 2 s
    windows) with B draws per step."""
    wl = workloads.workload("small", B=B)
    D = len(wl["dets"])
    n = gwx.colored_noise(wl["noise_seed"], 0, D, wl["L"], wl["fs"], wl["f_lo"])
    S = gwx.welch_psd(n, wl["fs"], wl["seg_len"], wl["seg_stride"])
    out = {}
    for name in ("definition_a_fused", "definition_b"):
        def run(i):
            if name == "definition_b":
                return gwx.simulate_batch_padded(wl["prior"], wl["param_seed"], i, n, S, wl["seg_len"], wl["fs"],
                                                 wl["f_lo"], wl["dets"], 0.0, B, wl["N"], N_pad)
            return gwx.simulate_batch(wl["prior"], wl["param_seed"], i, n, S, wl["seg_len"], wl["fs"], wl["f_lo"],
                                      wl["dets"], 0.0, B, wl["N"])
        for i in range(3):
            run(i)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        e0.record()
        for i in range(reps):
            run(step_counter(rank, 60000 + i))
        e1.record()
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1) / reps
        out[name] = {"ms_per_step": ms, "injections_per_s": B / (ms * 1e-3)}
    out.update(workload="1024 Hz, 2 s windows (N = 2048), H1+L1, %d draws per step" % B, N_pad=N_pad,
               note="Definition B pads to %d samples (%.0f s), so inspirals up to ~%.0f s long do not wrap into "
                    "the window" % (N_pad, N_pad / wl["fs"], N_pad / wl["fs"] - wl["T"] / 2))
    return out


def timed_steps(torch, sm, flush, rank, first, count, clocks=None, dist=None):
    """Run `count` simulator steps from counter `first`, each bracketed by CUDA events on
    the launching stream with the L2 flush before the first event; returns (per-step ms,
    per-step ms of the fused call from after the wait for the side-stream preparation,
    wall seconds, kernels launched)."""
    ev = [[torch.cuda.Event(enable_timing=True) for _ in range(3)] for _ in range(count)]
    torch.cuda.synchronize()
    if dist is not None:
        dist.barrier()
    if clocks is not None:
        clocks.start()
    l0 = sm.launches
    t0 = time.perf_counter()
    for i in range(count):
        flush.zero_()
        ev[i][0].record()
        sm.step(step_counter(rank, first + i), mark=ev[i][1])
        # the step ends when its fused pass and the next batch's preparation (side
        # stream) are both done, so no work of the step runs during the L2 flush
        torch.cuda.current_stream().wait_stream(sm.side)
        ev[i][2].record()
    torch.cuda.synchronize()
    wall = time.perf_counter() - t0
    if dist is not None:
        dist.barrier()
    return ([e[0].elapsed_time(e[2]) for e in ev], [e[1].elapsed_time(e[2]) for e in ev], wall,
            sm.launches - l0)


def launch_shape_record(shape):
    """What the fused pass's launch shape bits mean (staged shapes run in place)."""
    staged = bool(shape & 8)
    return {"autotuned": shape, "staged_crop_and_filter": staged, "two_buffer_passes": bool(shape & 1) and not staged,
            "blocks_per_sm": (shape >> 1) & 3 or "as many as fit"}


def roofline_alu(torch, wl, sim_ms_mean, clk):
    """Roofline object of the fused call: algorithmic FP32 flops per launch / its mean
    CUDA-event duration, against the FP32 peak of this GPU (SM count from the device,
    maximum SM clock), with the fraction at the sampled median clock beside it."""
    B, D, N = wl["B"], len(wl["dets"]), wl["N"]
    mhz, mhz_src = sm_max_mhz(clk)
    n_sm, peak = fp32_peak(torch, mhz)
    achieved = flops_per_injection(wl) * B / (sim_ms_mean * 1e-3) / 1e12
    out = {"bound": "alu", "achieved": achieved, "peak": peak, "unit": "TFLOP/s", "frac": achieved / peak,
           "traffic": traffic_per_launch(wl),
           "kernel": "simulate_prepared call (k_whiten_filter, k_simulate), timed from after the "
                     "wait for the side-stream preparation",
           "flops_per_injection": flops_per_injection(wl), "injections_per_launch": B,
           "algorithmic_bytes_per_launch": B * D * N * 4,
           "peak_basis": "%d SMs (cudaGetDeviceProperties) x %d FP32 lanes x 2 flop x %.0f MHz (%s); derived, not "
                         "measured" % (n_sm, FP32_LANES_PER_SM, mhz, mhz_src),
           "sm_count": n_sm, "avg_launch_ms": sim_ms_mean,
           "hbm_gbs_output_only": B * D * N * 4 / (sim_ms_mean * 1e-3) / 1e9}
    if clk and clk.get("sm_mhz"):
        out["frac_at_sampled_sm_clock"] = achieved / fp32_peak(torch, clk["sm_mhz"])[1]
    return out


def hl3_leg(gwx, torch, rank, args, flush, steps=200):
    """The same pipelined step on the four-second, three-detector geometry (H1+L1+V1,
    2048 Hz, N = 8192, 2048 draws per step; 201 MB of output, so the 256 MiB flush
    between steps matters), background every --background-every steps."""
    wl = workloads.workload("hl3")
    sim = gwx.simulator.Simulator(wl, pipeline=True, background_every=args.background_every)
    shape = sim.autotune(step_counter(rank, 79999))
    for i in range(args.warmup):
        sim.step(step_counter(rank, 80000 + i))
    step_ms, sim_ms, _, _ = timed_steps(torch, sim, flush, rank, 80000 + args.warmup, steps)
    del sim
    ms = statistics.mean(step_ms)
    roof = roofline_alu(torch, wl, statistics.mean(sim_ms), None)
    roof["launch_shape"] = launch_shape_record(shape)
    return {"workload": describe(wl), "steps": steps, "ms_per_step": ms, "injections_per_s": wl["B"] / (ms * 1e-3),
            "roofline": roof}


def conv_leg(gwx, torch, reps=20):
    """The ResNet's stage-1 convolution at its training shape (512 windows x 512 steps,
    64 -> 64 channels, kernel 5, bfloat16 operands, FP32 outputs): the implicit GEMM
    (gwx_conv1d_bf16 and its backward with the residual-gradient addend) against the
    im2col rows + dense product route, CUDA events over `reps` calls each."""
    B, T, C, O, k = 512, 512, 64, 64, 5
    g = torch.Generator(device="cuda").manual_seed(7)
    x = torch.randn((B, T, C), device="cuda", generator=g).to(torch.bfloat16)
    W = (torch.randn((O, k * C), device="cuda", generator=g) * (2.0 / (k * C)) ** 0.5).to(torch.bfloat16)
    dz = torch.randn((B, T, O), device="cuda", generator=g)
    add = torch.randn((B, T, C), device="cuda", generator=g)
    lib = gwx._lib.load()
    nb = lib.gwx_conv1d_bf16_backward_workspace(B, T, C, O, k)
    ws = gwx._workspace(nb, x.device)
    cols = torch.empty((B * T, k * C), dtype=torch.bfloat16, device="cuda")
    dxe = torch.empty((B, T, C), dtype=torch.float32, device="cuda")

    def implicit_fwd():
        gwx.conv1d_bf16(x, W, k)

    def implicit_bwd():
        gwx.conv1d_bf16_backward(dz, x, W, k, addend=add, workspace=ws)

    def explicit_fwd():
        gwx._check(lib.gwx_im2col(gwx._ptr(x), B, T, C, k, 1, 2, k * C, gwx._ptr(cols), gwx._stream()))
        gwx.dense_bf16(cols, W, None, act=gwx.ACT_NONE, out_dtype=torch.float32)

    def explicit_bwd():
        gwx._check(lib.gwx_im2col(gwx._ptr(x), B, T, C, k, 1, 2, k * C, gwx._ptr(cols), gwx._stream()))
        dcols, _, _ = gwx.dense_bf16_backward(cols, W, None, dz.reshape(B * T, O), act=gwx.ACT_NONE)
        gwx._check(lib.gwx_col2im(gwx._ptr(dcols), B, T, C, k, 1, 2, k * C, gwx._ptr(add), gwx._ptr(dxe),
                                  gwx._stream()))

    def timed(fn):
        for _ in range(3):
            fn()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(reps):
            fn()
        e1.record()
        torch.cuda.synchronize()
        return e0.elapsed_time(e1) / reps

    t = {"implicit_forward_ms": timed(implicit_fwd), "implicit_backward_ms": timed(implicit_bwd),
         "im2col_forward_ms": timed(explicit_fwd), "im2col_backward_ms": timed(explicit_bwd)}
    peaks = _measured_peaks()
    hbm = float(peaks.get("hbm_gbs") or 6800.0)
    fwd_bytes = B * T * C * 2 + O * k * C * 2 + B * T * O * 4      # x read, W read, z written
    gbs = fwd_bytes / (t["implicit_forward_ms"] * 1e-3) / 1e9
    t["shape"] = {"B": B, "T": T, "C": C, "O": O, "k": k}
    t["forward_flop"] = 2 * B * T * O * k * C
    t["roofline_forward"] = {"bound": "hbm", "achieved": gbs, "peak": hbm, "unit": "GB/s", "frac": gbs / hbm,
                             "algorithmic_bytes": fwd_bytes,
                             "peak_basis": "measured copy bandwidth (MEASURED_PEAKS.json)" if peaks.get("hbm_gbs")
                             else "fallback 6800 GB/s"}
    return t


def flow_resnet_leg(gwx, torch, rank, steps=1500, batch=512, events=64, pretrain_steps=800, pretrain_batch=256,
                    pretrain_lr=1e-4):
    """The flow with the paper's ResNet-1D data summary (stem, (5, 3, 3) residual blocks of
    64 / 128 / 256 channels, group norm, kernel 5; convolutions on the tensor cores) in
    place of the spectral-feature network, trained jointly with AdamW on 512-draw batches
    of the non-spinning two-detector workload; importance sampling of the 64 two-detector
    events of U{2000..50000} draws as in the flow leg.  A second arm first pre-trains the ResNet with VICReg on the raw
    whitened strain (Sec. 4.1: two views per source that differ in the merger time,
    expander 64 -> 128 -> 24, weights 1, 1, 5; 800 steps of 256 view pairs at a learning
    rate of 1e-4 -- at 1e-3 or 3e-4 the flow trained after it was behind the plain arm),
    then trains the flow the same way."""
    import paper_2407_19048_gb300.simulator  # noqa: F401
    from paper_2407_19048_gb300.flow import FlowPosterior
    from paper_2407_19048_gb300.pretrain import VICRegPretrainer
    wl = workloads.workload("small_nonspinning", B=batch)
    wl_ev = dict(workloads.workload("small_nonspinning", B=events), param_seed=777)
    sim_ev = gwx.simulator.Simulator(wl_ev)
    y_ev, _, _ = sim_ev.step(step_counter(rank, 0))
    y_ev = y_ev.clone()
    psd_ev = sim_ev.psd.clone()
    del sim_ev
    counts = workloads.ragged_counts(4, events, 2000, 50000)

    def arm(pretrain):
        sim = gwx.simulator.Simulator(wl, pipeline=True, background_every=16)
        fp = FlowPosterior(wl, layers=16, hidden=256, context=64, seed=0, lr=3e-4, weight_decay=2e-3,
                           embedding="resnet")
        out = {}
        if pretrain:
            pt = VICRegPretrainer(fp, batch=pretrain_batch, lr=pretrain_lr, seed=7)
            pt.step(0)
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            trace = []
            for k in range(1, pretrain_steps + 1):
                loss, terms = pt.step(k)
                if k % max(1, pretrain_steps // 8) == 0 or k == 1 or k == pretrain_steps:
                    trace.append((k, loss.clone(), terms.clone()))
            torch.cuda.synchronize()
            out["pretraining"] = {
                "steps": pretrain_steps, "view_pairs_per_step": pretrain_batch, "lr": pretrain_lr,
                "s": time.perf_counter() - t0,
                "loss": [(k, float(l.item())) for k, l, _ in trace],
                "terms_last": [float(v) for v in trace[-1][2].cpu()],
                "terms_note": "invariance, variance x, variance x', covariance x, covariance x'"}
            del pt
        y, th, _ = sim.step(step_counter(rank, 90000))
        fp.train_step(y, th, update=False)
        torch.cuda.synchronize()
        # the first `eager` steps issued call by call, the rest as CUDA-graph replays (one
        # graph per simulator buffer set, captured on first use; the replay timing starts
        # after the captures)
        eager = min(20, steps)
        timed = eager + 4
        graphs, losses = {}, []
        t0 = time.perf_counter()
        for i in range(steps):
            if i == eager:
                torch.cuda.synchronize()
                t_eager = time.perf_counter() - t0
            if i == timed:
                torch.cuda.synchronize()
                t1 = time.perf_counter()
            y, th, _ = sim.step(step_counter(rank, 90001 + i))
            if i < eager:
                loss = fp.train_step(y, th)
            else:
                g = graphs.get(y.data_ptr())
                if g is None:
                    g = graphs[y.data_ptr()] = fp.capture_train_step(y, th)
                g.replay()
                fp.note_replay()
                loss = fp._loss
            if i % max(1, steps // 8) == 0 or i == steps - 1:
                losses.append((i, loss.clone()))
        torch.cuda.synchronize()
        t2 = time.perf_counter()
        train_s = t2 - t0
        step_eager = 1e3 * t_eager / eager if steps > eager else None
        step_graph = 1e3 * (t2 - t1) / (steps - timed) if steps > timed else None
        ncap = len(graphs)
        del sim, graphs
        out.update({"train_steps": steps, "batch": batch, "train_s": train_s, "step_ms": step_graph,
                    "step_ms_eager": step_eager, "graph_captures": ncap,
                    "loss": [(i, float(l.item())) for i, l in losses],
                    "importance_sampling": is_compare(gwx, torch, fp, wl_ev, y_ev, psd_ev, counts,
                                                      workloads.tc_grid(wl_ev))})
        out["resnet_params"] = sum(p.numel() for _, p, _ in fp.resnet.tensors())
        return out

    res = dict(summary="ResNet-1D", **arm(False))
    if pretrain_steps > 0:
        res["vicreg_pretrained"] = arm(True)
    return res


def tmarg_leg(gwx, torch, events=64, lo=2000, hi=50000, reps=3, oversample=None, n_tc=None):
    """The likelihood with the merger time integrated out (`gwx_log_likelihood_tmarg`)
    alone, at the importance-sampling scale: `events` two-detector events of the non-spinning workload
    with U{lo..hi} prior samples each, the merger time integrated over the prior's window
    on a grid 16 times finer than the sampling interval (u = 16 inverse transforms of
    n = N/2 = 1024 packed points per sample; `oversample` and `n_tc` override u and the
    window's length in samples).  CUDA-event time per call, best of `reps`.
    Roofline: the u transforms' 5 n log2 n flops per sample (the band products and the
    log-sum-exp not counted) against the FP32 peak."""
    import numpy as np
    import paper_2407_19048_gb300.simulator  # noqa: F401
    wl = dict(workloads.workload("small_nonspinning", B=events), param_seed=777)
    sim = gwx.simulator.Simulator(wl)
    y, _, _ = sim.step(step_counter(0, 0))
    counts = workloads.ragged_counts(4, events, lo, hi)
    offs = torch.from_numpy(np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)).cuda()
    S = int(counts.sum())
    theta, _ = gwx.sample_prior(wl["prior"], 5, 0, S, wl["L"], wl["N"])
    tc_lo, n_tc0, u0 = workloads.tc_grid(wl)
    u = u0 if oversample is None else int(oversample)
    n_tc = n_tc0 if n_tc is None else int(n_tc)
    out = torch.empty(S, dtype=torch.float64, device="cuda")

    def call():
        gwx.log_likelihood_tmarg(y, sim.psd, wl["seg_len"], wl["fs"], wl["f_lo"], wl["dets"], 0.0, tc_lo, n_tc, u,
                                 theta, offs, out=out)

    call()
    torch.cuda.synchronize()
    best = None
    for _ in range(reps):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        call()
        e1.record()
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1)
        best = ms if best is None else min(best, ms)
    n = wl["N"] // 2
    flops = u * 5 * n * int(math.log2(n))
    mhz, mhz_src = sm_max_mhz(None)
    n_sm, peak = fp32_peak(torch, mhz)
    achieved = flops * S / (best * 1e-3) / 1e12
    return {"samples": S, "events": events, "grid": {"tc_lo": tc_lo, "n_tc": n_tc, "oversample": u},
            "ms_per_call": best, "ns_per_sample": best * 1e6 / S, "samples_per_s": S / (best * 1e-3),
            "roofline": {"bound": "alu", "achieved": achieved, "peak": peak, "unit": "TFLOP/s",
                         "frac": achieved / peak, "flops_per_sample": flops,
                         "peak_basis": "%d SMs x %d FP32 lanes x 2 flop x %.0f MHz (%s); derived" %
                                       (n_sm, FP32_LANES_PER_SM, mhz, mhz_src)}}


def is_compare(gwx, torch, fp, wl, y_ev, psd, counts, grid, seed=5, reps=3):
    """Importance sampling of events y_ev [E][D][N] with counts[e] draws each, from the
    prior and from the flow, every draw scored by the likelihood with the merger time
    integrated out over `grid` and weighted (ln w = ln L + ln prior - ln q).  Device
    time (CUDA events) of draws + ln L + weights, best of `reps`; every repetition draws
    the same samples (the same counter), so the per-event ESS and efficiency (with their
    medians) do not depend on which repetition was fastest."""
    import numpy as np
    offs = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    S = int(offs[-1])
    offs_d = torch.from_numpy(offs).cuda()
    tc_lo, n_tc, u = grid
    out = {}
    for arm in ("prior", "flow"):
        best, keep = None, None
        for rep in range(reps):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            e0.record()
            if arm == "flow":
                theta, _, lrat = fp.sample(y_ev, offs_d, seed, 0, S=S)
            else:
                theta, _ = gwx.sample_prior(wl["prior"], seed, 0, S, wl["L"], wl["N"])
                lrat = None
            lnl = gwx.log_likelihood_tmarg(y_ev, psd, wl["seg_len"], wl["fs"], wl["f_lo"], wl["dets"], 0.0, tc_lo,
                                           n_tc, u, theta, offs_d)
            _, ess, eff, _ = gwx.importance_weights(lnl, offs_d, lrat)
            e1.record()
            torch.cuda.synchronize()
            ms = e0.elapsed_time(e1)
            if best is None or ms < best:
                best, keep = ms, (ess.cpu().numpy(), eff.cpu().numpy())
        ess, eff = keep
        out[arm] = {"ess_total": float(ess.sum()), "ess_median": float(np.median(ess)),
                    "efficiency_median": float(np.median(eff)), "chain_ms": best,
                    "ess_per_s": float(ess.sum()) / (best * 1e-3),
                    "ess_per_event": [round(float(v), 3) for v in ess]}
    pe, fe = np.array(out["prior"]["ess_per_event"]), np.array(out["flow"]["ess_per_event"])
    out["per_event_ess_ratio_median"] = float(np.median(fe / np.maximum(pe, 1e-300)))
    out["events_flow_ahead"] = int(np.sum(fe > pe))
    out["samples"] = S
    out["events"] = len(counts)
    out["likelihood"] = ("gwx_log_likelihood_tmarg: merger time integrated out over [%g, %g) s on a %g us grid"
                         % (tc_lo, tc_lo + n_tc / wl["fs"], 1e6 / (u * wl["fs"])))
    return out


def flow_leg(gwx, torch, rank, steps=12000, events=64, pp_events=200, pp_samples=500, lr=1e-3, batch=4096,
             layers=16, hidden=256, clip=1.0):
    """The learned part (the flow trained on 4096-draw batches of the two-detector workload)
    and its importance-sampling judge (64 events of U{2000..50000} draws).

    The conditional coupling flow (16 affine coupling layers, conditioners 72 -> 256 ->
    256 -> 8; embedding 1968 -> 512 -> 512 -> 64 on log group powers, inter-detector
    cross spectra and lag-one spectral products; tcgen05 dense layers) is trained with
    AdamW (lr 1e-3, weight decay 2e-3, gradient norm clipped at 1) on batches of the
    non-spinning two-detector workload, one CUDA-graph replay of the C-ABI training
    call per step, with the schedule of Sec. 5: epochs of 160,000 simulations, the
    learning rate divided by 10 after 10 epochs without a better validation loss, stop
    after 50 (or at the step budget), best epoch restored.  Then: 20,000 posterior draws
    of one event (the paper's inference size); importance sampling of 64 events with
    U{2000..50000} draws each from the flow and from the prior, every draw scored by the
    likelihood with the merger time integrated out (the flow does not model it; spins
    are zero in the model and the events); a PP test of the flow's marginals; a
    streaming loop of 1000 events; sky maps."""
    import math
    import numpy as np
    import paper_2407_19048_gb300.simulator  # noqa: F401
    from paper_2407_19048_gb300.flow import FlowPosterior
    wl = workloads.workload("small_nonspinning", B=batch)
    grid = workloads.tc_grid(wl)
    sim = gwx.simulator.Simulator(wl, pipeline=True, background_every=16)
    fp = FlowPosterior(wl, layers=layers, hidden=hidden, context=64, embed_hidden=512, group=4, seed=0, lr=lr,
                       weight_decay=2e-3, clip=clip)
    # fixed validation set: 4 x 4096 simulations from counters no training batch uses
    sim_v = gwx.simulator.Simulator(dict(wl, B=16384, param_seed=911))
    yv, thv, _ = sim_v.step(step_counter(rank, 7))
    yv, thv = yv.clone(), thv.clone()
    del sim_v
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    hist = fp.fit(sim, steps, step_counter(rank, 40000), (yv, thv))
    torch.cuda.synchronize()
    train_s = time.perf_counter() - t0
    del yv, thv
    # training step alone (no simulation) on one resident batch, eager and as a graph replay
    y1, th1, _ = sim.step(step_counter(rank, 39999))
    y1, th1 = y1.clone(), th1.clone()
    fp_t = FlowPosterior(wl, layers=layers, hidden=hidden, context=64, embed_hidden=512, group=4, seed=1)
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    for _ in range(3):
        fp_t.train_step(y1, th1)
    ev0.record()
    for _ in range(50):
        fp_t.train_step(y1, th1)
    ev1.record()
    torch.cuda.synchronize()
    step_ms = ev0.elapsed_time(ev1) / 50
    graph = fp_t.capture_train_step(y1, th1)
    for _ in range(3):
        graph.replay()
    ev0.record()
    for _ in range(50):
        graph.replay()
    ev1.record()
    torch.cuda.synchronize()
    step_graph_ms = ev0.elapsed_time(ev1) / 50
    del graph, fp_t, y1, th1
    # events: the importance-sampling workload's 64 events of the same generator (other
    # parameter seed)
    wl_ev = dict(workloads.workload("small_nonspinning", B=events), param_seed=777)
    sim_ev = gwx.simulator.Simulator(wl_ev)
    y_ev, th_ev, _ = sim_ev.step(step_counter(rank, 0))
    y_ev, th_ev = y_ev.clone(), th_ev.clone()
    # posterior sampling latency: 20,000 draws for one event
    one = torch.tensor([0, 20000], dtype=torch.int64, device="cuda")
    lat = []
    y1 = y_ev[:1].contiguous()
    for rep in range(23):
        torch.cuda.synchronize()
        a = time.perf_counter()
        fp.sample(y1, one, 11, rep, S=20000)
        torch.cuda.synchronize()
        if rep >= 3:
            lat.append(time.perf_counter() - a)
    lat.sort()
    # sky maps: 20,000 draws + marginal likelihood + weights + HEALPix map
    sky = {}
    for nside in (32, 64, 128):
        times = []
        for rep in range(13):
            torch.cuda.synchronize()
            a0 = time.perf_counter()
            theta1, _, lr1 = fp.sample(y1, one, 17, rep, S=20000)
            lnl1 = gwx.log_likelihood_tmarg(y1, sim_ev.psd, wl_ev["seg_len"], wl_ev["fs"], wl_ev["f_lo"],
                                            wl_ev["dets"], 0.0, *grid, theta1, one)
            w1, _, _, _ = gwx.importance_weights(lnl1, one, lr1)
            gwx.skymap(theta1, nside, weights=w1)
            torch.cuda.synchronize()
            if rep >= 3:
                times.append(time.perf_counter() - a0)
        times.sort()
        sky[str(nside)] = times[len(times) // 2] * 1e3
    # sky density (the paper's map: 20,000 draws, then the flow's density at every pixel;
    # ~0.6 / 1.2 / 2.4 s at NSIDE 32 / 64 / 128 on an A40)
    sky_density = {}
    for nside in (32, 64, 128):
        times = []
        for rep in range(13):
            torch.cuda.synchronize()
            a0 = time.perf_counter()
            theta1, lq1, _ = fp.sample(y1, one, 19, rep, S=20000)
            fp.skymap(y1, theta1, lq1, nside)
            torch.cuda.synchronize()
            if rep >= 3:
                times.append(time.perf_counter() - a0)
        times.sort()
        sky_density[str(nside)] = times[len(times) // 2] * 1e3
    # importance sampling, flow vs prior, 64 events x U{2000..50000} draws
    counts = workloads.ragged_counts(4, events, 2000, 50000)
    isamp = is_compare(gwx, torch, fp, wl_ev, y_ev, sim_ev.psd, counts, grid)
    # PP test: percentile of each truth among its event's flow draws, per flow coordinate
    wl_pp = dict(workloads.workload("small_nonspinning", B=pp_events), param_seed=779)
    sim_pp = gwx.simulator.Simulator(wl_pp)
    y_pp, th_pp, _ = sim_pp.step(step_counter(rank, 2))
    offs_pp = torch.arange(pp_events + 1, dtype=torch.int64, device="cuda") * pp_samples
    theta_s, _, lr_s = fp.sample(y_pp, offs_pp, 13, 0, S=pp_events * pp_samples)
    xs = gwx.flow_targets(theta_s, fp.mean, fp.scale).cpu().numpy().reshape(pp_events, pp_samples, 8)
    ok = np.isfinite(lr_s.cpu().numpy()).reshape(pp_events, pp_samples)
    xt = gwx.flow_targets(th_pp, fp.mean, fp.scale).cpu().numpy()
    ks = []
    for p in range(8):
        pct = np.array([np.mean(xs[e, ok[e], p] < xt[e, p]) if ok[e].any() else 0.5 for e in range(pp_events)])
        uu = np.sort(pct)
        n = len(uu)
        ks.append(float(max(np.max(np.arange(1, n + 1) / n - uu), np.max(uu - np.arange(n) / n))))
    # streaming: 1000 events of U{2000..50000} draws, one at a time, flow vs prior proposal
    from paper_2407_19048_gb300.scorer import Scorer
    n_srv = 1000
    wl_srv = dict(workloads.workload("small_nonspinning", B=n_srv), param_seed=780)
    sim_srv = gwx.simulator.Simulator(wl_srv)
    y_srv, _, _ = sim_srv.step(step_counter(rank, 3))
    counts_srv = workloads.ragged_counts(6 + rank, n_srv, 2000, 50000)
    serving = {}
    for name, flow in (("prior", None), ("flow", fp)):
        sc = Scorer(wl_srv, int(counts_srv.max()), sim_srv.psd, flow=flow, tmarg=grid)
        for e in range(5):
            sc.score(y_srv[e:e + 1], int(counts_srv[e]), e)
        torch.cuda.synchronize()
        lat_srv, ess = [], []
        t0 = time.perf_counter()
        for e in range(n_srv):
            a = time.perf_counter()
            ess.append(sc.score(y_srv[e:e + 1], int(counts_srv[e]), e)[0])
            lat_srv.append(time.perf_counter() - a)
        wall = time.perf_counter() - t0
        lat_ms = np.array(lat_srv) * 1e3
        serving[name] = {"events_per_s": n_srv / wall, "latency_ms_p50": float(np.percentile(lat_ms, 50)),
                         "latency_ms_p99": float(np.percentile(lat_ms, 99)), "ess_total": float(np.sum(ess)),
                         "ess_median": float(np.median(ess)), "ess_per_s": float(np.sum(ess)) / wall}
        del sc
    del sim, sim_ev, sim_pp, sim_srv
    return {"shape": fp.shape, "params": fp.n_params, "batch": batch, "train_s": train_s,
            "simulations_per_s": hist["steps_run"] * batch / train_s, "schedule": hist,
            "train_step_ms": step_ms, "train_step_graph_ms": step_graph_ms,
            "sample_20000_ms": {"p50": lat[len(lat) // 2] * 1e3, "min": lat[0] * 1e3, "max": lat[-1] * 1e3},
            "skymap_density_20000_ms": dict(sky_density, note="sample_posterior 20k + flow_skymap (the flow's density "
                                                              "at every HEALPix pixel centre), median of 10, host time"),
            "skymap_20000_ms": dict(sky, note="sample_posterior 20k + log_likelihood_tmarg + importance_weights + "
                                              "skymap (HEALPix nested, importance-weighted histogram), median of 10, "
                                              "host time"),
            "importance_sampling": isamp,
            "pp_test": {"events": pp_events, "draws_per_event": pp_samples, "ks_distance": ks,
                        "ks_95pct_critical": 1.36 / math.sqrt(pp_events),
                        "coords": ["Mc", "q", "D_L", "cos theta_JN", "RA", "sin dec", "psi", "phic"]},
            "serving": dict(serving, events=n_srv, draws="U{2000..50000} per event",
                            per_event="draws (prior or flow) + log_likelihood_tmarg + importance_weights + host read"),
            "note": "loss = batch mean of -ln q_x(x) in standardised coordinates; validation loss = mean -ln q_r of "
                    "16,384 fixed simulations; the merger time is integrated out of the likelihood, spins are zero "
                    "in the model and the events"}


def cufft_leg(gwx, torch, sim, wl, fused_ms):
    """The shared-memory FFT kernels against cuFFT (called through torch.fft) on the
    batch's shape, B x D rows of N real samples.  cuFFT is a timing baseline here only:
    nothing on the product path calls it."""
    B, D, N = sim.y.shape
    F = N // 2 + 1
    x = sim.y.clone()
    X = torch.empty((B, D, F), dtype=torch.complex64, device=x.device)
    Xc = torch.empty_like(X)
    yo = torch.empty_like(x)
    Wt = torch.rand((D, F), dtype=torch.float32, device=x.device)
    lib = gwx._lib.load()
    ws, nb = gwx._workspace(lib.gwx_whiten_workspace(D, N), x.device)

    def ours_whiten():
        gwx._check(lib.gwx_whiten(gwx._ptr(x), gwx._ptr(sim.psd), wl["seg_len"], wl["fs"], wl["f_lo"], B, D, N,
                                  gwx._ptr(yo), gwx._ptr(ws), nb, gwx._stream()))

    def cufft_whiten():
        torch.fft.rfft(x, dim=-1, out=Xc)
        Xc.mul_(Wt)
        torch.fft.irfft(Xc, n=N, dim=-1, out=yo)

    def timed(fn, reps=20):
        for _ in range(3):
            fn()
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(reps):
            fn()
        b.record()
        torch.cuda.synchronize()
        return a.elapsed_time(b) / reps

    res = {"rows": B * D, "N": N,
           "gwx_rfft_ms": timed(lambda: gwx.rfft(x, out=X)),
           "cufft_rfft_ms": timed(lambda: torch.fft.rfft(x, dim=-1, out=Xc)),
           "gwx_irfft_ms": timed(lambda: gwx.irfft(X, N, out=yo)),
           "cufft_irfft_ms": timed(lambda: torch.fft.irfft(Xc, n=N, dim=-1, out=yo)),
           "gwx_whiten_ms": timed(ours_whiten),
           "cufft_whiten_ms": timed(cufft_whiten),
           "gwx_fused_simulate_ms": fused_ms,
           "note": "inputs (201 MB) exceed L2; the fused pass also crops, evaluates and injects the waveforms"}
    return res


# The main figures of the further legs, as the printed line names them: where they lie in the record.
LEG_FIGURES = {
    "hl3_ms": "hl3.ms_per_step", "log_likelihood_ms": "log_likelihood.ms_per_call",
    "importance_eff_per_s": "log_likelihood.importance.value", "tmarg_ms": "log_likelihood_tmarg.ms_per_call",
    "tmarg_frac": "log_likelihood_tmarg.roofline.frac", "serving_events_per_s": "serving.events_per_s",
    "serving_p99_ms": "serving.latency_ms_p99", "gemm_ms": "gemm_bf16.ms", "cublas_ms": "gemm_bf16.cublas_ms",
    "dense_gelu_ms": "gemm_bf16.dense_bias_gelu_ms", "whiten_ms": "fft_vs_cufft.gwx_whiten_ms",
    "cufft_whiten_ms": "fft_vs_cufft.cufft_whiten_ms", "flow_step_ms": "flow.train_step_ms",
    "flow_step_graph_ms": "flow.train_step_graph_ms", "flow_sample_20000_ms": "flow.sample_20000_ms.p50",
    "flow_skymap_ms": "flow.skymap_20000_ms.64", "flow_ess_per_s": "flow.importance_sampling.flow.ess_per_s",
    "prior_ess_per_s": "flow.importance_sampling.prior.ess_per_s", "resnet_step_ms": "flow_resnet.step_ms",
    "conv_forward_ms": "conv1d_stage1.implicit_forward_ms", "conv_backward_ms": "conv1d_stage1.implicit_backward_ms",
    "padded_b_ms": "padded_grid.definition_b.ms_per_step"}


def short_line(record):
    """The line to print from the whole record: every scalar of the top level, the configuration and the clocks as they
    are, the figures of the bounds and of the end-to-end loop without their notes, and the legs' main figures.  The
    record itself runs to 23,000 characters (per-event lists, loss curves), which callers that keep the end of the
    output cut off at its front, where the value stands."""
    line = {k: v for k, v in record.items() if not isinstance(v, (dict, list))}
    for k in ("config", "clocks"):
        line[k] = record[k]
    for k, drop in (("roofline", ("kernel", "peak_basis", "launch_shape")), ("e2e", ("path",)),
                    ("cpu_baseline", ("sample",))):
        line[k] = record[k] and {n: v for n, v in record[k].items() if n not in drop}
    legs = {}
    for name, path in LEG_FIGURES.items():
        v = record
        for part in path.split("."):
            v = v.get(part) if isinstance(v, dict) else None
        if v is not None:
            legs[name] = float("%.5g" % v)
    line["legs"] = legs
    return line


def run_gpu(args, wl):
    import torch
    import torch.distributed as dist
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    dd = dist if world > 1 else None
    import paper_2407_19048_gb300 as gwx
    import paper_2407_19048_gb300.simulator  # noqa: F401
    gwx.init()
    sim = gwx.simulator.Simulator(wl, pipeline=True, background_every=args.background_every)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    B, D, N, L = wl["B"], len(wl["dets"]), wl["N"], wl["L"]
    # the fused pass's launch shape for this (N, D), chosen by timing the bit-identical
    # candidates before the warm-up
    shape = sim.autotune(step_counter(rank, 1 << 19))

    for i in range(args.warmup):
        sim.step(step_counter(rank, i))
    clocks = ClockSampler(local)
    step_ms, sim_ms, t_wall, launches = timed_steps(torch, sim, flush, rank, args.warmup, args.steps, clocks, dd)
    clk = clocks.stop()
    total_s = max_over_ranks(sum(step_ms) * 1e-3, dd)
    value = world * B * args.steps / total_s

    if args.only_step:
        if rank == 0:
            print(json.dumps({"metric": "whitened injections/sec", "value": value, "unit": "injections/s",
                              "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
                              "ms_per_step": 1e3 * total_s / args.steps, "config": {"workload": describe(wl)},
                              "launch_shape": shape, "roofline": roofline_alu(torch, wl, statistics.mean(sim_ms), clk),
                              "note": "--only-step profiling run: no end-to-end, likelihood or CPU legs"}), flush=True)
        if world > 1:
            dist.destroy_process_group()
        return 0

    # the same loop with a fresh background (colored noise + Welch PSD) every step
    sim1 = gwx.simulator.Simulator(wl, pipeline=True, background_every=1)
    n1 = min(args.steps, 500)
    for i in range(args.warmup):
        sim1.step(step_counter(rank, args.warmup + args.steps + i))
    ms1, _, _, _ = timed_steps(torch, sim1, flush, rank, 2 * args.warmup + args.steps, n1)
    value_bg1 = world * B * n1 / max_over_ranks(sum(ms1) * 1e-3, dd)
    del sim1

    # end to end: background strain from pinned host memory in, products out to pinned
    # host memory.  Batch i's whitened output leaves on a copy stream while batch i + 1
    # is computed (two output buffers in the pipelined simulator); the parameters and
    # offsets are read back on the launching stream.
    host_bg = torch.empty((D, L), dtype=torch.float32, pin_memory=True)
    host_bg.copy_(sim.noise)
    host_y = [torch.empty((B, D, N), dtype=torch.float32, pin_memory=True) for _ in range(2)]
    host_th = torch.empty((11, B), dtype=torch.float64, pin_memory=True)
    host_off = torch.empty(B, dtype=torch.int64, pin_memory=True)
    del sim
    sim_e2e = gwx.simulator.Simulator(wl, noise_on_device=False, pipeline=True, background_every=1)
    copy_stream = torch.cuda.Stream()
    ev_ready = torch.cuda.Event()
    ev_copied = [torch.cuda.Event(), torch.cuda.Event()]
    h2d = host_bg.numel() * 4
    d2h = host_y[0].numel() * 4 + host_th.numel() * 8 + host_off.numel() * 8
    main_stream = torch.cuda.current_stream()

    def e2e_steps(first, count):
        for i in range(count):
            slot = i % 2
            if i >= 2:   # y of this slot is rewritten below: its copy to the host must be done
                main_stream.wait_event(ev_copied[slot])
            sim_e2e.noise.copy_(host_bg, non_blocking=True)
            y, th, off = sim_e2e.step(step_counter(rank, first + i))
            host_th.copy_(th, non_blocking=True)
            host_off.copy_(off, non_blocking=True)
            ev_ready.record(main_stream)
            copy_stream.wait_event(ev_ready)
            with torch.cuda.stream(copy_stream):
                host_y[slot].copy_(y, non_blocking=True)
                ev_copied[slot].record(copy_stream)
        main_stream.wait_stream(copy_stream)

    e2e_steps(0, max(3, args.warmup))
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    n_e2e = min(args.steps, 1000)
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    e2e_steps(args.warmup + 100, n_e2e)
    b.record()
    b.synchronize()
    e2e_s = max_over_ranks(a.elapsed_time(b) * 1e-3, dd)
    e2e_value = world * B * n_e2e / e2e_s
    del sim_e2e
    # the device-to-host link alone: the step's output bytes copied from device memory to
    # pinned host memory, three times on one stream (splitting the copy over 2, 4 or 8
    # streams measured the same rate), the bound of the end-to-end loop
    dev_y = torch.zeros_like(host_y[0], device="cuda")
    host_y[0].copy_(dev_y, non_blocking=True)
    torch.cuda.synchronize()
    a.record()
    for _ in range(3):
        host_y[0].copy_(dev_y, non_blocking=True)
    b.record()
    b.synchronize()
    d2h_link_gbs = 3 * dev_y.numel() * 4 / (a.elapsed_time(b) * 1e-3) / 1e9
    e2e_d2h_gbs = d2h * n_e2e / e2e_s / 1e9
    del dev_y, host_y

    hl3 = hl3_leg(gwx, torch, rank, args, flush)
    wl_hl3 = workloads.workload("hl3")
    sim_h = gwx.simulator.Simulator(wl_hl3, pipeline=True, background_every=args.background_every)
    for i in range(3):
        sim_h.step(step_counter(rank, 85000 + i))
    ll = loglike_leg(gwx, torch, wl_hl3, rank)
    fft_cmp = cufft_leg(gwx, torch, sim_h, wl_hl3, hl3["roofline"]["avg_launch_ms"])
    del sim_h
    serve = serving_leg(gwx, torch, rank)
    gemm = gemm_leg(gwx, torch)
    flow = flow_leg(gwx, torch, rank)
    flow_resnet = flow_resnet_leg(gwx, torch, rank)
    tmarg = tmarg_leg(gwx, torch)
    conv1d = conv_leg(gwx, torch)
    padded = padded_leg(gwx, torch, rank)

    roof = roofline_alu(torch, wl, statistics.mean(sim_ms), clk)
    roof["launch_shape"] = launch_shape_record(shape)

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        rate, t_step, sample, cores = oracle_rate(wl, background_every=args.background_every)
        cpu = {"value": rate, "unit": "injections/s", "cores": cores, "kind": "oracle", "sample": sample}

    if world > 1:
        dist.barrier()
    if rank == 0:
        record = {
            "metric": "whitened injections/sec", "value": value, "unit": "injections/s", "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * total_s / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic (seeded coloured aLIGO-fit noise, Philox prior draws)",
            "config": bench_config(wl, args, world),
            "roofline": roof,
            "cpu_baseline": cpu,
            "e2e": {"value": e2e_value, "unit": "injections/s", "h2d_bytes_per_step": h2d,
                    "d2h_bytes_per_step": d2h,
                    "path": "every step: background strain H2D from pinned host memory, welch_psd, prepare_batch "
                            "and simulate_prepared, whitened batch + parameters + offsets D2H to pinned host "
                            "memory; batch i's output copy overlaps batch i + 1's compute",
                    "steps": n_e2e, "d2h_gbs": e2e_d2h_gbs, "d2h_link_gbs": d2h_link_gbs,
                    "d2h_frac_of_link": e2e_d2h_gbs / d2h_link_gbs},
            "gpu_launches": launches,
            "value_background_every_step": value_bg1,
            "clocks": clk,
            "hl3": hl3,
            "log_likelihood": ll,
            "fft_vs_cufft": fft_cmp,
            "serving": serve,
            "gemm_bf16": gemm,
            "flow": flow,
            "flow_resnet": flow_resnet, "log_likelihood_tmarg": tmarg, "conv1d_stage1": conv1d,
            "padded_grid": padded,
            "wall_s_timed_region": t_wall,
        }
        if args.record:
            with open(args.record, "w") as fh:
                fh.write(json.dumps(record) + "\n")
        print(json.dumps(short_line(record)), flush=True)
    if world > 1:
        dist.destroy_process_group()
    return 0


def main(argv=None):
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=4000)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="gwx", choices=["gwx", "reference"])
    ap.add_argument("--workload", default=WORKLOAD, choices=sorted(workloads.WORKLOADS))
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--reference-draws-per-core", type=int, default=8,
                    help="draws per host core in each step of the oracle arm")
    ap.add_argument("--background-every", type=int, default=16,
                    help="regenerate the background and its PSD every this many steps")
    ap.add_argument("--batch", type=int, default=None, help="draws per step (default: the workload's)")
    ap.add_argument("--record", default=None, metavar="PATH", help="write every leg's figures to this file (JSON)")
    ap.add_argument("--only-step", action="store_true",
                    help="time only the device step (no end-to-end or log-likelihood leg); for profiling")
    ap.add_argument("--only-loglike", default=None, metavar="LO,HI",
                    help="run only the log-likelihood leg with U{LO..HI} samples per event; for profiling")
    ap.add_argument("--only-chain", default=None, metavar="E,LO,HI",
                    help="time the importance-sampling chains alone (prior and an untrained flow) on E "
                         "events of U{LO..HI} draws")
    ap.add_argument("--only-tmarg", default=None, metavar="E,LO,HI[,U,NTC]",
                    help="run only the merger-time-marginalised likelihood on E events of U{LO..HI} samples "
                         "(optionally oversampling U and a window of NTC samples)")
    ap.add_argument("--only-gemm", default=None, metavar="M,N,K",
                    help="run only the bfloat16 product leg at this shape; for profiling")
    ap.add_argument("--only-flow-sample", default=None, metavar="E,S",
                    help="run only posterior sampling of the (untrained) default flow, E events x S draws, five "
                         "times; for profiling")
    ap.add_argument("--only-flow", default=None, metavar="STEPS",
                    help="run only the coupling-flow leg with this many training steps; for profiling")
    ap.add_argument("--only-conv", default=None, metavar="REPS",
                    help="run only the ResNet stage-1 convolution leg (implicit GEMM vs im2col rows); for profiling")
    ap.add_argument("--only-resnet", default=None, metavar="STEPS",
                    help="run only the ResNet-1D flow leg with this many training steps; for profiling")
    args = ap.parse_args(argv)
    if args.warmup < 3:
        ap.error("--warmup must be at least 3")
    wl = workloads.workload(args.workload)
    if args.batch is not None:
        wl["B"] = args.batch
    if args.impl == "reference":
        return run_reference(args, wl)
    if args.only_gemm:
        import torch
        import paper_2407_19048_gb300 as gwx
        gwx.init()
        shape = tuple(int(v) for v in args.only_gemm.split(","))
        print(json.dumps({"gemm_bf16": gemm_leg(gwx, torch, shape)}), flush=True)
        return 0
    if args.only_flow_sample:
        import torch
        import paper_2407_19048_gb300 as gwx
        import paper_2407_19048_gb300.simulator  # noqa: F401
        from paper_2407_19048_gb300.flow import FlowPosterior
        gwx.init()
        E, S = (int(v) for v in args.only_flow_sample.split(","))
        wl2 = workloads.workload("small_nonspinning", B=E)
        y, th, _ = gwx.simulator.Simulator(wl2).step(0)
        fp = FlowPosterior(wl2)
        offs = torch.arange(E + 1, dtype=torch.int64, device="cuda") * S
        ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        fp.sample(y, offs, 1, 0, S=E * S)
        ev0.record()
        for rep in range(5):
            fp.sample(y, offs, 1, rep, S=E * S)
        ev1.record()
        torch.cuda.synchronize()
        print(json.dumps({"flow_sample": {"events": E, "draws": E * S, "ms": ev0.elapsed_time(ev1) / 5}}), flush=True)
        return 0
    if args.only_chain:
        import torch
        import paper_2407_19048_gb300 as gwx
        import paper_2407_19048_gb300.simulator  # noqa: F401
        from paper_2407_19048_gb300.flow import FlowPosterior
        gwx.init()
        E, lo, hi = (int(v) for v in args.only_chain.split(","))
        # the importance-sampling events and the benchmark flow's shape, untrained: the same kernels and
        # amounts of work as the trained flow's chain (its ESS figures mean nothing)
        wl_ev = dict(workloads.workload("small_nonspinning", B=E), param_seed=777)
        sim_ev = gwx.simulator.Simulator(wl_ev)
        y_ev, _, _ = sim_ev.step(step_counter(0, 0))
        fp = FlowPosterior(workloads.workload("small_nonspinning", B=4096), layers=16, hidden=256, context=64,
                           embed_hidden=512, group=4, seed=0)
        isamp = is_compare(gwx, torch, fp, wl_ev, y_ev.clone(), sim_ev.psd, workloads.ragged_counts(4, E, lo, hi),
                           workloads.tc_grid(wl_ev))
        print(json.dumps({"chain_ms": {a: isamp[a]["chain_ms"] for a in ("prior", "flow")},
                          "samples": isamp["samples"], "events": E, "flow": "untrained"}), flush=True)
        return 0
    if args.only_flow:
        import torch
        import paper_2407_19048_gb300 as gwx
        import paper_2407_19048_gb300.simulator  # noqa: F401
        gwx.init()
        print(json.dumps({"flow": flow_leg(gwx, torch, 0, steps=int(args.only_flow))}), flush=True)
        return 0
    if args.only_conv:
        import torch
        import paper_2407_19048_gb300 as gwx
        gwx.init()
        print(json.dumps({"conv1d_stage1": conv_leg(gwx, torch, reps=int(args.only_conv))}), flush=True)
        return 0
    if args.only_resnet:
        import torch
        import paper_2407_19048_gb300 as gwx
        import paper_2407_19048_gb300.simulator  # noqa: F401
        gwx.init()
        print(json.dumps({"flow_resnet": flow_resnet_leg(gwx, torch, 0, steps=int(args.only_resnet), pretrain_steps=0)}),
              flush=True)
        return 0
    if args.only_tmarg:
        import torch
        import paper_2407_19048_gb300 as gwx
        f = [int(v) for v in args.only_tmarg.split(",")]
        gwx.init()
        print(json.dumps({"log_likelihood_tmarg": tmarg_leg(gwx, torch, f[0], f[1], f[2],
                                                            oversample=f[3] if len(f) > 3 else None,
                                                            n_tc=f[4] if len(f) > 4 else None)}), flush=True)
        return 0
    if args.only_loglike:
        import torch
        import paper_2407_19048_gb300 as gwx
        import paper_2407_19048_gb300.simulator  # noqa: F401
        lo, hi = (int(v) for v in args.only_loglike.split(","))
        gwx.init()
        print(json.dumps({"log_likelihood": loglike_leg(gwx, torch, wl, 0, lo, hi)}), flush=True)
        return 0
    return run_gpu(args, wl)


if __name__ == "__main__":
    sys.exit(main())
