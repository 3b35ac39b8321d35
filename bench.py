"""Benchmark: GaussianImage image fitting on GB300.

Workload (one GPU): a 768x512 synthetic RGB image (Kodak-shaped) fitted by
70,000 2D Gaussians (560K parameters), FP32, tile 16; one step = formation,
binning, render + L2 loss, backward and Adam, replayed from a CUDA graph.
Metric: fit iterations per second (whole job; N GPUs fit N independent
images, weak scaling, no collective). Also reported: render FPS
(formation + binning + render), Gaussian-pixel evaluations per second, the
roofline of the dominant kernel, a batched-vs-plain comparison on uneven
image batches, and the FP64 CPU oracle timed on this host (cpu_baseline).

Timing: W untimed warm-up steps, then K steps, each bracketed by CUDA events
on the launching stream with an L2 flush (a 256 MB write) before it, outside
the timed window; barrier + synchronize before and after; max over ranks.

``--impl reference`` times the FP64 CPU oracle (the reference arm of this
build) on the same workload and prints its own JSON line.
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import synth  # noqa: E402

METRIC = "fit iter/s + render FPS (768×512, 70k Gaussians); batched vs plain at equal PSNR"
WORKLOAD = "c1_768x512_70k"
LR = (1e-3, 1e-2, 1e-2)
# sigma = 1/2 |L^-1 d|^2: dx (FADD), z1 = m11 dx (FMUL), z2 = m21 dx + m22 dy (FFMA),
# z1^2 (FMUL), z1^2 + z2^2 (FFMA) = 7 flop; exp on the SFU.
FWD_FLOP_PER_EVAL = 13   # sigma 7 + 3 FFMA (accumulate)
BWD_FLOP_PER_EVAL = 24   # sigma 7 + 3 FFMA (dL/dc') + FMUL + 2 FFMA (<G, c'>) + FMUL (e) + FADD + FMUL + FADD + FFMA (moments)
# DRAM bytes (read + write) per launch of the ALU-bound kernels at this
# workload, from one ncu --set full capture of each
# (profiles/k_backward_c1_768x512_70k.md, profiles/k_render_c1_768x512_70k.md).
NCU_TRAFFIC_BYTES = {"k_backward": 20.628e6, "k_render": 16.187e6}
# SFU_LANES: ex2 results per clock per SM as measured by gi_alu_peaks on GB300
# (9.99e12 ex2/s at 2064 MHz over 152 SMs = 32).
SMS, FP32_LANES, SFU_LANES, SM_MAX_MHZ = 152, 128, 32, 2070.0
FP32_PEAK_TFLOPS = SMS * FP32_LANES * 2 * SM_MAX_MHZ * 1e6 / 1e12   # 80.5 (FMA = 2 flops)


def max_over_ranks(torch, x, device):
    """Maximum of x over the ranks of the default process group (x itself
    without one): the job's time is its slowest replica's."""
    if not (torch.distributed.is_available() and torch.distributed.is_initialized()):
        return float(x)
    t = torch.tensor([float(x)], device=device, dtype=torch.float64)
    torch.distributed.all_reduce(t, op=torch.distributed.ReduceOp.MAX)
    return float(t.item())


def job_value(world, units_per_rank, t_max):
    """Whole-job throughput: every rank's units over the slowest rank's time."""
    return world * units_per_rank / t_max


def env_rank():
    return int(os.environ.get("RANK", "0")), int(os.environ.get("WORLD_SIZE", "1")), int(
        os.environ.get("LOCAL_RANK", "0"))


def pack(w):
    return np.concatenate([w.means, w.chol, w.color], axis=1).astype(np.float32)


def binning_launches(n, W, H, T):
    """Kernels the fit step's binning launches. The count-matrix path (at most
    2048 tiles and 128-Gaussian rows x tiles <= 2^20; the projection writes the
    counts): column scan and placement, the placement alone for at most 8,192
    counts (chunks of 128 Gaussians up to 8,192 of them, else 256). Otherwise
    emit + one onesweep per LSD pass (digits of at most 9 bits) + ranges."""
    tiles = ((W + T - 1) // T) * ((H + T - 1) // T)
    if tiles <= 2048 and max(1, (n + 127) // 128) * tiles <= (1 << 20):
        chunk = 128 if n <= 8192 else 256
        return 1 if max(1, (n + chunk - 1) // chunk) * tiles <= 8192 else 2
    bits = max(1, math.ceil(math.log2(max(tiles, 2))))
    return 2 + (bits + 8) // 9


def evals_per_render(ranges, W, H, T):
    """Gaussian-pixel evaluations: sum over tiles of list length x in-image pixels."""
    tw, th = (W + T - 1) // T, (H + T - 1) // T
    ln = (ranges[:, 1] - ranges[:, 0]).astype(np.int64).reshape(th, tw)
    pw = np.minimum(T, W - np.arange(tw) * T)
    ph = np.minimum(T, H - np.arange(th) * T)
    return int((ln * ph[:, None] * pw[None, :]).sum()), int((ln * T * T).sum())


class Clocks:
    """nvidia-smi sampler running during the timed region."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int, path: str | None):
        self.index, self.path, self.p = index, path, None

    def __enter__(self):
        try:
            self.p = subprocess.Popen(["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.Q}",
                                       "--format=csv,noheader,nounits", "-lms", "200"],
                                      stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except Exception:
            self.p = None
        return self

    def __exit__(self, *a):
        self.rows = []
        if self.p is None:
            return
        time.sleep(0.3)
        self.p.terminate()
        try:
            out, _ = self.p.communicate(timeout=5)
        except Exception:
            self.p.kill()
            out = ""
        for line in out.splitlines():
            parts = [x.strip() for x in line.split(",")]
            if len(parts) >= 9:
                self.rows.append(parts)
        if self.path:
            with open(self.path, "w") as f:
                f.write(self.Q + "\n" + out)

    def summary(self):
        if not getattr(self, "rows", None):
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        mhz = [float(r[1]) for r in self.rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in self.rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in self.rows for i in range(4) if "Active" in r[5 + i]
                          and "Not" not in r[5 + i]})
        return {"sm_mhz": statistics.median(mhz) if mhz else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(self.rows)}


def cpu_baseline(w, T, budget_s=20.0):
    """The FP64 oracle as it stands: full fit steps on this workload."""
    import oracle
    p = pack(w).astype(np.float64)
    m = np.zeros_like(p)
    v = np.zeros_like(p)
    lr = np.tile(np.array([LR[0]] * 2 + [LR[1]] * 3 + [LR[2]] * 3), (p.shape[0], 1))
    steps, t0 = 0, time.perf_counter()
    while True:
        r = oracle.forward_backward(p[:, 0:2].astype(np.float32), p[:, 2:5].astype(np.float32),
                                    p[:, 5:8].astype(np.float32), w.target, T)
        g = np.concatenate([r["grads"]["means"], r["grads"]["chol"], r["grads"]["color"]], axis=1)
        p, m, v = oracle.adam(p, g, m, v, steps + 1, lr)
        steps += 1
        el = time.perf_counter() - t0
        if el > budget_s or steps >= 50:
            break
    return {"value": steps / el, "unit": "iter/s", "cores": oracle.num_threads(), "kind": "oracle",
            "sample": f"{steps} full fit steps of {WORKLOAD} (FP64 C oracle, OpenMP) in {el:.1f} s"}


def run_reference(args):
    rank, world, _ = env_rank()
    if rank != 0:
        return 0
    import oracle
    w = synth.workload(WORKLOAD)
    T = args.tile
    p = pack(w).astype(np.float64)
    m = np.zeros_like(p)
    v = np.zeros_like(p)
    lr = np.tile(np.array([LR[0]] * 2 + [LR[1]] * 3 + [LR[2]] * 3), (p.shape[0], 1))
    times = []
    for s in range(args.warmup + args.steps):
        t0 = time.perf_counter()
        r = oracle.forward_backward(p[:, 0:2].astype(np.float32), p[:, 2:5].astype(np.float32),
                                    p[:, 5:8].astype(np.float32), w.target, T)
        g = np.concatenate([r["grads"]["means"], r["grads"]["chol"], r["grads"]["color"]], axis=1)
        p, m, v = oracle.adam(p, g, m, v, s + 1, lr)
        if s >= args.warmup:
            times.append(time.perf_counter() - t0)
    tot = sum(times)
    val = args.steps / tot
    line = {"impl": "reference", "metric": METRIC, "value": val, "unit": "iter/s", "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * tot / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": {"workload": f"{WORKLOAD} (768x512 RGB, 70,000 Gaussians, tile {T})"},
            "cpu_baseline": {"value": val, "unit": "iter/s", "cores": oracle.num_threads(), "kind": "oracle",
                             "sample": f"{args.steps} full fit steps of {WORKLOAD} per timed run"},
            "e2e": {"value": val, "unit": "iter/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


def _time(torch, stream, fn, reps, flush=None):
    """Average device ms of fn() over reps calls (CUDA events on `stream`,
    optional L2 flush before each call, outside the timed window)."""
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(reps)]
    for a, b in ev:
        if flush is not None:
            flush.zero_()
        a.record(stream)
        fn()
        b.record(stream)
    torch.cuda.synchronize()
    return sum(a.elapsed_time(b) for a, b in ev) / reps


def batched_vs_plain(gi, torch, n_images, steps, stream):
    """Images of uneven sizes fitted in one launch per stage (tile edge and
    render split chosen by the autotuner) vs the same images one at a time
    with the same configuration (identical arithmetic, so equal PSNR)."""
    ws = synth.batch_workload(n_images)
    tg = [torch.from_numpy(w.target).cuda() for w in ws]
    pr = [torch.from_numpy(pack(w)).cuda() for w in ws]
    tune = gi.autotune(tg, pr, steps=5, warmup=2, lr=LR)
    T, sp = tune["tile"], tune["render_split"]
    fit = gi.Fit(tg, pr, tile=T, lr=LR, render_split=sp)
    fit.step(2)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    fit.step(steps)
    e1.record(stream)
    e1.synchronize()
    t_b = e0.elapsed_time(e1) / 1e3
    mse_b = fit.mse()
    fit.close()
    plain = [gi.Fit([t], [p], tile=T, lr=LR, render_split=sp) for t, p in zip(tg, pr)]
    for f in plain:
        f.step(2)
    torch.cuda.synchronize()
    e0.record(stream)
    for f in plain:
        f.step(steps)
    e1.record(stream)
    e1.synchronize()
    t_p = e0.elapsed_time(e1) / 1e3
    mse_p = [f.mse()[0] for f in plain]
    for f in plain:
        f.close()
    # the same batched fit with the render fed from the device tile queue
    # (descending list length, persistent blocks): identical results
    fq = gi.Fit(tg, pr, tile=T, lr=LR, render_split=sp, tile_queue=True)
    fq.step(2)
    torch.cuda.synchronize()
    e0.record(stream)
    fq.step(steps)
    e1.record(stream)
    e1.synchronize()
    t_q = e0.elapsed_time(e1) / 1e3
    same_q = fq.mse() == mse_b
    fq.close()
    psnr = lambda e: 10 * math.log10(1.0 / e) if e > 0 else float("inf")  # noqa: E731
    d = [abs(psnr(a) - psnr(b)) for a, b in zip(mse_b, mse_p)]
    dpsnr = max(d)
    return {"images": n_images, "steps": steps, "sizes": "uniform over 256x256, 512x384, 768x512, 1024x768",
            "gaussians": int(sum(w.n for w in ws)), "tile": T, "render_split": sp,
            "autotune_ms_per_step": {f"{k[0]}/{k[1]}": v for k, v in tune["ms_per_step"].items()},
            "render_schedule": "tile order (one block per tile)",
            "batched_image_steps_per_s": n_images * steps / t_b, "plain_image_steps_per_s": n_images * steps / t_p,
            "tile_queue_image_steps_per_s": n_images * steps / t_q, "tile_queue_same_loss": same_q,
            "batched_images_fitted_per_s": n_images / t_b, "plain_images_fitted_per_s": n_images / t_p,
            "speedup": t_p / t_b, "max_abs_dpsnr_db": dpsnr, "mean_abs_dpsnr_db": sum(d) / len(d),
            "mean_psnr_db_batched": sum(psnr(a) for a in mse_b) / len(mse_b),
            "mean_psnr_db_plain": sum(psnr(b) for b in mse_p) / len(mse_p)}


def long_fit(gi, torch, stream, T, steps, log_path=None, every=5000, paper=False, cov="cholesky", keep=False):
    """The full-length fit of the 768x512, 70k-Gaussian workload: `steps`
    graph-replayed steps (no L2 flush: steady state) in chunks of `every`,
    each timed with CUDA events; PSNR of the first step's render and after
    every chunk (also written as JSON lines to log_path). The pair capacity
    leaves room for the Gaussians to grow. With cov="rs" the covariance is
    fitted in the rotation-scaling form (Sec. 3.1, Eq. 2-3), starting from
    angles uniform in [-pi, pi) and scales log-uniform in [1, 8]."""
    w = synth.workload(WORKLOAD)
    if paper:
        # App. C.1 / Sec. 4.1: raw parameters (theta = atanh(2 mu / (W, H) - 1),
        # Cholesky diagonal or scales without their +0.5), Adan, lr 1e-3
        # halved every 20000.
        p = pack(w).astype(np.float64)
        p[:, 0:2] = np.arctanh(np.clip(p[:, 0:2] / [w.W, w.H] * 2 - 1, -0.999, 0.999))
        if cov == "rs":
            p[:, 2:5] = synth.init_gaussians_rs(w.n, w.W, w.H, 0)[1]
            p[:, 3:5] -= 0.5
        else:
            p[:, 2] -= 0.5
            p[:, 4] -= 0.5
        fit = gi.Fit([torch.from_numpy(w.target).cuda()], [torch.from_numpy(p.astype(np.float32)).cuda()], tile=T,
                     lr=(1e-3, 1e-3, 1e-3), capacity_factor=4.0, param_mode="paper", optimizer="adan",
                     lr_halve_every=20000, cov=cov)
    else:
        fit = gi.Fit([torch.from_numpy(w.target).cuda()], [torch.from_numpy(pack(w)).cuda()], tile=T, lr=LR,
                     capacity_factor=4.0)
    fit.step(1)
    torch.cuda.synchronize()
    psnr = lambda e: 10 * math.log10(1.0 / e) if e > 0 else float("inf")  # noqa: E731
    p1 = psnr(fit.mse()[0])
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    done, t, traj = 1, 0.0, [[1, p1]]
    log = open(log_path, "w") if log_path else None
    while done < steps:
        n = min(every - (done % every), steps - done)
        e0.record(stream)
        fit.step(n)
        e1.record(stream)
        e1.synchronize()
        t += e0.elapsed_time(e1) / 1e3
        done += n
        traj.append([done, psnr(fit.mse()[0])])
        if log:
            log.write(json.dumps({"step": done, "psnr_db": traj[-1][1], "pairs": int(fit.k.item()),
                                  "seconds": t}) + "\n")
    if log:
        log.close()
    err = gi.device_errors(clear=True)
    out = {"steps": steps, "iter_s": (steps - 1) / t, "seconds": t, "psnr_db_step1": p1,
           "psnr_db_final": traj[-1][1], "psnr_db_trajectory": traj, "pairs_final": int(fit.k.item()),
           "l2": "not flushed between steps (steady state)", "device_errors": int(err)}
    kept = fit.params.clone() if keep else None
    fit.close()
    return (out, kept) if keep else out


def codec_finetune(gi, torch, stream, T, params, steps=10000, every=2500, bits=6, stages=2, size=8):
    """Attribute quantisation-aware fine-tuning (Sec. 3.3-3.4) of the
    Gaussians a 50k-step fit with the paper's recipe ended at: b = 6 bits for
    the Cholesky vector, 2-stage RVQ with 8-entry codebooks for the colour,
    FP16 positions (K-means and quantiser ranges set on the host), Adan at
    that fit's final learning rate (2.5e-4, after two halvings). Reports the
    PSNR of the unquantised fit, of the quantised render before fine-tuning
    (step 1's forward), after `steps` steps, the step rate and the size of
    the encoded stream."""
    w = synth.workload(WORKLOAD)
    psnr = lambda e: 10 * math.log10(1.0 / e) if e > 0 else float("inf")  # noqa: E731
    lr = 2.5e-4
    plain = gi.Fit([torch.from_numpy(w.target).cuda()], [params], tile=T, lr=(lr, lr, lr), capacity_factor=4.0,
                   param_mode="paper", optimizer="adan", use_graph=False)
    plain.render()
    torch.cuda.synchronize()
    img = plain.images()[0]
    ref = torch.from_numpy(w.target).cuda()
    p_plain = psnr(float(((img.clamp(0, 1) - ref) ** 2).mean()))
    plain.close()
    spec = gi.codec_init(params, bits=bits, stages=stages, size=size, param_mode="paper")
    fit = gi.Fit([ref], [params], tile=T, lr=(lr, lr, lr), capacity_factor=4.0, param_mode="paper",
                 optimizer="adan", codec=spec)
    fit.step(1)
    torch.cuda.synchronize()
    p1 = psnr(fit.mse()[0])
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    done, t, traj = 1, 0.0, [[1, p1]]
    while done < steps:
        n = min(every, steps - done)
        e0.record(stream)
        fit.step(n)
        e1.record(stream)
        e1.synchronize()
        t += e0.elapsed_time(e1) / 1e3
        done += n
        traj.append([done, psnr(fit.mse()[0])])
    stream_ = fit.encode()  # renders the current parameters once
    img = fit.images()[0]
    p_final = psnr(float(((img.clamp(0, 1) - ref) ** 2).mean()))
    # decode + render of the encoded stream (the codec's decoder), L2 flushed
    m_, l_, c_ = gi.codec_decode(stream_)
    rdr = gi.Renderer(w.W, w.H, w.n, T, capacity=fit.capacity)
    rdr(m_, l_, c_)
    flush_ = torch.empty(64 * 1024 * 1024, dtype=torch.float32, device="cuda")

    def decode_render():
        mm, ll, cc = gi.codec_decode(stream_)
        rdr(mm, ll, cc)

    dr_ms = _time(torch, stream, decode_render, 50, flush_)
    del flush_
    err = gi.device_errors(clear=True)
    n = w.n
    bits_total = stream_["bits"]
    out = {"steps": steps, "iter_s": (steps - 1) / t, "psnr_db_unquantised": p_plain,
           "psnr_db_quantised_before": p1, "psnr_db_trajectory": traj, "psnr_db_final_render": p_final,
           "commitment_loss": float(fit.codec_out[0].item()), "bits": bits_total,
           "decode_render_fps": 1e3 / dr_ms, "decode_render_ms": dr_ms,
           "bpp": bits_total / (w.W * w.H), "config": {"bits": bits, "stages": stages, "size": size, "lr": lr,
                                                       "ema_decay": fit.codec["ema_decay"]},
           "psnr_note": "training-loss PSNR of the step's render (unclamped) in the trajectory; the "
                        "unquantised and final figures are PSNR of the clamped render",
           "device_errors": int(err)}
    fit.close()
    return out


def oracle_c0_times(reps=3):
    """The FP64 oracle on the 256x256, 2k-Gaussian workload (tile 16): median
    ms of a forward (support rule, binning, render, loss), a forward +
    backward, and a full fit step (forward + backward + Adam)."""
    import oracle
    w = synth.workload("c0_256x256_2k")
    T = 16
    p = pack(w).astype(np.float64)
    lr = np.tile(np.array([LR[0]] * 2 + [LR[1]] * 3 + [LR[2]] * 3), (p.shape[0], 1))

    def fwd():
        rect, cnt = oracle.rect_rule(w.means, w.chol, w.color, w.W, w.H, T)
        ids, rg, _ = oracle.bin_tiles(rect, cnt, w.W, w.H, T)
        oracle.loss(oracle.render(w.means, w.chol, w.color, ids, rg, w.W, w.H, T), w.target)

    def fb():
        return oracle.forward_backward(w.means, w.chol, w.color, w.target, T)

    def step():
        r = fb()
        g = np.concatenate([r["grads"]["means"], r["grads"]["chol"], r["grads"]["color"]], axis=1)
        oracle.adam(p, g, np.zeros_like(p), np.zeros_like(p), 1, lr)

    res = {}
    for name, fn in (("forward", fwd), ("forward_backward", fb), ("step", step)):
        ts = []
        for _ in range(reps):
            t0 = time.perf_counter()
            fn()
            ts.append(time.perf_counter() - t0)
        res[name] = 1e3 * statistics.median(ts)
    return {"workload": "c0_256x256_2k (256x256, 2,000 Gaussians, tile 16)", "ms": res,
            "cores": oracle.num_threads()}


def large_image(gi, torch, stream, flush, T=16, reps=20):
    """2040x1356 synthetic image, 30% of the means in 10% of the area:
    forward-only render FPS and fit-step (forward + backward) throughput."""
    out = {}
    for name in ("c2_2040x1356_100k", "c2_2040x1356_200k"):
        w = synth.workload(name)
        tq = {}
        for queue in (True, False):  # the tile-queue schedule first, then the default (kept below)
            fit = gi.Fit([torch.from_numpy(w.target).cuda()], [torch.from_numpy(pack(w)).cuda()], tile=T, lr=LR,
                         tile_queue=queue)
            fit.step(3)
            render_ms = _time(torch, stream, fit.render, reps, flush)
            step_ms = _time(torch, stream, lambda: fit.step(1), reps, flush)
            if queue:
                tq = {"render_ms": render_ms, "fit_step_ms": step_ms}
                fit.close()
        p = fit.params
        _, rect, cnt = gi.project(p[:, 0:2].contiguous(), p[:, 2:5].contiguous(), p[:, 5:8].contiguous(), w.W, w.H, T)
        bins = gi.bin_tiles(rect, cnt, None, w.W, w.H, T)
        ev_in, ev_all = evals_per_render(bins.ranges.cpu().numpy(), w.W, w.H, T)
        out[name] = {"render_fps": 1e3 / render_ms, "render_ms": render_ms, "fit_step_ms": step_ms,
                     "fit_iter_s": 1e3 / step_ms, "pairs": bins.K, "evals_per_render": ev_in,
                     "fwd_bwd_evals_per_s": ev_all / (step_ms * 1e-3), "tile_queue": tq}
        fit.close()
    return out


def ablation(gi, torch, stream, flush, T=16, reps=100, fit_steps=10000, n_gauss=None):
    """Table 3's representation ablation on the 768x512 image: the paper's
    merged colour (8 parameters, accumulated summation), separate opacity
    with accumulated summation ("w/o M", 9 parameters) and sorted
    alpha-blending ("w/o AR + w/o M"), with the workload's 70,000 Gaussians
    or its first n_gauss (Table 3 uses 30,000). The 9-parameter forms start
    from c = 2 c', o = sigmoid(0) = 1/2 (the same initial accumulated image).
    Per form: fit-step and render time (L2 flushed before each), and the PSNR
    after `fit_steps` Adam steps."""
    w = synth.workload(WORKLOAD)
    n = w.n if n_gauss is None else n_gauss
    tgt = torch.from_numpy(w.target).cuda()
    psnr = lambda e: 10 * math.log10(1.0 / e) if e > 0 else float("inf")  # noqa: E731
    out = {"gaussians": n}
    for form in ("merged", "separate", "blend"):
        p = pack(w)[:n]
        kw = {}
        if form != "merged":
            p = p.copy()
            p[:, 5:8] *= 2.0
            kw = {"opacity": form, "opacity_logits": [torch.zeros(n, device="cuda")]}
        fit = gi.Fit([tgt], [torch.from_numpy(p).cuda()], tile=T, lr=LR, capacity_factor=4.0, **kw)
        fit.step(3)
        step_ms = _time(torch, stream, lambda: fit.step(1), reps, flush)
        render_ms = _time(torch, stream, fit.render, reps, flush)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        fit.step(fit_steps - 3 - reps)
        e1.record(stream)
        e1.synchronize()
        long_s = e0.elapsed_time(e1) / 1e3
        fit.render()
        torch.cuda.synchronize()
        img = fit.images()[0]
        out[form] = {"fit_iter_s": 1e3 / step_ms, "fit_step_ms": step_ms, "render_fps": 1e3 / render_ms,
                     "render_ms": render_ms, "steady_iter_s": (fit_steps - 3 - reps) / long_s,
                     "psnr_db": psnr(float(((img.clamp(0, 1) - tgt) ** 2).mean())), "steps": fit_steps,
                     "params_per_gaussian": 8 if form == "merged" else 9,
                     "device_errors": int(gi.device_errors(clear=True))}
        fit.close()
    base = out["merged"]
    for form in ("separate", "blend"):
        out[form]["step_time_vs_merged"] = out[form]["fit_step_ms"] / base["fit_step_ms"]
        out[form]["render_time_vs_merged"] = out[form]["render_ms"] / base["render_ms"]
    out["paper_context"] = {"fps": {"w/o AR + w/o M": 2340, "w/o M": 2555, "merged": 2565},
                            "train_s": {"w/o AR + w/o M": 104.76, "w/o M": 98.54, "merged": 91.06},
                            "hw": "V100, Kodak, 30k Gaussians, 50k steps (Table 3)"}
    return out


def codec_decode(gi, torch, stream, flush, T=16, reps=50):
    """RVQ decode (FP16 means, 2-stage 256-entry codebooks) then render, at
    768x512 with 50,000 Gaussians; and decode alone over a batch of 64 such
    Gaussian sets (3.2M Gaussians) in one call."""
    w = synth.workload("c4_768x512_50k")
    n = w.n
    cb = torch.from_numpy(synth.codebooks(4000)).cuda()
    idx = torch.from_numpy(synth.vq_indices(n, 4000)).cuda()
    m16 = torch.from_numpy(w.means.astype(np.float16)).cuda()
    means, chol, color = gi.vq_decode(m16, idx, cb)
    _, rect, cnt = gi.project(means, chol, color, w.W, w.H, T)
    K = gi.bin_tiles(rect, cnt, None, w.W, w.H, T).K
    r = gi.Renderer(w.W, w.H, n, T, capacity=int(K * 1.5) + 4096)

    out1 = (torch.empty((n, 2), dtype=torch.float32, device="cuda"),
            torch.empty((n, 3), dtype=torch.float32, device="cuda"),
            torch.empty((n, 3), dtype=torch.float32, device="cuda"))

    def decode_render():
        mm, ll, cc = gi.vq_decode(m16, idx, cb, out=out1)
        r(mm, ll, cc)

    dr_ms = _time(torch, stream, decode_render, reps, flush)
    nb = 64 * n
    idx_b = torch.from_numpy(synth.vq_indices(nb, 4001)).cuda()
    m16_b = torch.from_numpy(np.tile(w.means, (64, 1)).astype(np.float16)).cuda()
    out_b = (torch.empty((nb, 2), dtype=torch.float32, device="cuda"),
             torch.empty((nb, 3), dtype=torch.float32, device="cuda"),
             torch.empty((nb, 3), dtype=torch.float32, device="cuda"))
    dec_ms = _time(torch, stream, lambda: gi.vq_decode(m16_b, idx_b, cb, out=out_b), reps, flush)
    bytes_dec = nb * (4 + 4 + 32)
    assert gi.device_errors(clear=True) == 0
    return {"workload": "768x512, 50,000 Gaussians, FP16 means, 2x256-entry RVQ codebooks", "decode_render_fps":
            1e3 / dr_ms, "decode_render_ms": dr_ms, "batch64_decode": {"gaussians": nb, "ms": dec_ms,
            "gaussians_per_s": nb / (dec_ms * 1e-3), "gb_per_s": bytes_dec / (dec_ms * 1e-3) / 1e9}}


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=10)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--tile", type=int, default=16)
    ap.add_argument("--no-batched", action="store_true")
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--no-extra", action="store_true", help="skip the large-image and codec measurements")
    ap.add_argument("--batch-images", type=int, default=64)
    ap.add_argument("--batch-steps", type=int, default=2000, help="fit steps of the batched vs plain comparison")
    ap.add_argument("--long-steps", type=int, default=50000, help="steps of the full-length fit (0 = skip)")
    ap.add_argument("--out", default=os.path.join(ROOT, "bench_out"), help="folder for the long fits' PSNR logs")
    args = ap.parse_args()
    args.warmup = max(3, args.warmup)
    if args.impl == "reference":
        return run_reference(args)

    import torch
    rank, world, local = env_rank()
    torch.cuda.set_device(local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    import paper_2403_08551_gb300 as gi
    gi.load()
    T = args.tile
    stream = torch.cuda.current_stream()

    w = synth.workload(WORKLOAD, index=rank)
    target = torch.from_numpy(w.target).cuda()
    params = torch.from_numpy(pack(w)).cuda()
    fit = gi.Fit([target], [params], tile=T, lr=LR)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")

    for _ in range(args.warmup):
        fit.step(1)
    torch.cuda.synchronize()

    def barrier():
        if world > 1:
            torch.distributed.barrier()
        torch.cuda.synchronize()

    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    os.makedirs(args.out, exist_ok=True)
    with Clocks(local, os.path.join(args.out, f"clocks_rank{rank}.csv") if rank == 0 else None) as clk:
        barrier()
        for i in range(args.steps):
            flush.zero_()
            ev[i][0].record(stream)
            fit.step(1)
            ev[i][1].record(stream)
        barrier()
    step_ms = sum(a.elapsed_time(b) for a, b in ev)
    t_max = max_over_ranks(torch, step_ms / 1e3, "cuda")
    value = job_value(world, args.steps, t_max)

    # Stage breakdown from a separate, instrumented fit of the same image:
    # CUDA events recorded between the stages of every step (event nodes in
    # the graph stop the launches of neighbouring stages from overlapping, so
    # these steps are slower than the timed ones above).
    fit_i = gi.Fit([target], [fit.params.clone()], tile=T, lr=LR, stage_events=True)
    fit_i.step(args.warmup)
    n_s = max(20, min(args.steps, 200))
    stage = np.zeros(5)
    for i in range(n_s):
        flush.zero_()
        fit_i.step(1)
        stage += np.array(fit_i.stage_times())
    stage_ms = stage / n_s
    fit_i.close()

    # Render FPS: formation + binning + render (no backward), flushed L2.
    n_r = max(20, args.steps // 2)
    evr = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(n_r)]
    for i in range(n_r):
        flush.zero_()
        evr[i][0].record(stream)
        fit.render()
        evr[i][1].record(stream)
    torch.cuda.synchronize()
    render_ms = sum(a.elapsed_time(b) for a, b in evr) / n_r
    # The same forward through the per-stage C-ABI calls, launched eagerly.
    p_r = fit.params.clone()
    m_r, l_r, c_r = p_r[:, 0:2].contiguous(), p_r[:, 2:5].contiguous(), p_r[:, 5:8].contiguous()
    rdr = gi.Renderer(w.W, w.H, w.n, T, capacity=fit.capacity)
    rdr(m_r, l_r, c_r)
    render_eager_ms = _time(torch, stream, lambda: rdr(m_r, l_r, c_r), n_r, flush)

    # Evaluations per render for the current parameters.
    p_now = fit.params.clone()
    rec, rect, cnt = gi.project(p_now[:, 0:2].contiguous(), p_now[:, 2:5].contiguous(), p_now[:, 5:8].contiguous(),
                                w.W, w.H, T)
    bins = gi.bin_tiles(rect, cnt, None, w.W, w.H, T)
    ev_in, ev_all = evals_per_render(bins.ranges.cpu().numpy(), w.W, w.H, T)
    K = bins.K

    # End to end through the public API with host buffers. Per step the
    # step's target image (4.7 MB) crosses the host link from pinned host
    # memory and the loss is read back. Two ways: the fit reads the pinned
    # target itself inside the render (set_target_source: the transfer
    # overlaps the render's accumulation), reported as e2e; or an explicit
    # copy into the context before each step (e2e_copy).
    host_tgt = torch.from_numpy(w.target.reshape(-1)).pin_memory()
    host_loss = torch.empty(fit.loss_sum.shape, dtype=torch.float64).pin_memory()
    n_e = max(20, args.steps // 2)

    def e2e_run(copy):
        eve = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(n_e)]
        for i in range(n_e):
            flush.zero_()
            eve[i][0].record(stream)
            if copy:
                fit.targets.copy_(host_tgt, non_blocking=True)
            fit.step(1)
            host_loss.copy_(fit.loss_sum, non_blocking=True)
            eve[i][1].record(stream)
        torch.cuda.synchronize()
        s_ = sum(a.elapsed_time(b) for a, b in eve) / 1e3
        out_ = {"value": world * n_e / s_ if world == 1 else None, "unit": "iter/s",
                "h2d_bytes_per_step": int(host_tgt.numel() * 4), "d2h_bytes_per_step": int(host_loss.numel() * 8)}
        if world > 1:
            out_["value"] = job_value(world, n_e, max_over_ranks(torch, s_, "cuda"))
        return out_

    e2e_copy = e2e_run(True)
    e2e_copy["mode"] = "cudaMemcpyAsync of the pinned target into the context, then the step"
    fit.set_target_source(host_tgt)
    e2e = e2e_run(False)
    e2e["mode"] = ("zero-copy: each step's render reads the pinned host target over the host link "
                   "(set_target_source), overlapped with its accumulation")
    fit.set_target_source(None)

    # Roofline of the dominant kernel (backward or render), FP32-pipe bound.
    names = ["formation", "binning", "render", "backward", "update"]
    bwd_tflops = BWD_FLOP_PER_EVAL * ev_all / (stage_ms[3] * 1e-3) / 1e12
    fwd_tflops = FWD_FLOP_PER_EVAL * ev_all / (stage_ms[2] * 1e-3) / 1e12
    dom = "backward" if stage_ms[3] >= stage_ms[2] else "render"
    ach = bwd_tflops if dom == "backward" else fwd_tflops
    roof = {"kernel": "k_backward" if dom == "backward" else "k_render", "bound": "alu", "achieved": ach,
            "peak": FP32_PEAK_TFLOPS, "unit": "TFLOP/s", "frac": ach / FP32_PEAK_TFLOPS,
            "traffic": (NCU_TRAFFIC_BYTES.get("k_backward" if dom == "backward" else "k_render")
                        if T == 16 else None), "traffic_unit": "bytes per launch (ncu dram read + write)",
            "traffic_source": "constant from one ncu capture of the current kernel at this workload "
                              "(profiles/k_backward_c1_768x512_70k.md); not measured in this run",
            "peak_source": "derived: 152 SMs x 128 FP32 lanes x 2 flop/FMA x 2070 MHz",
            "sfu_frac": (ev_all / (stage_ms[3 if dom == 'backward' else 2] * 1e-3))
            / (SMS * SFU_LANES * SM_MAX_MHZ * 1e6)}

    out = {"metric": METRIC, "value": value, "unit": "iter/s", "n_gpus": world, "steps": args.steps,
           "warmup": args.warmup, "ms_per_step": 1e3 * t_max / args.steps, "higher_is_better": True,
           "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
           "config": {"workload": f"{WORKLOAD}: 768x512 RGB synthetic image, 70,000 Gaussians, tile {T}, "
                                  f"FP32 Adam (lr 1e-3 means, 1e-2 others)", "global_batch": world,
                      "parallelism": f"replica x{world} (independent images)",
                      "render_schedule": "tile order (one block per tile)",
                      "l2": "flushed (256 MB write) before every timed step"},
           "render_fps": 1e3 / render_ms, "render_ms": render_ms,
           "render_fps_modes": {"graph": 1e3 / render_ms, "eager": 1e3 / render_eager_ms},
           "stage_ms": dict(zip(names, [float(x) for x in stage_ms])),
           "stage_ms_note": "separate instrumented pass (CUDA events between stages, L2 flushed)",
           "pairs": K, "evals_per_render": ev_in, "evals_per_render_padded": ev_all,
           "fwd_evals_per_s": ev_all / (stage_ms[2] * 1e-3), "bwd_evals_per_s": ev_all / (stage_ms[3] * 1e-3),
           "gpu_launches": args.steps * (4 + binning_launches(w.n, w.W, w.H, T)), "roofline": roof, "e2e": e2e,
           "e2e_copy": e2e_copy,
           "paper_context": {"render_fps": 2092.17, "fit_iter_s": 469.1, "hw": "V100 (Table 1a, Kodak)"}}
    out["fit_psnr_db_after"] = 10 * math.log10(1.0 / max(fit.mse()[0], 1e-30))
    if rank == 0:
        out["clocks"] = clk.summary()
    if not args.no_batched and rank == 0:
        out["batched"] = batched_vs_plain(gi, torch, args.batch_images, args.batch_steps, stream)
    if not args.no_extra and rank == 0:
        out["large_image"] = large_image(gi, torch, stream, flush)
        out["codec"] = codec_decode(gi, torch, stream, flush)
        out["ablation"] = ablation(gi, torch, stream, flush)
        out["ablation_30k"] = ablation(gi, torch, stream, flush, n_gauss=30000)
    if args.long_steps > 1 and not args.no_extra and rank == 0:
        out["fit_long"] = long_fit(gi, torch, stream, T, args.long_steps,
                                   os.path.join(args.out, "fit_long_psnr.jsonl"))
        out["fit_long_paper_recipe"], fitted = long_fit(gi, torch, stream, T, args.long_steps,
                                                        os.path.join(args.out, "fit_long_paper_psnr.jsonl"),
                                                        paper=True, keep=True)
        out["codec_finetune"] = codec_finetune(gi, torch, stream, T, fitted)
        # the same fine-tuning with 2 x 256-entry colour codebooks: the 2 x 8
        # codebook (64 colours for 70,000 Gaussians) is the PSNR ceiling above
        out["codec_finetune_b256"] = codec_finetune(gi, torch, stream, T, fitted, size=256)
        out["fit_long_paper_recipe_rs"] = long_fit(gi, torch, stream, T, args.long_steps,
                                                   os.path.join(args.out, "fit_long_paper_rs_psnr.jsonl"),
                                                   paper=True, cov="rs")
    if not args.no_cpu and rank == 0:
        out["cpu_baseline"] = cpu_baseline(w, T)
        out["cpu_baseline"]["oracle_c0"] = oracle_c0_times()
    fit.close()
    if world > 1:
        torch.distributed.barrier()
        torch.distributed.destroy_process_group()
    if rank == 0:
        print(json.dumps(out), flush=True)
    return 0


if __name__ == "__main__":
    sys.exit(main())
