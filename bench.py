#!/usr/bin/env python3
"""Benchmark of the recombination hot path on GB300.

Workload: one periodic (24 kpc)^3 box of 256^3 cells (log-normal density,
sigma_lnrho = 0.8, k^2 spectrum; Gaussian peculiar velocities, sigma_v =
1 km/s), 1e8 Ly-alpha packets per step, the 400-step schedule z = 1800 -> 600.
A step is one pass of the whole hot path: packet allocation, transport
(lya_transport) and the per-cell update (rec_step, tally mode).  The state is
advanced untimed to step 170 (z ~ 1140, mid-recombination), then W warm-up
steps and K timed steps run; inputs (0.7-1.2 GB of fields) exceed the 129 MB
L2, so no flush is needed between steps.

Prints one JSON line: cell-steps/s of the mixed form (value) with packets/s,
the plain FP64 form beside it, the HBM roofline of the dominant kernel
(packet march), the oracle timed on the host cores, an end-to-end number
through the public API with host buffers, clocks and the kernel count.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]
Under torchrun each rank runs its own box (different seed): weak scaling, no
data-path collective; the timing is the max over ranks.
"""
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
sys.path.insert(0, ROOT)

METRIC = "cell-steps/s & Lyα packets/s at 256^3: mixed vs FP64 form, % HBM roofline"
N_SIDE, N_PACKETS, N_STEPS, Z0, Z1 = 256, 100_000_000, 400, 1800.0, 600.0
S0 = 170  # first warm-up step (z ~ 1140)


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=30)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--n", type=int, default=N_SIDE)
    ap.add_argument("--packets", type=int, default=N_PACKETS)
    ap.add_argument("--no-fp64", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--prep", type=int, default=S0, help="untimed steps before the warm-up (profiling: 0)")
    ap.add_argument("--no-batched", action="store_true", help="skip the batched 64-box measurement")
    ap.add_argument("--no-scatter", action="store_true", help="skip the scattering Monte-Carlo measurement")
    ap.add_argument("--no-adjoint", action="store_true", help="skip the adjoint (reverse sweep) measurement")
    ap.add_argument("--no-512", action="store_true", help="skip the 512^3 / 1e9-packet measurement")
    return ap.parse_args()


def workload(n, packets):
    from paper_2312_11448_gb300.inputs import BoxConfig, make_box, z_schedule
    cfg = BoxConfig("box256", n, 0.8, 1.0, packets, N_STEPS, Z0, Z1, None, "mixed")
    return cfg, z_schedule(Z0, Z1, N_STEPS)


def describe(cfg, form):
    return (f"{cfg.n}^3 periodic box (24 kpc), sigma_lnrho={cfg.sigma_lnrho}, sigma_v={cfg.sigma_v} km/s, "
            f"{cfg.n_packets:.0e} Lya packets/step, tally mixing, {form} form, steps {S0}+ of {N_STEPS} "
            f"(z {Z0:.0f}->{Z1:.0f})")


# ---------------------------------------------------------------------------- clocks
class Clocks:
    """nvidia-smi samples every 200 ms in the background."""

    def __init__(self, gpu_index):
        self.path = os.path.join("/tmp", f"rec_bench_clocks_{os.getpid()}.csv")
        q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")
        try:
            self.f = open(self.path, "w")
            self.p = subprocess.Popen(["nvidia-smi", f"--query-gpu={q}", "--format=csv,noheader,nounits", "-lms",
                                       "200", "-i", str(gpu_index)], stdout=self.f, stderr=subprocess.DEVNULL)
        except Exception:
            self.p = None
        self.windows = []

    def mark(self):
        return time.time()

    def window(self, t0, t1):
        self.windows.append((t0, t1))

    def summary(self):
        if self.p is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.p.terminate()
        self.p.wait()
        self.f.close()
        rows = []
        for line in open(self.path):
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                rows.append((float(parts[1]), float(parts[2]), float(parts[3]), parts[5:9]))
            except ValueError:
                continue
        os.unlink(self.path)
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        # samples under load: above half the peak observed power
        pmax = max(r[2] for r in rows)
        load = [r for r in rows if r[2] >= 0.5 * pmax] or rows
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in load for i, v in enumerate(r[3]) if v.lower() == "active"})
        return {"sm_mhz": statistics.median(r[0] for r in load), "sm_max_mhz": max(r[1] for r in rows),
                "reasons": reasons, "samples_under_load": len(load), "power_w_max": pmax}


# ------------------------------------------------------------------------------ GPU arm
_FIELDS = {}


def fields_of(cfg, seed):
    from paper_2312_11448_gb300.inputs import make_box as fields
    if (cfg, seed) not in _FIELDS:
        _FIELDS[(cfg, seed)] = fields(cfg, seed=seed)
    return _FIELDS[(cfg, seed)]


def make_box(cfg, precision, seed):
    import torch
    from paper_2312_11448_gb300 import rec
    delta, U = fields_of(cfg, seed)
    # a non-default stream, so that steps can also be captured as CUDA graphs
    return rec.Box(cfg.n, delta, U, cfg.n_packets, precision=precision, mixing="tally", seed=seed,
                   stream=torch.cuda.Stream()), delta, U


def advance(box, zs, s_from, s_to):
    for s in range(s_from, s_to):
        box.transport(s, zs[s])
        box.step(s, zs[s], zs[s + 1])


def algorithmic_bytes(precision, n3, emitted, queued, crossings, newton_passes):
    """Algorithmic bytes (each datum counted once per use) of the kernel groups.
    emit:  per packet its packet-prefix entry, home temperature and velocity;
           a tally increment if resonant at home, else a queue entry written.
    march: per queued packet its queue entry and tally increment, one velocity
           per cell visited after the home cell (one per face crossing).
    rec_step: per Newton pass delta, x_e (mixed: its binary32 (x, 1-x) cache),
           T, tally; final pass reads delta, x_e (+ cache), T, tally, velocity and
           writes x_e (+ cache), T, velocity, emission, tally."""
    if precision == "mixed":
        v, t, d, e, qe = 16, 4, 4, 4, 32
    else:
        v, t, d, e, qe = 32, 8, 8, 8, 96
    home = emitted - queued
    emit = emitted * (4 + t + v) + home * 4 + queued * qe
    march = queued * (qe + 4) + crossings * v
    if precision == "mixed":
        pass_b = d + 8 + t + 4  # the binary32 (x, 1-x) cache replaces x
        final_b = (d + 8 + 8 + t + 4 + v) + (8 + 8 + t + v + e + 4)
    else:
        pass_b = d + 8 + t + 4
        final_b = (d + 8 + t + 4 + v) + (8 + t + v + e + 4)
    step = n3 * (pass_b * newton_passes + final_b)
    alloc = n3 * (3 * e + 4)
    return dict(emit=emit, march=march, rec_step=step, alloc=alloc)


def method_bytes(precision, n3, emitted, queued, crossings, newton_passes):
    """Algorithmic bytes of the method itself (the per-unit figures of the
    measurement plan), without the library's own intermediate traffic (the
    march queue, the (x, 1-x) cache):
      transport, per packet: 16 B at emission + 4 B tally, and per cell
        crossing one velocity (16 B binary32 / 32 B binary64);
      rec_step, per cell: 20 B (FP64 form 28 B) per Newton evaluation pass
        (delta, x_e, T, tally) + 64 B (100 B) for the final pass (reads delta,
        x_e, T, tally, U; writes x_e, T, U, emission weight, tally zero).
    Split by kernel: emission = 16 B per packet + 4 B per packet absorbed at
    home; march = 4 B per queued packet + one velocity per crossing."""
    v = 16 if precision == "mixed" else 32
    pass_b, final_b = (20, 64) if precision == "mixed" else (28, 100)
    home = emitted - queued
    emit = emitted * 16 + home * 4
    march = queued * 4 + crossings * v
    step = n3 * (pass_b * newton_passes + final_b)
    return dict(emit=emit, march=march, rec_step=step, whole=emit + march + step)


def time_form(cfg, zs, precision, W, K, seed, dist, clocks, prep=S0, graph=False):
    import torch
    from paper_2312_11448_gb300 import tune
    box, delta, U = make_box(cfg, precision, seed)
    # transport tuning from the committed autotuner table, when it has this workload
    tuned = tune.apply_table(box, tune.workload_key(cfg.n, cfg.n_packets, precision))
    box.state_init(zs[0])
    advance(box, zs, 0, prep)
    s_timed = prep + W
    advance(box, zs, prep, s_timed)
    box.ensure_stats(K)
    box.timing(True)
    stream = box.stream
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    t0 = clocks.mark()
    e0.record(stream)
    for k in range(K):
        s = s_timed + k
        box.transport(s, zs[s], slot=k)
        box.step(s, zs[s], zs[s + 1], slot=k)
    e1.record(stream)
    torch.cuda.synchronize()
    clocks.window(t0, clocks.mark())
    ms = e0.elapsed_time(e1)
    kt = box.kernel_times()
    box.timing(False)
    st = box.stats_all()[:K]
    emitted = sum(r["emitted"] for r in st) / K
    queued = sum(r["queued"] for r in st) / K
    crossings = sum(r["crossings"] for r in st) / K
    passes = sum(r["newton_passes"] for r in st) / K
    flags = 0
    for r in st:
        flags |= r["flags"]
    if flags & 4 or not math.isfinite(st[-1]["X_e"]) or emitted < cfg.n_packets:
        raise RuntimeError(f"{precision} form: invalid state (flags={flags}, X_e={st[-1]['X_e']}, emitted={emitted})")
    ab = algorithmic_bytes(precision, box.n3, emitted, queued, crossings, passes)
    mb = method_bytes(precision, box.n3, emitted, queued, crossings, passes)
    out = dict(ms=ms, kt=kt, emitted=emitted, queued=queued, crossings=crossings, passes=passes, flags=flags, ab=ab,
               mb=mb,
               Xe=st[-1]["X_e"], box=box, delta=delta, U=U,
               tuning=dict(box.tuning(), source="autotuner table" if tuned else "defaults"))
    if graph:
        # the next K steps as one CUDA graph launch per step (rec_graph_step)
        s0 = s_timed + K
        box.graph_step(s0, zs[s0], zs[s0 + 1])  # instantiates the executable graph
        s0 += 1
        torch.cuda.synchronize()
        e0.record(stream)
        for k in range(K):
            s = s0 + k
            box.graph_step(s, zs[s], zs[s + 1], slot=k)
        e1.record(stream)
        torch.cuda.synchronize()
        out["graph_ms"] = e0.elapsed_time(e1)
        gst = box.stats_all()[:K]
        if any(r["flags"] & 4 for r in gst) or not math.isfinite(gst[-1]["X_e"]):
            raise RuntimeError("graph steps: invalid state")
    return out


def time_e2e(cfg, zs, res, K):
    """Same step through the public API with host buffers: per step the fields
    (delta, velocity) come from pinned host memory and x_e, T go back.  The
    copies are pipelined as a caller streaming fields would: step k+1's fields
    go up on an upload stream into a device staging buffer while step k
    computes (one device-to-device copy puts them in place at the start of the
    step), and step k's x_e and T come down on a download stream while step
    k+1's transport runs (which does not write them); the step's rec_step
    waits for that download.  Every step's copies are inside the timed region:
    the first upload before the first step, the last download before the end."""
    import torch
    box = res["box"]
    stream = box.stream
    up, down = torch.cuda.Stream(), torch.cuda.Stream()
    h_delta = box.delta.cpu().pin_memory()
    h_vel = box.vel4.cpu().pin_memory()
    h_x = torch.empty_like(box.x, device="cpu").pin_memory()
    h_T = torch.empty_like(box.T, device="cpu").pin_memory()
    st_delta, st_vel = torch.empty_like(box.delta), torch.empty_like(box.vel4)
    s_base = S0 + 3 + K  # continue after the timed window (any in-range steps)
    ev = lambda: torch.cuda.Event()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record(stream)
    up.wait_event(e0)
    with torch.cuda.stream(up):
        st_delta.copy_(h_delta, non_blocking=True)
        st_vel.copy_(h_vel, non_blocking=True)
    uploaded = ev()
    uploaded.record(up)
    downloaded = None
    for k in range(K):
        s = min(s_base + k, N_STEPS - 1)
        stream.wait_event(uploaded)
        with torch.cuda.stream(stream):
            box.delta.copy_(st_delta)
            box.vel4.copy_(st_vel)
        consumed = ev()
        consumed.record(stream)
        if k + 1 < K:  # the next step's fields go up while this step computes
            up.wait_event(consumed)
            with torch.cuda.stream(up):
                st_delta.copy_(h_delta, non_blocking=True)
                st_vel.copy_(h_vel, non_blocking=True)
            uploaded = ev()
            uploaded.record(up)
        box.transport(s, zs[s])
        if downloaded is not None:
            stream.wait_event(downloaded)  # the previous step's x_e, T are down before rec_step rewrites them
        box.step(s, zs[s], zs[s + 1])
        stepped = ev()
        stepped.record(stream)
        down.wait_event(stepped)
        with torch.cuda.stream(down):
            h_x.copy_(box.x, non_blocking=True)
            h_T.copy_(box.T, non_blocking=True)
        downloaded = ev()
        downloaded.record(down)
    stream.wait_event(downloaded)
    e1.record(stream)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1)
    h2d = h_delta.numel() * h_delta.element_size() + h_vel.numel() * h_vel.element_size()
    d2h = h_x.numel() * h_x.element_size() + h_T.numel() * h_T.element_size()
    return ms, h2d, d2h


def time_adjoint(cfg, zs, n_window=20, seed=1):
    """The adjoint workload of the 256^3 configuration: FP64 form, tally mode,
    a window of n_window steps of the 400-step schedule ending at the node
    nearest z* = 1100, objective the visibility function there.  Forward:
    transport + rec_step per step with the tallies stored and ceil(sqrt(N))
    checkpoints; reverse: segment replays (rec_step) and rec_step_adjoint per
    step.  Reports ms per reverse step (replay included), the forward FP64 step
    beside it and the peak device memory, with the memory formula for the full
    400-step run."""
    import torch
    from paper_2312_11448_gb300 import rec
    from paper_2312_11448_gb300.autograd import Trajectory
    k_star = int(np.argmin(np.abs(zs - 1100.0)))
    k0 = k_star - n_window
    zw = zs[k0:k_star + 1]
    delta, U = fields_of(cfg, seed)
    torch.cuda.reset_peak_memory_stats()
    base = torch.cuda.memory_allocated()
    box = rec.Box(cfg.n, delta, U, cfg.n_packets, precision="fp64", mixing="tally", seed=seed,
                  stream=torch.cuda.Stream())
    box.state_init(zw[0])  # Saha state at the window start (the timing does not depend on it)
    with torch.cuda.stream(box.stream):
        x0 = box.x.clone()
        T0 = box.T.clone()
    traj = Trajectory(box, zw, run_transport=True)
    stream = box.stream
    e = [torch.cuda.Event(enable_timing=True) for _ in range(3)]
    torch.cuda.synchronize()
    e[0].record(stream)
    Xe = traj.forward(x0, T0)
    e[1].record(stream)
    J, dJ = rec.objective(zw, Xe, 2, 1100.0)
    g_delta, g_T0, g_x0, g_a = traj.backward(dJ)
    e[2].record(stream)
    torch.cuda.synchronize()
    fwd_ms, rev_ms = e[0].elapsed_time(e[1]), e[1].elapsed_time(e[2])
    nonfinite = {k: int((~torch.isfinite(v)).sum()) for k, v in
                 (("delta", g_delta), ("T0", g_T0), ("x0", g_x0), ("a", g_a))}
    finite = not any(nonfinite.values())
    peak = torch.cuda.max_memory_allocated() - base
    cell_state = 8 + 8 + 32  # x_e, T, double4 velocity per checkpoint or replay state
    n3 = cfg.n ** 3
    full = {"tallies_gb": N_STEPS * n3 * 4 / 1e9,
            "checkpoints_gb": math.ceil(math.sqrt(N_STEPS)) * n3 * cell_state / 1e9,
            "replay_states_gb": math.ceil(math.sqrt(N_STEPS)) * n3 * cell_state / 1e9}
    full["total_gb"] = sum(full.values())
    box.close()
    del traj, g_delta, g_T0, g_x0, g_a
    torch.cuda.empty_cache()
    return {"workload": (f"{cfg.n}^3, FP64 form, tally mode, steps {k0}..{k_star} of {N_STEPS} (z {zw[0]:.0f} -> "
                         f"{zw[-1]:.0f}) from the Saha state at z {zw[0]:.0f}, objective: visibility at "
                         f"z* = {zw[-1]:.0f}, checkpoints every "
                         f"{traj_k(n_window)} steps"),
            "forward_ms_per_step": fwd_ms / n_window, "reverse_ms_per_step": rev_ms / n_window,
            "J": J, "finite_gradients": finite, "nonfinite_counts": nonfinite, "peak_device_gb": peak / 1e9,
            "full_run_memory_estimate": full, "gpu_launch_groups": "transport, rec_step, rec_step_adjoint"}


def time_512(W=2, K=3):
    """The 512^3 configuration (sigma_lnrho 1.2, sigma_v 2 km/s, 1e9 packets per
    step, 600 steps z 1800 -> 500), mixed form, from the Saha state at the node
    nearest z = 1140 (the 256^3 line's redshift; advancing there step by step
    would take minutes), W untimed and K timed steps."""
    import torch
    from paper_2312_11448_gb300.inputs import CONFIGS, z_schedule
    from paper_2312_11448_gb300 import tune
    cfg = CONFIGS["box512_mixed"]
    zs = z_schedule(cfg.z_start, cfg.z_end, cfg.n_steps)
    k0 = int(np.argmin(np.abs(zs - 1140.0)))
    box, delta, U = make_box(cfg, "mixed", 1)
    tuned = tune.apply_table(box, tune.workload_key(cfg.n, cfg.n_packets, "mixed"))
    box.state_init(zs[k0])
    advance(box, zs, k0, k0 + W)
    box.ensure_stats(K)
    box.timing(True)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record(box.stream)
    for k in range(K):
        s = k0 + W + k
        box.transport(s, zs[s], slot=k)
        box.step(s, zs[s], zs[s + 1], slot=k)
    e1.record(box.stream)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1)
    kt = box.kernel_times()
    st = box.stats_all()[:K]
    box_tuning = box.tuning()
    box.close()
    del delta, U
    _FIELDS.pop((cfg, 1), None)  # 2 GB of host fields
    torch.cuda.empty_cache()
    emitted = sum(r["emitted"] for r in st) / K
    queued = sum(r["queued"] for r in st) / K
    crossings = sum(r["crossings"] for r in st) / K
    passes = sum(r["newton_passes"] for r in st) / K
    requeued = sum(r["requeued"] for r in st) / K
    if any(r["flags"] & 4 for r in st) or emitted < cfg.n_packets:
        raise RuntimeError("512^3 steps: invalid state")
    n3 = cfg.n ** 3
    mb = method_bytes("mixed", n3, emitted, queued, crossings, passes)
    peak, kind = measured_peaks()
    march_ms = kt["march"][0] / K
    return {"workload": (f"512^3 periodic box (24 kpc), sigma_lnrho 1.2, sigma_v 2 km/s, {cfg.n_packets:.0e} Lya "
                         f"packets/step, tally mixing, mixed form, steps {k0 + W}+ of {cfg.n_steps} (z "
                         f"{zs[k0]:.0f}) from the Saha state at step {k0}"),
            "value": n3 * K / (ms * 1e-3), "unit": "cell-steps/s", "ms_per_step": ms / K, "steps": K, "warmup": W,
            "packets_per_s": emitted * K / (ms * 1e-3), "crossings_per_packet": crossings / max(emitted, 1),
            "kernel_ms_per_step": {g: v[0] / K for g, v in kt.items() if v[1]},
            "tuning": dict(box_tuning, source="autotuner table" if tuned else "defaults"),
            "requeued_per_step": requeued,
            "march_roofline": {"bound": "hbm", "achieved": mb["march"] / (march_ms * 1e-3) / 1e9, "peak": peak,
                               "unit": "GB/s", "frac": mb["march"] / (march_ms * 1e-3) / 1e9 / peak,
                               "peak_source": f"{kind} hbm_gbs"},
            "whole_step_frac": mb["whole"] / (ms / K * 1e-3) / 1e9 / peak}


def traj_k(S):
    return max(1, math.ceil(math.sqrt(S)))


def time_batched(W, K, prep=60, n_boxes=64):
    """The batched workload: 64 boxes with sides uniform in {32,48,64,96,128},
    sigma_lnrho uniform in [0.1, 1.5], 1e6 packets per 32^3 scaled by volume,
    mixed form, tally mixing, z 1600 -> 700 in 200 steps; one context: a step
    is three launches for all boxes (persistent allocation + emission, march,
    persistent rec_step).  Timed after `prep` + W untimed steps, K steps with
    kernel timing (per-group times), then K steps as captured CUDA graphs
    (rec_graph_step), the line's value."""
    import torch
    from paper_2312_11448_gb300 import rec
    from paper_2312_11448_gb300.inputs import batched_configs, make_box as fields, z_schedule
    cfgs = batched_configs(7, n_boxes)
    boxes = []
    for i, c in enumerate(cfgs):
        d, U = fields(c, seed=100 + i)
        boxes.append((c.n, d, U, c.n_packets))
    zs = z_schedule(cfgs[0].z_start, cfgs[0].z_end, cfgs[0].n_steps)
    batch = rec.Batch(boxes, precision="mixed", mixing="tally", seed=7, stream=torch.cuda.Stream())
    del boxes
    from paper_2312_11448_gb300 import tune
    tuned = tune.apply_table(batch, tune.batch_key(n_boxes, "mixed"))
    batch.state_init(zs[0])
    for s in range(prep + W):
        batch.transport(s, zs[s])
        batch.step(s, zs[s], zs[s + 1])
    batch.timing(True)
    stream = batch.stream
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record(stream)
    emitted = 0
    for k in range(K):
        s = prep + W + k
        batch.transport(s, zs[s])
        batch.step(s, zs[s], zs[s + 1])
    e1.record(stream)
    torch.cuda.synchronize()
    ms_direct = e0.elapsed_time(e1)
    kt = batch.kernel_times()
    batch.timing(False)
    # the same steps as one captured graph per step (executable graph updated in place)
    s0 = prep + W + K
    batch.graph_step(s0, zs[s0], zs[s0 + 1])
    torch.cuda.synchronize()
    e0.record(stream)
    for k in range(K):
        s = s0 + 1 + k
        batch.graph_step(s, zs[s], zs[s + 1])
    e1.record(stream)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1)
    batch.sync()  # raises if a bounded device-side wait expired
    st = batch.stats()
    emitted = sum(r["emitted"] for r in st)
    flags = 0
    for r in st:
        flags |= r["flags"]
    cells = sum(c.n ** 3 for c in cfgs)
    tuning = batch.tuning()
    batch.close()
    torch.cuda.empty_cache()
    if flags & 4 or emitted < sum(c.n_packets for c in cfgs):
        raise RuntimeError(f"batched: invalid state (flags={flags}, emitted={emitted})")
    sides = sorted({c.n for c in cfgs})
    return {"workload": (f"{n_boxes} boxes, sides in {sides} (uniform draw), sigma_lnrho U[0.1,1.5], 1e6 packets "
                         f"per 32^3 scaled by volume, mixed form, tally mixing, steps {prep + W}+ of 200 "
                         f"(z 1600->700), one context"),
            "value": cells * K / (ms * 1e-3), "unit": "cell-steps/s", "ms_per_step": ms / K, "steps": K,
            "api": "rec_graph_step: one CUDA graph per step (3 kernels), executable graph updated in place",
            "direct_ms_per_step": ms_direct / K,
            "warmup": W, "cells": cells, "packets_per_step": emitted,
            "packets_per_s": emitted * K / (ms * 1e-3),
            "kernel_ms_per_step": {g: v[0] / K for g, v in kt.items() if v[1]},
            "launches_per_step": sum(v[1] for v in kt.values()) / K, "flags": flags,
            "tuning": dict(tuning, source="autotuner table" if tuned else "defaults")}


# ---------------------------------------------------- resonant-scattering Monte Carlo
# GB300 FP64 peak from its nominal 1.25 TFLOP/s: 0.625e12 fused multiply-adds per
# second; a separate multiply or add issues at the same rate, so the peak counts
# FP64 instructions.
# Roofline of the Monte-Carlo kernels (profiles/k_scatter_mc_z1700.md): ncu
# counts on one launch of the bench workload (8192 photons capped at 2e4 steps,
# 1.57e8 photon steps, one scattering per 10.5 steps), amortised per photon
# step.  The binary64 kernel is bound by its binary64 pipe (94.2 SM-cycles of
# that pipe per step: sm__pipe_fp64_cycles_active x sm__cycles_active / steps);
# the mixed kernel by instruction issue (17.6 warp instructions per step:
# smsp__inst_executed / steps).  Peaks: every SM's binary64 pipe busy every
# cycle, and one warp instruction per cycle per SM sub-partition, at the
# 2070 MHz maximum SM clock of the 152 SMs.
_SM_CYCLES_PER_S = 152 * 2.070e9
MC_PROFILE = {
    "fp64": {"bound": "fp64-pipe", "kernel": "k_scatter (binary64)", "per_step": 94.2, "per_scatter": 0.0,
             "peak": _SM_CYCLES_PER_S, "unit": "G SM-cycles/s of the binary64 pipe",
             "note": "94.2 binary64-pipe SM-cycles per photon step (ncu), peak = every SM's pipe every cycle"},
    "mixed": {"bound": "issue", "kernel": "k_scatter_mixed (binary32 + double-float)", "per_step": 17.6,
              "per_scatter": 0.0, "peak": 4 * _SM_CYCLES_PER_S, "unit": "G warp instructions/s",
              "note": "17.6 warp instructions per photon step (ncu), peak = one per cycle per SM sub-partition"},
}


def scatter_workload():
    from paper_2312_11448_gb300.inputs import density_field, velocity_field
    n, z = 32, 1700.0
    return n, z, density_field(n, 0.8, 11).ravel(), velocity_field(n, 1.0, 11)


def time_scatter(cpu=True, arith="fp64", photons_per_lane=1):
    """Appendix A Monte Carlo (lya_scatter_mc) in a 32^3 box (sigma_lnrho 0.8,
    sigma_v 1 km/s, Saha x_e) at z = 1700 with the true expansion rate; photons
    end by photo-ionisation after ~2e4 scatterings.  Throughput over the whole
    launch, tail included.  arith: "fp64" (binary64, the oracle's operation
    order) or "mixed" (binary32 with double-float position and frequency);
    photons_per_lane photons per resident lane (lanes refill from a counter,
    so more photons than lanes shorten the relative tail)."""
    import torch
    from paper_2312_11448_gb300 import rec
    n, z, d, U = scatter_workload()
    box = rec.Box(n, d, U, 1000, precision="mixed", mixing="full", seed=11)
    box.state_init(z)
    lanes = torch.cuda.get_device_properties(torch.cuda.current_device()).multi_processor_count * 2 * 256
    n_ph = lanes * photons_per_lane
    kw = dict(x_lost=2000.0, max_steps=1_000_000, arith=arith)
    box.scatter_mc(z, 2048, records=False, **kw)  # warm-up (module load, Voigt nodes)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record(box.stream)
    _, st = box.scatter_mc(z, n_ph, records=False, step=1, **kw)
    e1.record(box.stream)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1)
    steps_s = st["steps"] / (ms * 1e-3)
    scat_s = st["scatterings"] / (ms * 1e-3)
    out = {"workload": f"Appendix A Monte Carlo, {n}^3 box (24 kpc, sigma_lnrho 0.8, sigma_v 1 km/s), Saha x_e, "
                       f"z = {z:.0f}, zeta = 1, eps = 0.1, {n_ph} photons ({photons_per_lane} per resident lane), "
                       f"{'binary64' if arith == 'fp64' else 'mixed (binary32 + double-float)'} arithmetic",
           "arith": arith, "photons_per_s": n_ph / (ms * 1e-3), "steps_per_s": steps_s, "scatterings_per_s": scat_s,
           "ms": ms, "photons": n_ph, "fates": dict(zip(rec.MC_FATES, st["count"])),
           "sampler_caps": st["sampler_caps"], "steps_per_photon": st["steps"] / n_ph, "gpu_launches": 2}
    prof = MC_PROFILE.get(arith)
    if prof:  # instruction counts per step and per scattering from the committed ncu summary
        ach = prof["per_step"] * steps_s + prof["per_scatter"] * scat_s
        out["roofline"] = {"bound": prof["bound"], "kernel": prof["kernel"], "achieved": ach / 1e9,
                           "peak": prof["peak"] / 1e9, "unit": prof["unit"], "frac": ach / prof["peak"],
                           "traffic": None, "note": prof["note"]}
    if cpu:
        out["cpu_baseline"] = scatter_cpu_baseline(box, n, z, n_ph, kw)
    box.close()
    return out


def scatter_cpu_baseline(box, n, z, n_photons, kw, sample=32):
    """The oracle's Monte Carlo on the first `sample` photons of the same run (one core)."""
    import numpy as np
    import oracle as O
    cp = O.default_cosmo()
    P = (np.arange(n ** 3 + 1, dtype=np.int64) * n_photons // n ** 3).astype(np.uint32)
    mp = O.mc_params(z, seed=11, step=1, x_lost=kw["x_lost"], max_steps=kw["max_steps"])
    t0 = time.perf_counter()
    rec_, _ = O.lya_mc(cp, mp, n, box.host("delta").astype(np.float64), box.host("x"), P,
                       U=box.host("vel4")[:, :3].astype(np.float64), k0=0, k1=sample)
    dt = time.perf_counter() - t0
    return {"value": float(rec_["n_steps"].sum()) / dt, "unit": "steps/s", "cores": 1, "kind": "oracle",
            "photons_per_s": sample / dt,
            "sample": f"oracle Monte Carlo, first {sample} photons of the same run; {platform_name()}"}


# ------------------------------------------------------------------------ oracle (CPU)
def oracle_sample(cfg, zs, sample_packets, threads=0):
    """The oracle as it stands on one host core: one rec_step over every cell and
    the transport of `sample_packets` packets of the step; returns seconds.
    threads > 0: the transport runs in the OpenMP build of the same source on that
    many threads (the rec_step stays single-threaded)."""
    import oracle as O
    from paper_2312_11448_gb300.inputs import doppler_quantiles, pack_vel4
    cp = O.default_cosmo()
    delta, U = fields_of(cfg, 1)
    z = zs[S0]
    x = O.saha_xe(cp, z, delta)
    T = np.full(delta.size, O.background(cp, z)["Tg"])
    emis = O.rates(cp, z, T[0])["alpha"] * (O.background(cp, z)["nH"] * delta * x) ** 2
    v4 = pack_vel4(U, np.float32)
    t0 = time.perf_counter()
    tally, cnt, _ = O.transport(cp, cfg.n, z, 1, S0, sample_packets, emis.astype(np.float32), v4,
                                T.astype(np.float32), doppler_quantiles().astype(np.float32), precision="f32",
                                threads=threads)
    t_tr = time.perf_counter() - t0
    t0 = time.perf_counter()
    O.rec_step(cp, cfg.n, zs[S0], zs[S0 + 1], delta, x, T, U=U, tally=tally, mixing="tally")
    t_st = time.perf_counter() - t0
    return t_tr, t_st


def oracle_step_estimate(cfg, zs, sample_packets, threads=0):
    """Seconds of one whole oracle step on this workload, from the transport of
    `sample_packets` and of half as many (the time is affine in the packet
    count: a fixed part for the allocation over every cell, then a cost per
    packet) plus one rec_step over every cell.  Returns (step s, transport s of
    the sample, rec_step s, fixed transport s, transport s per packet)."""
    sample_packets = min(sample_packets, cfg.n_packets)
    half = max(1, sample_packets // 2)
    t_tr, t_st = oracle_sample(cfg, zs, sample_packets, threads)
    t_half, _ = oracle_sample(cfg, zs, half, threads)
    per = max(t_tr - t_half, 0.0) / max(sample_packets - half, 1)
    fixed = max(t_tr - per * sample_packets, 0.0)
    return fixed + per * cfg.n_packets + t_st, t_tr, t_st, fixed, per


def cpu_baseline_all_cores(cfg, zs, sample_packets=20_000_000):
    """The OpenMP build of the oracle's transport on every host core (the
    rec_step single-threaded), same workload and sample scaling."""
    cores = os.cpu_count() or 1
    sample_packets = min(sample_packets, cfg.n_packets)
    t_step, t_tr, t_st, fixed, per = oracle_step_estimate(cfg, zs, sample_packets, threads=cores)
    return {"value": cfg.n ** 3 / t_step, "unit": "cell-steps/s", "cores": cores, "kind": "oracle (OpenMP build)",
            "packets_per_s": 1.0 / per if per > 0 else None,
            "sample": (f"OpenMP build of the oracle source: transport of {sample_packets:.0e} and of half as many "
                       f"of the {cfg.n_packets:.0e} packets over {cores} threads ({t_tr:.2f} s for the sample; "
                       f"extrapolated affinely: {fixed:.2f} s fixed + {per * 1e6:.3f} s per 1e6 packets) + the "
                       f"single-threaded oracle rec_step over all {cfg.n}^3 cells ({t_st:.2f} s); "
                       f"{platform_name()}")}


def cpu_baseline(cfg, zs, sample_packets=4_000_000):
    sample_packets = min(sample_packets, cfg.n_packets)
    t_step, t_tr, t_st, fixed, per = oracle_step_estimate(cfg, zs, sample_packets)
    return {"value": cfg.n ** 3 / t_step, "unit": "cell-steps/s", "cores": 1, "kind": "oracle",
            "packets_per_s": 1.0 / per if per > 0 else None,
            "sample": (f"one oracle rec_step over all {cfg.n}^3 cells ({t_st:.2f} s) + oracle transport of "
                       f"{sample_packets:.0e} and of half as many of the {cfg.n_packets:.0e} packets ({t_tr:.2f} s "
                       f"for the sample), extrapolated affinely to the full packet count ({fixed:.2f} s fixed + "
                       f"{per * 1e6:.3f} s per 1e6 packets); single-threaded, {os.cpu_count()} host cores present "
                       f"({platform_name()})")}


def platform_name():
    import platform
    try:
        for line in open("/proc/cpuinfo"):
            if line.lower().startswith(("model name", "cpu part")):
                return f"{platform.machine()} {line.split(':', 1)[1].strip()}"
    except OSError:
        pass
    return platform.machine()


def measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        d = json.load(open(p))
        return d.get("hbm_gbs", 6800.0), "measured"
    return 6800.0, "fallback"


# Source text a kernel's counters depend on: the whole file, or for the march the
# traversal helpers and the march kernel itself (the emission, which shares the
# file, can change without changing a byte of the march).
PROFILED_SOURCE = {
    "march": ("k_march_256.md", "rec_transport.cu",
              (("// Traversal state of one packet.", "__device__ __forceinline__ void add_counters("),
               ("// March of the queued packets.", "// Region sweeps, between two march launches (one block)"))),
    "emit": ("k_emit_256.md", "rec_transport.cu", None),
    "rec_step": ("rec_step_passes_256.md", "rec_step.cu", None),
}


def source_hash(src_text, regions):
    """sha256 (16 hex digits) of the file, or of the concatenated marked regions."""
    import hashlib
    if regions is None:
        return hashlib.sha256(src_text.encode()).hexdigest()[:16]
    parts = []
    for a, b in regions:
        i = src_text.index(a)
        parts.append(src_text[i:src_text.index(b, i)])
    return hashlib.sha256("".join(parts).encode()).hexdigest()[:16]


def profiled_traffic(group):
    """dram bytes per launch of a kernel from its committed ncu summary
    (profiles/<kernel>_256.md), valid only while the source it depends on is
    unchanged (its hash is recorded beside the figure)."""
    if group not in PROFILED_SOURCE:
        return None
    md, src, regions = PROFILED_SOURCE[group]
    f = os.path.join(ROOT, "profiles", md)
    srcp = os.path.join(ROOT, "paper_2312_11448_gb300", "csrc", src)
    if not os.path.exists(f):
        return None
    try:
        h = source_hash(open(srcp).read(), regions)
    except ValueError:  # a marker is gone: the source was reorganised
        return None
    vals = {}
    for line in open(f):
        if ":" in line and line.strip().startswith(("traffic_bytes_per_launch", "source_sha256_16")):
            k, v = line.split(":", 1)
            vals[k.strip()] = v.strip().strip("`")
    if vals.get("source_sha256_16") != h:
        return None
    try:
        return float(vals["traffic_bytes_per_launch"])
    except (KeyError, ValueError):
        return None


# ------------------------------------------------------------------------ multi-rank
def rank_env():
    """(rank, world size, local rank) from the torchrun environment."""
    return int(os.environ.get("RANK", 0)), int(os.environ.get("WORLD_SIZE", 1)), int(os.environ.get("LOCAL_RANK", 0))


def rank_seed(rank):
    """Each rank runs its own independent box (weak scaling): seed 1 + rank."""
    return 1 + rank


def reduce_max(v, dist, device):
    """Max over ranks of a timing (the slowest rank sets the whole job's time)."""
    if dist is None:
        return v
    import torch
    t = torch.tensor([v], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_value(world, units_per_rank, K, ms_max):
    """Whole-job throughput: the units all ranks processed over the slowest rank's time."""
    return world * units_per_rank * K / (ms_max * 1e-3)


# ---------------------------------------------------------------------------- arms
def run_ours(args):
    import torch
    rank, world, local = rank_env()
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    torch.cuda.set_device(local)
    import __graft_entry__
    __graft_entry__.build()
    cfg, zs = workload(args.n, args.packets)
    K, W = args.steps, max(3, args.warmup)
    clocks = Clocks(local)
    mixed = time_form(cfg, zs, "mixed", W, K, seed=rank_seed(rank), dist=dist, clocks=clocks, prep=args.prep,
                      graph=True)
    fp64 = None
    if not args.no_fp64:
        fp64 = time_form(cfg, zs, "fp64", W, max(5, K // 3), seed=rank_seed(rank), dist=dist, clocks=clocks,
                         prep=args.prep)
    e2e = None if args.no_e2e else time_e2e(cfg, zs, mixed, K)
    big = None
    if not args.no_512 and world == 1:
        for r in (fp64,):
            if r:
                r["box"].close()
        torch.cuda.empty_cache()
        t0 = clocks.mark()
        big = time_512()
        clocks.window(t0, clocks.mark())
    adjoint = None
    if not args.no_adjoint and world == 1:
        for r in (fp64,):
            if r:
                r["box"].close()
        torch.cuda.empty_cache()
        t0 = clocks.mark()
        adjoint = time_adjoint(cfg, zs)
        clocks.window(t0, clocks.mark())
    batched = None
    if not args.no_batched:
        for r in (mixed, fp64):
            if r:
                r["box"].close()
        torch.cuda.empty_cache()
        t0 = clocks.mark()
        batched = time_batched(W=2, K=max(3, K // 6))
        clocks.window(t0, clocks.mark())
    scatter = None
    if not args.no_scatter and world == 1:
        t0 = clocks.mark()
        try:
            scatter = time_scatter(cpu=not args.no_cpu)
            scatter["mixed_arith"] = time_scatter(cpu=False, arith="mixed", photons_per_lane=4)
            scatter["mixed_arith"]["photons_per_s_over_fp64"] = (scatter["mixed_arith"]["photons_per_s"] /
                                                                 scatter["photons_per_s"])
        except Exception as exc:  # a secondary line: report, keep the main measurement
            scatter = {"error": f"{type(exc).__name__}: {exc}"}
        clocks.window(t0, clocks.mark())
    clk = clocks.summary()

    def max_over_ranks(v):
        return reduce_max(v, dist, "cuda")

    ms_mixed = max_over_ranks(mixed["ms"])
    ms_fp64 = max_over_ranks(fp64["ms"]) if fp64 else None
    ms_e2e = max_over_ranks(e2e[0]) if e2e else None
    ms_graph = max_over_ranks(mixed["graph_ms"]) if "graph_ms" in mixed else None
    n3 = cfg.n ** 3
    K64 = max(5, K // 3)
    if rank != 0:
        dist.barrier() if dist else None
        return
    value = job_value(world, n3, K, ms_mixed)
    peak, peak_kind = measured_peaks()
    groups = {g: v for g, v in mixed["kt"].items() if v[1]}
    dominant = max(("emit", "march", "rec_step", "alloc"), key=lambda g: groups.get(g, (0, 0))[0])
    names = {"emit": "k_emit<float, pow2> (packet emission + home-cell test)",
             "march": "k_march<float, pow2> (march of queued packets)",
             "rec_step": "rec_step (k_substep_tma: evaluation and final passes)", "alloc": "allocation (3 kernels)"}

    def roof(g):
        """frac on the method's bytes (method_bytes); the library's own count,
        which adds its intermediate traffic, beside it."""
        ms_g = groups[g][0] / K
        mb = mixed["mb"].get(g, mixed["ab"][g])
        ach = mb / (ms_g * 1e-3) / 1e9
        ach_b = mixed["ab"][g] / (ms_g * 1e-3) / 1e9
        return {"bound": "hbm", "kernel": names[g], "achieved": ach, "peak": peak, "unit": "GB/s",
                "frac": ach / peak, "peak_source": f"{peak_kind} hbm_gbs (of {peak_kind})",
                "algorithmic_bytes_per_launch": mb, "avg_launch_ms": ms_g,
                "bytes_rule": "method bytes (16 B/packet + 4 B/tally + 16 B/crossing; rec_step 20 B/pass + 64 B); "
                              "the march settles most crossings from a 4-byte copy of the velocity, so its fraction "
                              "on the method's 16 B can pass 1"
                if g != "alloc" else "library count (3 reads of r + prefix write per cell)",
                "with_library_traffic": {"algorithmic_bytes_per_launch": mixed["ab"][g], "achieved": ach_b,
                                         "frac": ach_b / peak}}

    def rec_step_two_pass(groups, k_steps, n3, peak):
        """rec_step against the fixed per-cell-step count of a step with two
        evaluation passes and the final pass (20 + 20 + 64 B mixed): the
        Halley update needs one pass where Newton needed two, which the
        method-byte fraction above does not credit.  The fraction of the
        passes that run is roofline_other.rec_step."""
        if "rec_step" not in groups:
            return None
        ms_s = groups["rec_step"][0] / k_steps
        b = 104 * n3
        return {"bytes_per_cell_step": 104, "ms_per_step": ms_s, "achieved": b / (ms_s * 1e-3) / 1e9,
                "frac": b / (ms_s * 1e-3) / 1e9 / peak, "unit": "GB/s", "peak": peak,
                "rule": "two evaluation passes counted; newton_passes of them run"}

    def whole_step(r, k_steps, ms_total):
        ms_s = ms_total / k_steps
        ach = r["mb"]["whole"] / (ms_s * 1e-3) / 1e9
        return {"bound": "hbm", "achieved": ach, "peak": peak, "unit": "GB/s", "frac": ach / peak,
                "algorithmic_bytes_per_step": r["mb"]["whole"], "ms_per_step": ms_s,
                "bytes_rule": "per packet 16 B + 4 B tally + 16 B per crossing (FP64 form 32 B), per cell 20 B per "
                              "Newton pass + 64 B final (FP64 form 28 B + 100 B)"}

    launches = sum(v[1] for v in mixed["kt"].values())
    out = {
        "metric": METRIC, "value": value, "unit": "cell-steps/s", "n_gpus": world, "steps": K, "warmup": W,
        "ms_per_step": ms_mixed / K, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "mixed: f32 transport + f32 per-cell coefficients, f64 x_e state/residual/sums", "data": "synthetic",
        "config": {"workload": describe(cfg, "mixed"), "n": cfg.n, "packets_per_step": cfg.n_packets,
                   "parallelism": f"{world} independent boxes (one per GPU)" if world > 1 else "single GPU",
                   "l2": "working set 0.74 GB (mixed) / 1.2 GB (fp64) > 129 MB L2, no flush needed"},
        "packets_per_s": world * mixed["emitted"] * K / (ms_mixed * 1e-3),
        "kernel_ms_per_step": {g: v[0] / K for g, v in mixed["kt"].items() if v[1]},
        "crossings_per_packet": mixed["crossings"] / max(mixed["emitted"], 1),
        "newton_passes": mixed["passes"], "X_e": mixed["Xe"], "flags": mixed["flags"],
        "roofline": dict(roof(dominant), traffic=profiled_traffic(dominant)),
        "roofline_other": {g: roof(g) for g in ("emit", "march", "rec_step", "alloc") if g in groups and g != dominant},
        "rec_step_per_cell_step": rec_step_two_pass(groups, K, n3, peak),
        "roofline_whole_step": whole_step(mixed, K, ms_mixed),
        "queued_fraction": mixed["queued"] / max(mixed["emitted"], 1),
        "tuning": mixed["tuning"],
        "gpu_launches": launches,
    }
    if fp64:
        out["fp64_form"] = {"value": world * n3 * K64 / (ms_fp64 * 1e-3), "unit": "cell-steps/s",
                            "ms_per_step": ms_fp64 / K64, "steps": K64,
                            "packets_per_s": world * fp64["emitted"] * K64 / (ms_fp64 * 1e-3),
                            "kernel_ms_per_step": {g: v[0] / K64 for g, v in fp64["kt"].items() if v[1]},
                            "mixed_over_fp64": (ms_fp64 / K64) / (ms_mixed / K),
                            "roofline_whole_step": whole_step(fp64, K64, ms_fp64)}
    if e2e:
        out["e2e"] = {"value": world * n3 * K / (ms_e2e * 1e-3), "unit": "cell-steps/s", "h2d_bytes_per_step": e2e[1],
                      "d2h_bytes_per_step": e2e[2],
                      "api": "rec.Box: per step H2D of delta and velocity (pinned host memory), lya_transport, "
                             "rec_step, D2H of x_e and T; copies on their own streams, overlapped with the "
                             "neighbouring step's compute"}
    if ms_graph:
        gms = ms_graph
        out["graph"] = {"ms_per_step": gms / K, "value": world * n3 * K / (gms * 1e-3), "unit": "cell-steps/s",
                        "api": "rec_graph_step: transport + rec_step captured as one CUDA graph per step, "
                               "executable graph updated in place", "steps": K}
    if big:
        out["box512"] = big
    if adjoint:
        if fp64:
            f_ms = ms_fp64 / K64
            f_step_ms = fp64["kt"]["rec_step"][0] / K64
            adjoint["fp64_forward_step_ms"] = f_ms
            adjoint["reverse_over_forward_step"] = adjoint["reverse_ms_per_step"] / f_ms
            adjoint["reverse_over_forward_rec_step"] = adjoint["reverse_ms_per_step"] / f_step_ms
        out["adjoint"] = adjoint
    if batched:
        out["batched"] = batched
    if scatter:
        out["scatter_mc"] = scatter
    out["clocks"] = clk
    if world == 1 and not args.no_cpu:
        out["cpu_baseline"] = cpu_baseline(cfg, zs)
        out["cpu_baseline_all_cores"] = cpu_baseline_all_cores(cfg, zs)
    print(json.dumps(out), flush=True)
    if dist:
        dist.barrier()


def run_reference(args):
    """The oracle (CPU, single-threaded) on the same workload and metric; each
    step is a bounded sample: one rec_step over every cell plus the transport
    of a fraction of the packets, scaled to the full packet count."""
    rank, world = int(os.environ.get("RANK", 0)), int(os.environ.get("WORLD_SIZE", 1))
    if rank != 0:
        return
    cfg, zs = workload(args.n, args.packets)
    sample = min(2_000_000, cfg.n_packets)
    K, W = args.steps, args.warmup
    for _ in range(W):
        oracle_sample(cfg, zs, sample)
    tot = 0.0
    for _ in range(K):
        tot += oracle_step_estimate(cfg, zs, sample)[0]
    ms = tot / K * 1e3
    value = cfg.n ** 3 / (ms * 1e-3)
    # an unsampled anchor: one whole oracle step (every packet) on a 64^3 box at
    # the same packets per cell, against the rate the sampled step assumes
    n_a = 64
    cfg_a, zs_a = workload(n_a, max(1, int(round(cfg.n_packets * (n_a / cfg.n) ** 3))))
    t_tr_a, t_st_a = oracle_sample(cfg_a, zs_a, cfg_a.n_packets)
    est_a = oracle_step_estimate(cfg_a, zs_a, cfg_a.n_packets // 16)[0]
    anchor = {"workload": describe(cfg_a, "oracle") + ", every packet transported",
              "ms_per_step": (t_tr_a + t_st_a) * 1e3, "cell_steps_per_s": n_a ** 3 / (t_tr_a + t_st_a),
              "packets_per_s": cfg_a.n_packets / t_tr_a,
              "estimate_from_a_1_16_sample_ms": est_a * 1e3,
              "note": "a whole oracle step at 64^3 (same packets per cell), and the same step estimated the "
                      "way the 256^3 line is (affine in the packets, from a sample and half of it)"}
    out = {"impl": "reference", "metric": METRIC, "value": value, "unit": "cell-steps/s", "n_gpus": 0, "steps": K,
           "warmup": W, "ms_per_step": ms, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
           "dtype": "f64 (oracle; binary32 transport arithmetic; transport sampled and extrapolated)", "data": "synthetic",
           "config": {"workload": describe(cfg, "oracle"), "n": cfg.n, "packets_per_step": cfg.n_packets,
                      "sampled": f"each timed step transports {sample:.0e} and {sample // 2:.0e} of the "
                                 f"{cfg.n_packets:.0e} packets and extrapolates the transport time affinely "
                                 f"(fixed allocation + cost per packet); ms_per_step is that estimate, not wall "
                                 f"time"},
           "cpu_baseline": {"value": value, "unit": "cell-steps/s", "cores": 1, "kind": "oracle",
                            "sample": f"per step: oracle rec_step over all cells + transport of {sample:.0e} and "
                                      f"{sample // 2:.0e} packets extrapolated to {cfg.n_packets:.0e}; "
                                      f"{platform_name()}"},
           "e2e": {"value": value, "unit": "cell-steps/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
           "unsampled_anchor": anchor}
    print(json.dumps(out), flush=True)


if __name__ == "__main__":
    a = parse()
    if a.impl == "reference":
        run_reference(a)
    else:
        run_ours(a)
