"""Benchmark of the smoothed image-method objective on GB300.

One step = one pass of the whole hot path over the large scene (square + 60
random segments = 64 walls, 256 x 256 receiver grid, K <= 2 i.e. 4097 wall
sequences, alpha = 100, hard sigmoid): received power of every receiver
(forward kernel), the min-power loss, its gradient w.r.t. power, and the
hand-written adjoint (gradient w.r.t. the TX and all wall end points).

Prints one JSON line (rank 0).  Multi-GPU (torchrun): every rank runs its own
replica (independent problem: its own TX position), no collective on the data
path; timing is the max over ranks ("weak" scaling).

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
"""
from __future__ import annotations

import argparse
import csv
import hashlib
import io
import json
import os
import statistics
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = ("path×RX evals/s fwd+adjoint, % FP32 roofline; time-to-optimum vs plain at 1e-3")
UNIT = "path×RX evals/s"
L2_FLUSH_BYTES = 256 << 20
TRAFFIC_FILE = os.path.join(ROOT, "profiles", "forward_large_scene_traffic.txt")


def workload_scene(rank: int = 0, rx_grid: int = 256, smoothing: str = "hard_sigmoid",
                   alpha: float = 100.0):
    from paper_2401_11882_gb300 import scenes
    sc = scenes.clutter_scene(60, rx_grid, 0, alpha, smoothing, 2, True)
    if rank:
        # an independent problem per rank: the TX moves along the grid's middle row
        sc = sc.replace(tx=np.array([0.5 + 0.011 * ((rank % 30) - 15), 0.2], np.float32))
    return sc


def workload_config(sc, n_cand):
    return {
        "workload": (f"square + 60 random segments ({sc.n_walls} walls, seed 0), "
                     f"{int(round(sc.n_rx ** 0.5))}x{int(round(sc.n_rx ** 0.5))} RX grid, "
                     f"K<={sc.max_order} ({n_cand} wall sequences), "
                     f"alpha={sc.alpha:g}, {sc.smoothing}; forward + min-loss + adjoint "
                     "(grad wrt TX and all wall end points)"),
        "n_walls": sc.n_walls, "n_rx": sc.n_rx, "max_order": sc.max_order, "alpha": sc.alpha,
        "smoothing": sc.smoothing, "evals_per_step": sc.n_rx * n_cand,
        "l2": "flushed between timed steps (256 MiB write)",
        "inputs": "resident in HBM",
    }


# ------------------------------------------------------------------ clocks
class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None

    def stop(self) -> dict | None:
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            out, _ = self.proc.communicate(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
            out, _ = self.proc.communicate()
        rows = [r for r in csv.reader(io.StringIO(out)) if len(r) >= 9]
        if not rows:
            return None
        sm = [float(r[1]) for r in rows if r[1].strip().replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].strip().replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({n for r in rows for n, v in zip(names, r[5:9]) if v.strip() == "Active"})
        loaded = [s for s in sm if mx and s >= 0.5 * max(mx)] or sm
        return {"sm_mhz": statistics.median(loaded) if loaded else None,
                "sm_max_mhz": max(mx) if mx else None, "reasons": reasons,
                "samples": len(rows)}


# ------------------------------------------------------------------ CPU oracle
def oracle_rate(sc, n_cand, budget_s: float = 8.0, max_rx: int = 4096):
    """Oracle forward over a growing prefix of the receivers until ~budget_s of wall time."""
    import oracle
    oracle.build()
    threads = os.cpu_count() or 1
    n = 16
    while True:
        t0 = time.perf_counter()
        oracle.power(sc.walls, sc.tx, sc.rx[:n], sc.max_order, sc.alpha, sc.smoothing,
                     sc.refl_coef, threads=threads)
        dt = time.perf_counter() - t0
        if dt >= budget_s or n >= max_rx:
            break
        n = min(max_rx, max(2 * n, int(n * budget_s / max(dt, 1e-3))))
    return n * n_cand / dt, threads, n, dt


# ------------------------------------------------------------------ reference arm
def run_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    from paper_2401_11882_gb300 import workload
    sc = workload_scene(0, args.rx_grid, args.smoothing, args.alpha)
    n_cand = workload.num_candidates(sc.n_walls, sc.max_order)
    import oracle
    oracle.build()
    threads = os.cpu_count() or 1
    n_rx = 2 * threads
    sub = sc.rx[:n_rx]
    for _ in range(args.warmup):
        oracle.power(sc.walls, sc.tx, sub[:threads], sc.max_order, sc.alpha, sc.smoothing)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        oracle.power(sc.walls, sc.tx, sub, sc.max_order, sc.alpha, sc.smoothing, threads=threads)
    dt = time.perf_counter() - t0
    value = args.steps * n_rx * n_cand / dt
    sample = f"{n_rx} receivers x {n_cand} sequences per step (forward power only)"
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT,
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * dt / args.steps, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": workload_config(sc, n_cand),
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": threads, "kind": "oracle",
                             "sample": sample},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


# ------------------------------------------------------------------ our arm
def file_hash(path: str) -> str:
    with open(path, "rb") as f:
        return hashlib.sha256(f.read()).hexdigest()[:16]


FORWARD_SOURCES = ("drt_forward.cu", "drt_path.cuh", "drt_path_pair.cuh", "drt_path_queue.cuh",
                   "drt_common.cuh")


def forward_source_hash() -> str:
    h = hashlib.sha256()
    for name in FORWARD_SOURCES:
        with open(os.path.join(ROOT, "paper_2401_11882_gb300", "csrc", name), "rb") as f:
            h.update(f.read())
    return h.hexdigest()[:16]


def measured_traffic():
    """DRAM bytes per forward launch from the committed ncu summary, if it was taken on
    the current forward kernel sources (key: value lines)."""
    try:
        d = {}
        with open(TRAFFIC_FILE) as f:
            for line in f:
                if ":" in line:
                    k, v = line.split(":", 1)
                    d[k.strip()] = v.strip()
        if d.get("kernel_sha256_16") == forward_source_hash():
            return float(d["dram_bytes_per_launch"])
    except (OSError, ValueError, KeyError):
        pass
    return None


def peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return json.load(f)
    except (OSError, ValueError):
        return {}


def run_ours(args):
    import torch
    import torch.distributed as dist

    import paper_2401_11882_gb300 as drt
    from paper_2401_11882_gb300 import workload

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if world > 1:
        dist.init_process_group("nccl", device_id=dev)

    sc = workload_scene(rank, args.rx_grid, args.smoothing, args.alpha)
    n_cand = drt.num_candidates(sc.n_walls, sc.max_order)
    work = workload.forward_work(sc.n_walls, sc.max_order, sc.n_rx)
    w = torch.tensor(sc.walls, device=dev)
    t = torch.tensor(sc.tx, device=dev)
    r = torch.tensor(sc.rx, device=dev)
    K, alpha, sm = sc.max_order, sc.alpha, sc.smoothing
    flush = torch.empty(L2_FLUSH_BYTES, dtype=torch.uint8, device=dev)

    ev = [[torch.cuda.Event(enable_timing=True) for _ in range(3)] for _ in range(args.steps)]

    def step(i=None):
        e = ev[i] if i is not None else None
        if e:
            e[0].record()
        P = drt.forward(w, t, r, K, alpha, sm)
        if e:
            e[1].record()
        loss, am = drt.min_loss(P)
        gtx, gw = drt.min_loss_vjp(w, t, r, K, alpha, sm, am)
        if e:
            e[2].record()
        return loss, gtx, gw

    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize(dev)
    if world > 1:
        dist.barrier()
    clocks = ClockSampler(local)
    clocks.start()
    time.sleep(0.3)
    torch.cuda.synchronize(dev)
    for i in range(args.steps):
        flush.zero_()
        step(i)
    torch.cuda.synchronize(dev)
    if world > 1:
        dist.barrier()
    clk = clocks.stop()
    step_ms = [ev[i][0].elapsed_time(ev[i][2]) for i in range(args.steps)]
    fwd_ms = [ev[i][0].elapsed_time(ev[i][1]) for i in range(args.steps)]
    total_ms = sum(step_ms)
    if world > 1:
        tt = torch.tensor([total_ms], device=dev, dtype=torch.float64)
        dist.all_reduce(tt, op=dist.ReduceOp.MAX)
        total_ms = float(tt.item())
    evals = sc.n_rx * n_cand
    value = world * args.steps * evals / (total_ms / 1e3)

    # end to end through the C ABI's host-array call (drt_objective_host), from pinned
    # host buffers: inputs H2D, loss, argmin, power and gradients D2H every step
    hw = torch.tensor(sc.walls).pin_memory()
    ht = torch.tensor(sc.tx).pin_memory()
    hr = torch.tensor(sc.rx).pin_memory()
    for _ in range(max(1, args.warmup)):
        drt.objective_host(hw, ht, hr, K, alpha, sm, device=dev, grad_walls=True)
    torch.cuda.synchronize(dev)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        out = drt.objective_host(hw, ht, hr, K, alpha, sm, device=dev, grad_walls=True)
    e2e_s = time.perf_counter() - t0
    if world > 1:
        tt = torch.tensor([e2e_s], device=dev, dtype=torch.float64)
        dist.all_reduce(tt, op=dist.ReduceOp.MAX)
        e2e_s = float(tt.item())
    h2d = hw.numel() * 4 + ht.numel() * 4 + hr.numel() * 4
    # loss, power, grad_tx, grad_walls and the 4-byte argmin drt_objective_host copies back
    d2h = sum(o.numel() * o.element_size() for o in out) + 4

    # extras (not part of the timed step): sigmoid forward, dense adjoint on the
    # 128-wall gradient scene
    extras = {}
    if rank == 0 and not args.no_extras:
        extras = measure_extras(drt, dev, sc, w, t, r)

    if rank != 0:
        if world > 1:
            dist.destroy_process_group()
        return 0

    pk = peaks()
    props = torch.cuda.get_device_properties(dev)
    sm_max = float(pk.get("sm_max_mhz") or (clk or {}).get("sm_max_mhz") or 2070.0)
    peak = workload.fp32_peak_tflops(props.multi_processor_count, sm_max)
    fwd_avg_s = (sum(fwd_ms) / len(fwd_ms)) / 1e3
    needed = workload.needed_flops(sc.n_walls, sc.max_order, sc.rx.shape[0], sc.smoothing)
    achieved = needed / fwd_avg_s / 1e12
    traffic = measured_traffic()
    cpu = None
    if not args.no_cpu_baseline and world == 1:
        rate, cores, n, dt = oracle_rate(sc, n_cand)
        cpu = {"value": rate, "unit": UNIT, "cores": cores, "kind": "oracle",
               "sample": f"first {n} receivers of the workload x {n_cand} sequences, "
                         f"forward power only, {dt:.1f} s"}
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": total_ms / args.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": workload_config(sc, n_cand),
        "roofline": {"bound": "alu", "achieved": achieved, "peak": peak, "unit": "TFLOP/s",
                     "frac": achieved / peak, "traffic": traffic,
                     "kernel": ((f"forward_pair_kernel<{sc.smoothing}>"
                                 if sc.smoothing in ("hard_sigmoid", "sigmoid") and sc.alpha <= 1e4
                                 else f"forward_kernel<{sc.smoothing}>")
                                + " (+ its chunk-sum kernel)"),
                     "peak_source": f"{props.multi_processor_count} SMs x 128 FP32 lanes x 2 "
                                    f"FLOP x {sm_max:.0f} MHz (max SM clock)",
                     "flops_per_launch": needed, "ms_per_launch": fwd_avg_s * 1e3,
                     "flops_by_convention": work["flops"],
                     "note": "achieved counts 40 FLOP per reflection and 20 per path of every "
                             "(receiver, sequence) pair and 40 per wall test of the lines of "
                             "sight; paths of validity exactly 0 are evaluated to their power "
                             "0 without their wall tests, so the convention's 40 FLOP per leg "
                             "x wall test of every path no longer describes the work"},
        "cpu_baseline": cpu,
        "e2e": {"value": world * args.steps * evals / e2e_s, "unit": UNIT,
                "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h},
        "gpu_launches": 5 * args.steps,
        "clocks": clk,
        "extra": extras,
    }
    print(json.dumps(line), flush=True)
    if world > 1:
        dist.destroy_process_group()
    return 0


def measure_extras(drt, dev, sc, w, t, r):
    import torch
    from paper_2401_11882_gb300 import scenes, workload

    def timed(fn, n=3):
        fn()
        torch.cuda.synchronize(dev)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(n):
            fn()
        b.record()
        torch.cuda.synchronize(dev)
        return a.elapsed_time(b) / n / 1e3

    out = {}
    n_cand = workload.num_candidates(sc.n_walls, sc.max_order)
    ev = sc.n_rx * n_cand
    for a_ in (10.0, 1000.0):
        s = timed(lambda: drt.forward(w, t, r, sc.max_order, a_, sc.smoothing))
        out[f"forward_alpha_{a_:g}_evals_per_s"] = ev / s
    s = timed(lambda: drt.forward(w, t, r, sc.max_order, sc.alpha, "sigmoid"))
    out["sigmoid_forward_evals_per_s"] = ev / s
    s = timed(lambda: drt.forward(w, t, r, sc.max_order, sc.alpha, "sigmoid",
                                  tile=drt.TileConfig(single_rx=True)))
    out["sigmoid_forward_one_rx_per_lane_evals_per_s"] = ev / s
    s = timed(lambda: drt.forward(w, t, r, sc.max_order, sc.alpha, "hard_sigmoid",
                                  tile=drt.TileConfig(single_rx=True)))
    out["hard_forward_one_rx_per_lane_evals_per_s"] = ev / s
    # 3D: the 64-wall scene as a room of 132 triangles, 128 x 128 receivers, K <= 2
    r3 = scenes.room3d(128)
    w3, t3, x3 = (torch.tensor(a, device=dev) for a in (r3.tris, r3.tx, r3.rx))
    n3 = r3.n_rx * workload.num_candidates(r3.n_tris, r3.max_order)
    s3h = timed(lambda: drt.forward3(w3, t3, x3, 2, 100.0, "hard_sigmoid"), 3)
    s3s = timed(lambda: drt.forward3(w3, t3, x3, 2, 100.0, "sigmoid"), 1)
    g3 = torch.full((r3.n_rx,), 1.0 / r3.n_rx, device=dev)
    v3h = timed(lambda: drt.vjp3(w3, t3, x3, 2, 100.0, "hard_sigmoid", g3), 2)
    v3s = timed(lambda: drt.vjp3(w3, t3, x3, 2, 100.0, "sigmoid", g3), 1)
    out["room3d_forward"] = {
        "workload": "64-wall scene as a room (walls extruded over z in [0, 1], floor, ceiling: "
                    "132 triangles), 128x128 receivers at z = 0.3, K<=2 (17425 sequences), alpha=100",
        "hard_ms": s3h * 1e3, "hard_evals_per_s": n3 / s3h,
        "sigmoid_ms": s3s * 1e3, "sigmoid_evals_per_s": n3 / s3s,
        "hard_vjp_ms": v3h * 1e3, "sigmoid_vjp_ms": v3s * 1e3,
        "note": "warps whose paths all have validity exactly 0 skip their obstruction loop; "
                "vjp = dense g = 1/R, gradient w.r.t. the TX and all 1188 corner coordinates"}
    # reflection points by the iterative path finder (10 Gauss-Newton steps on the MPT
    # cost, smoothed convergence check eps = 0.05) on the benchmark workload
    sm_h = timed(lambda: drt.forward_mpt(w, t, r, sc.max_order, sc.alpha, "hard_sigmoid", 10,
                                         0.05), 2)
    sm_s = timed(lambda: drt.forward_mpt(w, t, r, sc.max_order, sc.alpha, "sigmoid", 10, 0.05), 1)
    sf_h = timed(lambda: drt.forward_fpt(w, t, r, sc.max_order, sc.alpha, "hard_sigmoid", 10,
                                         0.05), 2)
    out["mpt_forward"] = {"workload": "benchmark workload, reflection points from 10 MPT steps "
                                      "(fermat_*: 10 Fermat path-tracing steps)",
                          "hard_ms": sm_h * 1e3, "hard_evals_per_s": ev / sm_h,
                          "sigmoid_ms": sm_s * 1e3, "sigmoid_evals_per_s": ev / sm_s,
                          "fermat_hard_ms": sf_h * 1e3, "fermat_hard_evals_per_s": ev / sf_h}
    # more walls than shared memory holds: square + 4092 segments, K <= 1, 64x64 receivers
    cs = scenes.clutter_scene(4092, 64, seed=1, alpha=100.0, smoothing="hard_sigmoid",
                              max_order=1)
    cw, ct, cr = (torch.tensor(a, device=dev) for a in (cs.walls, cs.tx, cs.rx))
    sc_h = timed(lambda: drt.forward(cw, ct, cr, 1, 100.0, "hard_sigmoid"), 1)
    n_tests = cs.n_rx * (1 + 2 * cs.n_walls) * cs.n_walls   # leg x wall tests per launch
    out["streamed_walls_4096"] = {
        "workload": "square + 4092 random segments (4096 walls, records in L2), 64x64 receivers, "
                    "K<=1 (4097 sequences), alpha=100, hard sigmoid",
        "ms": sc_h * 1e3, "evals_per_s": cs.n_rx * (1 + cs.n_walls) / sc_h,
        "tests_per_s": n_tests / sc_h}
    # coherent field (Eq. 7 with complex path fields, Fresnel TE, eps_r 5, wavelength 0.02)
    s = timed(lambda: drt.field(w, t, r, sc.max_order, sc.alpha, "hard_sigmoid", 0.02, 5.0))
    out["coherent_field_hard_evals_per_s"] = ev / s
    s = timed(lambda: drt.field(w, t, r, sc.max_order, sc.alpha, "sigmoid", 0.02, 5.0))
    out["coherent_field_sigmoid_evals_per_s"] = ev / s
    g = scenes.gradient_scene()
    gw, gt, gr = (torch.tensor(g.walls, device=dev), torch.tensor(g.tx, device=dev),
                  torch.tensor(g.rx, device=dev))
    gp = torch.full((g.n_rx,), 1.0 / g.n_rx, device=dev)
    gc = workload.num_candidates(g.n_walls, g.max_order)
    sf = timed(lambda: drt.forward(gw, gt, gr, 2, 100.0, "hard_sigmoid"), 2)
    sv = timed(lambda: drt.vjp(gw, gt, gr, 2, 100.0, "hard_sigmoid", gp), 2)
    sfs = timed(lambda: drt.forward(gw, gt, gr, 2, 100.0, "sigmoid"), 1)
    svs = timed(lambda: drt.vjp(gw, gt, gr, 2, 100.0, "sigmoid", gp), 1)
    # the forward keeps every path's leg visibilities (N_K x 3 x R floats, 3.2 GB here)
    # and the adjoint reads them instead of its first wall sweep
    _, gsv = drt.forward_save(gw, gt, gr, 2, 100.0, "sigmoid")
    sfss = timed(lambda: drt.forward_save(gw, gt, gr, 2, 100.0, "sigmoid"), 1)
    svss = timed(lambda: drt.vjp(gw, gt, gr, 2, 100.0, "sigmoid", gp, saved=gsv), 1)
    del gsv
    # coherent field and its adjoint (lambda 0.02, eps_r 5) on the same scene
    fE, _ = drt.field(gw, gt, gr, 2, 100.0, "hard_sigmoid", 0.02, 5.0)
    ffh = timed(lambda: drt.field(gw, gt, gr, 2, 100.0, "hard_sigmoid", 0.02, 5.0), 2)
    fvh = timed(lambda: drt.field_vjp(gw, gt, gr, 2, 100.0, "hard_sigmoid", 0.02, 5.0, fE, gp), 2)
    fEs, _ = drt.field(gw, gt, gr, 2, 100.0, "sigmoid", 0.02, 5.0)
    fvs = timed(lambda: drt.field_vjp(gw, gt, gr, 2, 100.0, "sigmoid", 0.02, 5.0, fEs, gp), 1)
    # the same with the field forward's saved leg visibilities
    fEs2, _, fsv = drt.field_save(gw, gt, gr, 2, 100.0, "sigmoid", 0.02, 5.0)
    ffss = timed(lambda: drt.field_save(gw, gt, gr, 2, 100.0, "sigmoid", 0.02, 5.0), 1)
    fvss = timed(lambda: drt.field_vjp(gw, gt, gr, 2, 100.0, "sigmoid", 0.02, 5.0, fEs2, gp,
                                       saved=fsv), 1)
    del fsv
    # batched descent on the first 64 scenes of the 4096-scene batch (4 starts each)
    from paper_2401_11882_gb300.batched import BatchedDescent
    full = scenes.scene_batch(64, 0)
    bd = BatchedDescent(full, history=0)
    bd.run(1)
    torch.cuda.synchronize(dev)
    bs = timed(lambda: bd.run(1), 2)
    out["batched_descent_64_scenes"] = {
        "workload": "first 64 scenes of the 4096-scene batch (W 8-256, R 64-4096, K 0-2), 4 starts "
                    "each, alpha=100, hard sigmoid; one step = forward + argmin + adjoint + Adam",
        "ms_per_step": bs * 1e3, "steps_per_s": 1.0 / bs}
    # batched descent on 3D rooms (Sec. VI): 64 rooms of 16-72 triangles, R 16-512,
    # K 0-2, 4 starts each, alpha 100, hard sigmoid
    full3 = scenes.scene_batch3(64, 0)
    bd3 = BatchedDescent(full3, history=0, box=(0.02, 0.02, 0.02, 0.98, 0.98, 0.98))
    bd3.run(1)
    torch.cuda.synchronize(dev)
    bs3 = timed(lambda: bd3.run(1), 3)
    ev3 = sum(full3.tx0.shape[1] * int(full3.rx_off[i + 1] - full3.rx_off[i]) *
              workload.num_candidates(int(full3.wall_off[i + 1] - full3.wall_off[i]),
                                      int(full3.max_order[i])) for i in range(full3.n_scenes))
    out["batched_descent_3d_64_rooms"] = {
        "workload": "64 rooms (square + 2-30 segments extruded, floor, ceiling: 16-72 "
                    "triangles), R 16-512, K 0-2, 4 starts each, alpha=100, hard sigmoid; one "
                    "step = forward + argmin + adjoint + Adam",
        "ms_per_step": bs3 * 1e3, "steps_per_s": 1.0 / bs3, "evals_per_s": ev3 / bs3}
    bd3.close()
    bd.close()
    # surrogate MLP (tcgen05 path), batch 8192
    from paper_2401_11882_gb300.surrogate import SurrogateMLP
    m = SurrogateMLP(dev, batch=8192)
    xm = torch.rand(8192, 2, device=dev)
    tm = torch.randn(8192, device=dev)
    mf = timed(lambda: m.forward(xm), 20)
    mb = timed(lambda: m.loss_grad(xm, tm), 20)
    mlp_flops = 2 * 8192 * (64 * 256 + 3 * 256 * 256 + 256)
    out["surrogate_mlp_batch_8192"] = {"forward_ms": mf * 1e3, "loss_grad_ms": mb * 1e3,
                                       "forward_tflops": mlp_flops / mf / 1e12}
    # inference on the 512 x 512 proposal grid: the fused tcgen05 kernel
    mg = SurrogateMLP(dev, batch=512 * 512)
    xg = torch.rand(512 * 512, 2, device=dev)
    mgf = timed(lambda: mg.forward(xg), 20)
    pk_bf16 = float(peaks().get("bf16_tflops") or 1899.4)
    gfl = 2 * 512 * 512 * (64 * 256 + 3 * 256 * 256 + 256)
    out["surrogate_mlp_inference_512x512"] = {
        "kernel": "tc_mlp_forward_kernel (fused, tcgen05)", "forward_ms": mgf * 1e3,
        "tflops": gfl / mgf / 1e12, "frac_of_measured_bf16_peak": gfl / mgf / 1e12 / pk_bf16}
    out["gradient_scene_dense"] = {
        "workload": "128 random segments, 128x128 RX grid, K<=2 (16385 sequences), alpha=100, "
                    "hard sigmoid, dense g = 1/R, grad wrt TX and 512 wall coordinates",
        "fwd_ms": sf * 1e3, "vjp_ms": sv * 1e3,
        "fwd_plus_adjoint_evals_per_s": g.n_rx * gc / (sf + sv),
        "sigmoid": {"fwd_ms": sfs * 1e3, "vjp_ms": svs * 1e3,
                    "fwd_plus_adjoint_evals_per_s": g.n_rx * gc / (sfs + svs),
                    "saved_visibilities": {"fwd_save_ms": sfss * 1e3, "vjp_saved_ms": svss * 1e3,
                                           "fwd_plus_adjoint_evals_per_s":
                                               g.n_rx * gc / (sfss + svss)}},
        "coherent_field": {"wavelength": 0.02, "eps_r": 5.0, "hard_fwd_ms": ffh * 1e3,
                           "hard_vjp_ms": fvh * 1e3, "sigmoid_vjp_ms": fvs * 1e3,
                           "sigmoid_saved_visibilities": {"fwd_save_ms": ffss * 1e3,
                                                          "vjp_saved_ms": fvss * 1e3}}}
    return out


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=30)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-extras", action="store_true")
    ap.add_argument("--rx-grid", type=int, default=256,
                    help="receiver grid side (256 = the benchmark workload; smaller for profiling)")
    ap.add_argument("--smoothing", default="hard_sigmoid",
                    choices=["hard_sigmoid", "sigmoid", "step"],
                    help="smoothing of the timed step (hard_sigmoid = the benchmark workload)")
    ap.add_argument("--alpha", type=float, default=100.0)
    args = ap.parse_args()
    if args.impl == "reference":
        return run_reference(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
