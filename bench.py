#!/usr/bin/env python
"""Throughput of the natively periodic FMM solve on GB300.

One step = one full solve (mean removal, P2M, M2M, M2L at every level, L2L,
L2P and the near-zone sum) of a seeded synthetic 256^3 density field,
order p = 6, with the input already resident in HBM.  The timed form is the
mixed-precision one (tensor-core M2L at levels >= 4); the plain FP32
form is timed on the same field in the same run, and the result's error
against PM is stated twice: by the library (fmm_plan_error_stats, exact at
256 sampled cells) and, with the CPU baseline, over every cell by the FP64
oracle's FFT PM.  Prints ONE JSON line.

    python bench.py [--gpus N --steps K --warmup W] [--impl ours|reference]
                    [--n 256 --L 5 --p 6 --precision fp32|bf16|bf16x3]

Under torchrun (N > 1) every rank solves its own field (independent replicas,
no communication); the value is the cells of all ranks over the slowest rank's
time.  ``--impl reference`` times the FP64 CPU oracle instead (rank 0 only).
"""
import argparse
import json

import numpy as np
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "FMM cells/s at 256^3 p=6: mixed-prec+learned vs plain FP32, L2 err ≤1e-4 vs PM"
# weights of the learned M2L table correction trained by
# `python -m paper_2011_07099_gb300.learn` (order 6, 64^3 training fields)
DEFAULT_CORRECTION = os.path.join(os.path.dirname(os.path.abspath(__file__)), "paper_2011_07099_gb300", "data",
                                  "correction_p6.npz")
UNIT = "cells/s"
FP32_FMA_PER_SM_PER_CLK = 128        # FP32 lanes per SM (4 partitions x 32)
SM_MAX_MHZ = 2070.0                  # used only when neither nvidia-smi nor MEASURED_PEAKS.json gives it


def _peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return json.load(f), "measured"
    except OSError:
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0,
                "sm_max_mhz": SM_MAX_MHZ}, "fallback"


class ClockSampler:
    """nvidia-smi samples of SM clock and throttle reasons during the timed region."""
    Q = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.lines = []

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except OSError:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def __exit__(self, *a):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self):
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            f = [x.strip() for x in ln.split(",")]
            if len(f) < 8:
                continue
            try:
                sm.append(float(f[0]))
                mx.append(float(f[1]))
            except ValueError:
                continue
            for name, v in zip(names, f[4:8]):
                if v.lower().startswith("active"):
                    reasons.add(name)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "samples": len(sm),
                "reasons": sorted(reasons)}


def _dist():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def slowest_rank_ms(ms, ws, device=None):
    """The step time of the whole job: the maximum over the ranks (one
    independent field per rank, no data-path collective; this all-reduce
    only aggregates the timing)."""
    if ws <= 1:
        return ms
    import torch
    import torch.distributed as dist
    t = torch.tensor([ms], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def whole_job_cells_per_s(ws, n, ms):
    """Cells of all ranks over the slowest rank's step time (weak scaling)."""
    return ws * n ** 3 / (ms / 1000.0)


def workload_density(n, field):
    from paper_2011_07099_gb300 import inputs
    # the headline workload: 1 + 0.5 lognormal(sigma = 0.5), k^-2 Gaussian field,
    # seeded per rank
    return inputs.lognormal(n, sigma=0.5, seed=5000 + field)


# DRAM bytes of the leaf stage and of the leaf level's M2L are not captured in
# this run; the spectra each writes and reads back once are stated instead
def measure_fp32_peak(B, dev, stream, reps=40):
    """The FP32 CUDA-core peak of this device, measured: the library's FMA
    probe (dependent FMA chains only, 2 CTAs of 1024 threads per SM), each
    launch timed with CUDA events on the launching stream, median of `reps`
    launches after 3 warm-ups; SM clocks are sampled meanwhile."""
    import torch
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    blocks, iters = 2 * sms, 20000
    out = torch.empty(blocks, dtype=torch.float32, device=dev)
    for _ in range(3):
        flops = B.fmm_probe_fma(out, blocks, iters, stream)
    torch.cuda.synchronize(dev)
    ms = []
    with ClockSampler(dev.index) as clk:
        for _ in range(reps):
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            B.fmm_probe_fma(out, blocks, iters, stream)
            e1.record(stream)
            e1.synchronize()
            ms.append(e0.elapsed_time(e1))
    med = statistics.median(ms)
    c = clk.summary() or {}
    max_mhz = c.get("sm_max_mhz") or SM_MAX_MHZ
    derived = sms * FP32_FMA_PER_SM_PER_CLK * 2 * max_mhz * 1e6 / 1e12
    return {"tflops": flops / (med / 1e3) / 1e12, "launch_ms": med, "sm_count": sms,
            "sm_mhz_median": c.get("sm_mhz"), "sm_max_mhz": max_mhz, "clock_reasons": c.get("reasons"),
            "derived_at_max_clock_tflops": derived,
            "how": f"fmm_probe_fma: {blocks} CTAs x 1024 threads x 8 FMA chains x {iters} x 16, CUDA events, "
                   f"median of {reps}"}


def near_flops(N, L, fields=4):
    """Arithmetic the near zone by spectral products executes per solve: with
    leaves of S cells, transforms on (2S - 1)^3 points of which NK =
    (2S - 1)^2 S frequencies are kept.  Sums: per leaf and frequency the leaf's
    own kernel and 13 pairs of opposite offsets, whose kernels are conjugate.
    Lines of the forward transform of the masses and of the four inverse ones
    to the S^3 cells: the symmetric halves of a line share their sums."""
    S = N >> L
    M, h = 2 * S - 1, S - 1
    mac = M * M * S * (13 * (4 + 8 * fields) + 6 * fields)
    line_real, line_fwd = h + 4 * h * h, 2 * h + h * (8 * h + 4)
    line_inv, line_cells = 6 * h + h * (8 * h + 2), S * (4 * h + 2)
    fwd = S * S * line_real + S * S * line_fwd + M * S * line_fwd          # x, y, z passes
    inv = M * S * line_inv + S * S * line_inv + S * S * line_cells
    return float(8 ** L * (mac + fwd + fields * inv))


def near_bytes(N, L, fields=4):
    """Source spectra and the fields' target spectra, each written and read once (FP32 complex)."""
    S = N >> L
    return 8.0 ** L * 2 * (1 + fields) * 8 * (2 * S - 1) ** 2 * S


def m2l_spectral_flops(lev, p, fields=4):
    """The spectral sums of one M2L level: per node and frequency 189 (level 2:
    37) offsets x 4 fields, 8 flop per complex multiply-add."""
    return 8.0 ** lev * (37 if lev == 2 else 189) * fields * 8 * (2 * p - 1) ** 2 * p


def m2l_tensor_flops(lev, p):
    """The tensor-core form executes, per frequency and parent, 27 x 16 x 128
    multiply-adds on both FP16 parts of the sources."""
    return 8.0 ** (lev - 1) * (2 * p - 1) ** 2 * p * 2 * 2.0 * 27 * 16 * 128


def cpu_baseline():
    """The FP64 oracle, as it stands, on the host cores: full solve of a 64^3
    lognormal field with the same order (p = 6) and leaf size (S = 8, L = 3),
    whose per-cell arithmetic matches the 256^3 p = 6 L = 5 workload within a
    few percent."""
    import numpy as np  # noqa: F401
    from oracle import fmm as ofmm
    rho = workload_density(64, 0)
    t, c = time.perf_counter(), time.process_time()
    ofmm.solve(rho, 3, 6)
    dt, cpu = time.perf_counter() - t, time.process_time() - c
    return {"value": 64 ** 3 / dt, "unit": UNIT, "cores": effective_cores(cpu, dt), "kind": "oracle",
            "cores_available": os.cpu_count(), "seconds": dt,
            "sample": "full oracle solve of a 64^3 lognormal field, p=6, L=3 (S=8), numpy FP64 on the host cores"}


def effective_cores(cpu_seconds, wall_seconds):
    """Threads the oracle kept busy on average: process CPU time over wall
    time (numpy's BLAS decides how many it starts)."""
    return round(cpu_seconds / wall_seconds, 1) if wall_seconds > 0 else 0.0


def pm_references(rho):
    """Part of the oracle leg: PM with the same Green's function (FFT
    convolution, FP64 host) and, secondary, the spectral PM with G_K."""
    import numpy as np
    from oracle import green, pm
    n = rho.shape[0]
    m = pm.masses(rho.astype(np.float64))
    return pm.pm(m, green.g_s1, green.grad_g_s1, green.self_term(n)), pm.pm_gk(m)


def accuracy_vs_pm(refs, phi, acc):
    """Relative L2 over all cells of a result against PM(G_S1) (primary: the
    same G in PM and FMM) and PM(G_K) (secondary)."""
    import numpy as np
    (pphi, pg), (kphi, kg) = refs
    rel = lambda a, b: float(np.linalg.norm(a.astype(np.float64) - b) / np.linalg.norm(b))
    return {"vs_pm_gs1": {"phi": rel(phi, pphi), "g": rel(acc, pg)},
            "vs_pm_gk": {"phi": rel(phi - phi.mean(), kphi - kphi.mean()), "g": rel(acc, kg)},
            "note": "relative L2 over all cells; PM(G_S1) is the primary reference (same G in PM and FMM)"}


def learned_correction(args):
    """The learned table correction the headline workload applies: the
    shipped order-6 weights (or --correction) in the tensor-core forms,
    None otherwise.  The weights file path is under "path"."""
    wpath = args.correction or (DEFAULT_CORRECTION if args.p == 6 else None)
    if args.precision == "fp32" or args.no_correction or not wpath or not os.path.exists(wpath):
        return None
    here = os.path.dirname(os.path.abspath(__file__))
    return {"path": wpath, "weights": os.path.relpath(wpath, here), "inference": "bf16",
            "applied_to": "M2L tables, levels 2..L"}


def near_fft_used(args):
    """The near zone's FP32 transforms (--near fft) are the form of 8-cell leaves."""
    return args.near == "fft" and (args.n >> args.L) == 8


def headline_config(args, learned, ws):
    """The `config` object of the headline workload; both arms print it."""
    n, L, p = args.n, args.L, args.p
    near = ("near zone by FFT on the doubled grid" if near_fft_used(args)
            else "near zone at the direct sum's accuracy")
    return {"workload": f"{n}^3 lognormal sigma=0.5 (seeded), order p={p}, L={L} (S={n >> L}), "
                        f"M2L levels>=4 {args.precision}, levels 2-3 extended-precision CUDA-core, {near}"
                        + (", learned table correction" if learned else ""),
            "N": n, "L": L, "order": p, "precision": args.precision, "near_zone": args.near if near_fft_used(args)
            else "direct",
            "learned_correction": None if learned is None else {k: v for k, v in learned.items() if k != "path"},
            "l2_flush": "256 MB buffer written between timed steps",
            "parallelism": f"replicas x{ws}"}


def run_reference(args):
    ws, rank, _ = _dist()
    if rank != 0:
        return 0
    from oracle import fmm as ofmm
    n, L, p = 64, 3, 6            # the cpu_baseline sample: levels 2 and 3, M2M and L2L, S = 8
    rho = workload_density(64, 0)
    for _ in range(args.warmup):
        ofmm.solve(rho, L, p)
    times = []
    c = time.process_time()
    for _ in range(args.steps):
        t = time.perf_counter()
        ofmm.solve(rho, L, p)
        times.append(time.perf_counter() - t)
    cores = effective_cores(time.process_time() - c, sum(times))
    ms = 1000.0 * statistics.mean(times)
    value = n ** 3 / (ms / 1000.0)
    sample = (f"FP64 numpy oracle (plain method, no correction), full solve of a {n}^3 lognormal sigma=0.5 "
              f"field per step with order p={p} and the workload's leaf size S=8 (L={L}); cells/s of the "
              f"sample stand for the {args.n}^3 workload")
    line = {"impl": "reference", "method": "the plain method in FP64 (CPU oracle): no tensor cores, no "
                                          "mixed precision, no learned correction",
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": headline_config(args, learned_correction(args), ws),
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "cores_available": os.cpu_count(),
                             "kind": "oracle", "sample": sample},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
            "gpu_launches": 0}
    print(json.dumps(line), flush=True)
    return 0


def _time_solves(B, plan, rho, phi, acc, steps, warmup, l2_flush, stream, barrier, timing=True):
    """W untimed solves, then `steps` solves each bracketed by CUDA events on
    the launching stream, with an L2 flush (256 MB write) between them.  The
    timed solves run as a user's do (the library overlaps independent stages
    on its own streams); the per-stage times come from two more solves with
    the library's stage timing on (which runs the stages one after another),
    outside the timed region.  Returns (per-step ms list, per-stage-time
    lists, wall seconds)."""
    import torch
    for _ in range(warmup):
        plan.solve(rho, phi, acc)
    torch.cuda.synchronize()
    step_ms, stage = [], []
    barrier()
    torch.cuda.synchronize()
    wall0 = time.perf_counter()
    for _ in range(steps):
        l2_flush.zero_()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        plan.solve(rho, phi, acc)
        e1.record(stream)
        e1.synchronize()
        step_ms.append(e0.elapsed_time(e1))
    torch.cuda.synchronize()
    barrier()
    wall = time.perf_counter() - wall0
    if timing:
        B.fmm_plan_set_timing(plan.handle, True)
        for _ in range(2):
            l2_flush.zero_()
            plan.solve(rho, phi, acc)
            stage.append(B.fmm_plan_stage_times(plan.handle))
        B.fmm_plan_set_timing(plan.handle, False)
    return step_ms, stage, wall


def device_check(B, plan):
    """fmm_plan_check after a loop of solves: "ok", or the error it reports
    (a bounded device wait that ran out makes those results invalid)."""
    rc = B.lib().fmm_plan_check(plan.handle)
    return "ok" if rc == B.FMM_OK else B.lib().fmm_error_string(rc).decode()


def launches_per_solve(L, tc, p=6, near_fft=False):
    # the library's dense forms (spectra limit 0; M2L by dense sums, the near zone by pairs): mean
    # (2) + P2M + M2M per level + M2L per level + L2L per level + near zone (1;
    # by FFT 4); M2L of the coarse levels (2-3, and every level above the leaves
    # at order >= 7) adds the range sums, tensor-core levels the split
    wide = lambda lev: lev <= 3 or (p >= 7 and lev < L)
    tc_first = max(4, L) if p >= 7 else 4
    m2l = sum(2 if (wide(lev) or (tc and lev >= tc_first)) else 1 for lev in range(2, L + 1))
    return 2 + 1 + (L - 2) + m2l + (L - 2) + (4 if near_fft else 1)


def launches_of_forms(forms, p, S):
    """Kernels an untimed periodic solve launches in the forms its plan runs
    (fmm_plan_get_forms: [0] the near zone, [l] the M2L of level l), for the
    case that the profiler counts none (profiled_launches): mean (2), P2M, M2M
    and L2L per level, near zone (spectral: source spectra, sums, inverse) and
    M2L: the spectral levels of one arithmetic share three launches, spectral
    tensor-core levels take four each (scale, spectra, products, inverse),
    dense ones one and their split or range sums."""
    from paper_2011_07099_gb300 import binding as B
    L = len(forms) - 1
    wide = lambda lev: lev <= 3 or (p >= 7 and lev < L) or S >= 16
    spectral = {wide(lev) for lev in range(2, L + 1) if forms[lev] == B.FMM_FORM_SPECTRAL}
    each = {B.FMM_FORM_SPECTRAL_TC: 4, B.FMM_FORM_DENSE_TC: 2}
    m2l = 3 * len(spectral) + sum(each.get(forms[lev], 2 if wide(lev) else 1) for lev in range(2, L + 1)
                                  if forms[lev] != B.FMM_FORM_SPECTRAL)
    return 2 + 1 + 2 * (L - 2) + m2l + (3 if forms[0] == B.FMM_FORM_SPECTRAL else 1)


def profiled_launches(solve):
    """Kernels of this library in one call of `solve`, as the CUDA profiler
    lists them (all are named fmm::...::k_*; copies and fills do not count).
    The first profile of a process may see nothing, so two are taken."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    n = 0
    for _ in range(2):
        try:
            with profile(activities=[ProfilerActivity.CUDA]) as prof:
                solve()
                torch.cuda.synchronize()
            n = sum(1 for e in prof.events() if "fmm::" in e.name and "k_" in e.name)
        except RuntimeError:   # another profiler holds the device: no count
            n = 0
    return n


def solve_roofline(n, L, p, tc, ms, peaks, fp32_tflops):
    """Ideal time of the whole solve, each step at its own bound (FP32 FMA,
    FP16 tensor at the BF16 rate, HBM bytes), against the measured step.  The
    near zone and each M2L level take the larger of their arithmetic and of
    their spectra's one round trip through HBM."""
    fp32 = fp32_tflops * 1e12
    f16 = peaks.get("bf16_tflops_sustained", 1700.0) * 1e12
    hbm = peaks.get("hbm_gbs", 6500.0) * 1e9
    p3 = p ** 3
    tc_first = max(4, L) if p >= 7 else 4
    t = {"near": max(near_flops(n, L) / fp32, near_bytes(n, L) / hbm), "m2l_cuda_cores": 0.0, "m2l_tensor": 0.0}
    for lev in range(2, L + 1):
        spectra = 8.0 ** lev * 2 * 5 * 8 * (2 * p - 1) ** 2 * p / hbm
        if tc and lev >= tc_first:
            t["m2l_tensor"] += max(m2l_tensor_flops(lev, p) / f16, spectra)
        else:
            t["m2l_cuda_cores"] += max(m2l_spectral_flops(lev, p) / fp32, spectra)
    bytes_ = 4 * n ** 3 * 2 + 4 * p3 * 8 ** L + 16 * n ** 3                # mean + P2M + the outputs
    bytes_ += sum(9 * 4 * p3 * 8 ** lev for lev in range(2, L))          # M2M
    bytes_ += sum(4 * 4 * p3 * 8 ** lev * 17 for lev in range(2, L))     # L2L (parent + children read/write)
    t["hbm_passes"] = bytes_ / hbm
    ideal = sum(t.values()) * 1e3
    return {"ideal_ms": ideal, "measured_ms": ms, "frac": ideal / ms,
            "terms_ms": {k: v * 1e3 for k, v in t.items()},
            "peaks": f"FP32 {fp32_tflops:.1f} TFLOP/s (measured, fmm_probe_fma), BF16 sustained and HBM from "
                     "MEASURED_PEAKS.json"}


def run_ours(args):
    import numpy as np
    import torch
    from paper_2011_07099_gb300 import binding, build

    ws, rank, local = _dist()
    if ws > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl")
    else:
        torch.cuda.set_device(0)
    dev = torch.device("cuda", torch.cuda.current_device())
    build.build()
    B = binding
    n, L, p = args.n, args.L, args.p
    prec = {"fp32": B.FMM_PREC_FP32, "bf16": B.FMM_PREC_BF16, "bf16x3": B.FMM_PREC_BF16X3}[args.precision]
    tc = prec != B.FMM_PREC_FP32

    def barrier():
        if ws > 1:
            import torch.distributed as dist
            dist.barrier()

    rho_host = workload_density(n, rank)
    rho = torch.from_numpy(rho_host).to(dev)
    phi = torch.empty((n, n, n), dtype=torch.float32, device=dev)
    acc = torch.empty((3, n, n, n), dtype=torch.float32, device=dev)
    l2_flush = torch.empty(64 * 1024 * 1024, dtype=torch.float32, device=dev)   # 256 MB > L2
    stream = torch.cuda.current_stream(dev)

    plan = B.Plan(n, L, p)
    if tc:
        plan.set_precision(prec)
    learned = learned_correction(args)
    if learned is not None:
        w = torch.from_numpy(np.load(learned["path"])["w"].astype(np.float32)).to(dev)
        B.fmm_plan_set_correction(plan.handle, w)   # tabulated once at plan time; BF16 inference
    near_fft = near_fft_used(args)
    if near_fft:
        B.fmm_plan_set_near_algorithm(plan.handle, B.FMM_NEAR_FFT)
    # the tile of each level on the dense tensor-core contraction, autotuned at
    # plan time (outside the timed region); none where all run spectral products
    tc_tiles = B.fmm_plan_autotune_tiles(plan.handle, rho)[:L + 1] if tc else None
    m2l_forms, _ = B.fmm_plan_get_forms(plan.handle)
    if tc:
        tc_tiles = [t if f == B.FMM_FORM_DENSE_TC else 0 for t, f in zip(tc_tiles, m2l_forms)]
    with ClockSampler(dev.index) as clk:
        step_ms, stage, wall = _time_solves(B, plan, rho, phi, acc, args.steps, args.warmup, l2_flush, stream,
                                            barrier)
    checks = {"timed_solves": device_check(B, plan)}
    ms = slowest_rank_ms(statistics.mean(step_ms), ws, dev)
    value = whole_job_cells_per_s(ws, n, ms)
    host_leg = rank == 0 and ws == 1 and not args.no_cpu_baseline
    result_phi = phi.cpu().numpy() if host_leg else None
    result_acc = acc.cpu().numpy() if host_leg else None
    # the library's own statement of this result's error against PM with
    # G_S1, measured exactly at sampled cells (outside the timed region)
    stmt_cells = 256

    def statement_of(pl, ph, ac):
        try:
            e_phi, e_g = pl.error_stats(rho, ph, ac, samples=stmt_cells, seed=1)
            return {"vs_pm_gs1": {"phi": e_phi, "g": e_g}, "cells": stmt_cells,
                    "source": "fmm_plan_error_stats (exact direct sum at sampled cells, GPU)"}
        except B.FMMError as e:   # reported in the line; the timed numbers stand
            return {"failed": str(e)}

    statement = statement_of(plan, phi, acc)
    checks["error_statement"] = device_check(B, plan)

    # what the learned correction gains on the timed field: the same form
    # without the correction, solved once (outside the timed region)
    gain = None
    if learned is not None:
        nplan = B.Plan(n, L, p)
        if tc:
            nplan.set_precision(prec)
        if near_fft:
            B.fmm_plan_set_near_algorithm(nplan.handle, B.FMM_NEAR_FFT)
        nphi = torch.empty_like(phi)
        nacc = torch.empty_like(acc)
        nplan.solve(rho, nphi, nacc)
        torch.cuda.synchronize(dev)
        checks["without_correction"] = device_check(B, nplan)
        gain = {"with_correction": statement.get("vs_pm_gs1"),
                "without_correction": statement_of(nplan, nphi, nacc).get("vs_pm_gs1"),
                "measured_by": f"fmm_plan_error_stats, {stmt_cells} cells (seed 1), same cells for both"}
        if host_leg:
            gain["without_correction_host_pm"] = ("pending", nphi.cpu().numpy(), nacc.cpu().numpy())
        nplan.close()
        del nphi, nacc

    # per-stage means over the timed steps
    nslot = len(stage[0])
    st = [statistics.mean(s[i] for s in stage) for i in range(nslot)]
    names = ["mean", "p2m", "m2m", "m2l", "l2l", "p2p_l2p"]
    stage_ms = {names[i]: st[i] for i in range(6)}
    for lev in range(2, L + 1):
        stage_ms[f"m2l_level{lev}"] = st[B.FMM_TIME_M2L_LEVEL0 + lev]

    # the plain FP32 form on the same field, same run (the comparison the metric
    # names: FP32 M2L, near zone by direct sum), and the two forms between it
    # and the headline (one change each), so the speed-up can be split up
    def time_form(form_prec, form_fft, form_learned):
        fplan = B.Plan(n, L, p)
        if form_prec != B.FMM_PREC_FP32:
            fplan.set_precision(form_prec)
        if form_learned is not None:
            B.fmm_plan_set_correction(fplan.handle, w)
        if form_fft:
            B.fmm_plan_set_near_algorithm(fplan.handle, B.FMM_NEAR_FFT)
        fms, fstage, _ = _time_solves(B, fplan, rho, phi, acc, max(1, min(args.steps, 3)),
                                      max(1, min(args.warmup, 2)), l2_flush, stream, barrier)
        fm = slowest_rank_ms(statistics.mean(fms), ws, dev)
        res = {"value": whole_job_cells_per_s(ws, n, fm), "ms_per_step": fm,
               "m2l_ms": statistics.mean(s_[B.FMM_TIME_M2L] for s_ in fstage),
               "p2p_ms": statistics.mean(s_[B.FMM_TIME_P2P] for s_ in fstage),
               "device_check": device_check(B, fplan)}
        fplan.close()
        return res

    plain = None
    forms = {}
    if tc and not args.no_plain:
        plain = time_form(B.FMM_PREC_FP32, False, None)
        checks["plain_fp32"] = plain.pop("device_check")
        if near_fft:
            forms["plain_fp32_near_fft"] = time_form(B.FMM_PREC_FP32, True, None)
            forms["mixed_near_direct"] = time_form(prec, False, learned)
        # phi/acc now hold the last form's result: the timed result was
        # copied to the host (host leg) and measured (error statement) above

    peaks, src = _peaks()
    fma = measure_fp32_peak(B, dev, stream)
    fp32_peak = fma["tflops"]
    near_s = stage_ms["p2p_l2p"] / 1000.0
    near_ach = near_flops(n, L) / near_s / 1e12
    roof_near = {"kernel": "k_ns_fwd + k_ns_mac + k_ns_inv (near zone by spectral products and L2P; the whole stage)",
                 "bound": "alu", "achieved": near_ach, "peak": fp32_peak, "unit": "TFLOP/s",
                 "frac": near_ach / fp32_peak, "traffic": None, "spectra_bytes": near_bytes(n, L),
                 "hbm_frac": near_bytes(n, L) / near_s / (peaks.get("hbm_gbs", 6500.0) * 1e9),
                 "peak_source": "measured (of measured): " + fma["how"], "fp32_probe": fma}
    roof_m2l = None
    if tc:
        tc_ms = stage_ms[f"m2l_level{L}"]
        ach = m2l_tensor_flops(L, p) / (tc_ms / 1000.0) / 1e12
        peak = peaks.get("bf16_tflops_sustained", 1700.0)
        roof_m2l = {"kernel": f"k_stc_amax + k_stc_fwd + k_stc_mac + k_stc_inv (level {L}, the whole level)",
                    "bound": "hbm/latency", "achieved": ach, "peak": peak, "unit": "TFLOP/s", "frac": ach / peak,
                    "traffic": None,
                    "peak_source": f"bf16_tflops_sustained ({src}, of measured); achieved counts the executed FP16 "
                                   "products of the spectral sums over the level's transforms and sums together"}
    roof = roof_near if (roof_m2l is None or stage_ms["p2p_l2p"] >= stage_ms[f"m2l_level{L}"]) else roof_m2l

    # end to end through the public host-buffer entry point
    hin = torch.from_numpy(rho_host).pin_memory()
    hphi = torch.empty((n, n, n), dtype=torch.float32).pin_memory()
    hacc = torch.empty((3, n, n, n), dtype=torch.float32).pin_memory()
    B.fmm_solve_host(plan.handle, hin, hphi, hacc, stream)
    e2e_steps = max(1, min(args.steps, 5))
    t0 = time.perf_counter()
    for _ in range(e2e_steps):
        B.fmm_solve_host(plan.handle, hin, hphi, hacc, stream)
    e2e_s = (time.perf_counter() - t0) / e2e_steps
    checks["e2e"] = device_check(B, plan)
    launches = (profiled_launches(lambda: plan.solve(rho, phi, acc)) if rank == 0 else 0) or launches_of_forms(
        m2l_forms, p, n >> L)
    plan.close()

    if rank != 0:
        if ws > 1:
            import torch.distributed as dist
            dist.destroy_process_group()
        return 0
    clocks = clk.summary()
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f32" if not tc else ("bf16x3" if prec == B.FMM_PREC_BF16X3 else "bf16"),
        "data": "synthetic",
        "config": dict(headline_config(args, learned, ws), tc_tiles=tc_tiles),
        "stage_ms": stage_ms,
        "stage_ms_source": "two solves with the library's stage timing on, which runs the stages one after another; "
                           "the timed steps overlap the near zone's transform and sums with the tree passes and the "
                           "coarse M2L levels with the tensor-core ones",
        "wall_s": wall,
        "roofline": roof,
        "roofline_near": roof_near,
        "roofline_m2l": roof_m2l,
        "e2e": {"value": ws * n ** 3 / e2e_s, "unit": UNIT, "h2d_bytes_per_step": 4 * n ** 3,
                "d2h_bytes_per_step": 16 * n ** 3},
        "gpu_launches": launches * args.steps,
        "solve_roofline": solve_roofline(n, L, p, tc, ms, peaks, fp32_peak),
        "clocks": clocks,
        "error_statement": statement,
        "device_checks": checks,
    }
    if plain is not None:
        line["plain_fp32"] = plain
        line["speedup_vs_plain_fp32"] = plain["ms_per_step"] / ms
    if forms:
        line["forms"] = forms
    if host_leg:
        line["cpu_baseline"] = cpu_baseline()
        refs = pm_references(rho_host)
        line["accuracy"] = accuracy_vs_pm(refs, result_phi, result_acc)
        if gain is not None:
            _, gphi, gacc = gain.pop("without_correction_host_pm")
            gain["whole_mesh"] = {"with_correction": line["accuracy"],
                                  "without_correction": accuracy_vs_pm(refs, gphi, gacc)}
    if gain is not None:
        line["learned_gain"] = gain
    print(json.dumps(line), flush=True)
    return 0


def run_batch(args):
    """The batching workload: 64 independent periodic fields with N drawn from
    {32, 48, 64, 96, 128}, order 4 or 6, lognormal sigma in [0.3, 1.5]
    (seeded), leaf levels autotuned, solved as one CUDA-graph launch."""
    import torch
    from paper_2011_07099_gb300 import binding as B, build, inputs
    torch.cuda.set_device(0)
    build.build()
    rng = np.random.Generator(np.random.PCG64(2000))
    nf = args.fields
    Ns = [int(x) for x in rng.choice([32, 48, 64, 96, 128], nf)]
    ps = [int(x) for x in rng.choice([4, 6], nf)]
    sig = rng.uniform(0.3, 1.5, nf)
    import tempfile
    os.environ.setdefault("FMM_AUTOTUNE_CACHE", os.path.join(tempfile.gettempdir(), "fmm_autotune.jsonl"))
    t0 = time.perf_counter()
    # with the near zone by FFT the fields whose N is 8 x a power of two take
    # 8-cell leaves (its leaf size); the others are autotuned (L = 0)
    near_fft = args.near == "fft"
    Ls = [(n // 8).bit_length() - 1 if near_fft and n % 8 == 0 and (n // 8) & (n // 8 - 1) == 0 and n >= 32 else 0
          for n in Ns]
    batch = B.Batch(Ns, Ls, ps, precision=B.FMM_PREC_BF16X3)
    if near_fft:
        B.fmm_batch_set_near_algorithm(batch.handle, B.FMM_NEAR_FFT)
    tune_s = time.perf_counter() - t0
    d = [torch.from_numpy(inputs.lognormal(n, sigma=float(s_), seed=2000 + i)).cuda() for i, (n, s_) in
         enumerate(zip(Ns, sig))]
    pots = [torch.empty((n, n, n), device="cuda") for n in Ns]
    accs = [torch.empty((3, n, n, n), device="cuda") for n in Ns]
    stream = torch.cuda.current_stream()
    for _ in range(args.warmup):
        batch.solve(d, pots, accs)
    torch.cuda.synchronize()
    l2_flush = torch.empty(64 * 1024 * 1024, dtype=torch.float32, device="cuda")
    times = []
    with ClockSampler(0) as clk:
        for _ in range(args.steps):
            l2_flush.zero_()
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            batch.solve(d, pots, accs)
            e1.record(stream)
            e1.synchronize()
            times.append(e0.elapsed_time(e1))
    batch.check()
    ms = statistics.mean(times)
    cells = sum(n ** 3 for n in Ns)
    line = {"metric": "FMM cells/s, batch of 64 uneven periodic fields (one graph launch)", "value": cells / (ms / 1e3),
            "unit": UNIT, "n_gpus": 1, "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "bf16x3", "data": "synthetic",
            "config": {"workload": f"{nf} fields, N in {{32,48,64,96,128}}, p in {{4,6}}, lognormal sigma U[0.3,1.5]"
                                   + (", near zone by FFT where the leaves hold 8 cells" if near_fft else ""),
                       "cells": cells, "levels": batch.levels, "N": Ns, "order": ps, "autotune_s": tune_s},
            "clocks": clk.summary()}
    print(json.dumps(line), flush=True)
    batch.close()
    return 0


def run_full512(args):
    """The full-scale workload: 512^3 (134M cells), order 8, L = 6 (S = 8),
    density 1 + lognormal(sigma 1.5) plus 4096 Plummer clumps; the mixed form
    (tensor-core bf16x3 M2L) against the plain FP32 form, errors against PM
    with G_S1 (libfmm mesh Green's function + cuFFT)."""
    import torch
    from paper_2011_07099_gb300 import binding as B, build, inputs, learn
    torch.cuda.set_device(0)
    build.build()
    n, L, p = 512, 6, 8
    dev = torch.device("cuda", 0)
    rho = inputs.config_density_torch(4, dev)
    out = {}
    l2_flush = torch.empty(64 * 1024 * 1024, dtype=torch.float32, device=dev)
    stream = torch.cuda.current_stream(dev)
    tphi, tacc = learn.pm_target(rho, n)
    with ClockSampler(0) as clk:
        for name, prec in (("mixed_bf16x3", B.FMM_PREC_BF16X3), ("plain_fp32", B.FMM_PREC_FP32)):
            plan = B.Plan(n, L, p)
            if prec:
                plan.set_precision(prec)
            if prec != B.FMM_PREC_FP32 and args.near == "fft":
                B.fmm_plan_set_near_algorithm(plan.handle, B.FMM_NEAR_FFT)   # the plain form keeps the direct sum
            phi = torch.empty((n, n, n), device=dev)
            acc = torch.empty((3, n, n, n), device=dev)
            ms, stage, _ = _time_solves(B, plan, rho, phi, acc, args.steps, max(1, args.warmup), l2_flush, stream,
                                        lambda: None)
            e_phi = float(((phi.double() - tphi.double()) ** 2).sum().sqrt() / (tphi.double() ** 2).sum().sqrt())
            e_g = float(((acc.double() - tacc.double()) ** 2).sum().sqrt() / (tacc.double() ** 2).sum().sqrt())
            st = [statistics.mean(s_[i] for s_ in stage) for i in range(len(stage[0]))]
            out[name] = {"ms_per_step": statistics.mean(ms), "cells_per_s": n ** 3 / (statistics.mean(ms) / 1e3),
                         "m2l_ms": st[B.FMM_TIME_M2L], "p2p_ms": st[B.FMM_TIME_P2P],
                         "vs_pm_gs1": {"phi": e_phi, "g": e_g}, "device_check": device_check(B, plan)}
            plan.close()
            del phi, acc
    line = {"metric": "FMM cells/s at 512^3 p=8 (full scale)", "value": out["mixed_bf16x3"]["cells_per_s"],
            "unit": UNIT, "n_gpus": 1, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": out["mixed_bf16x3"]["ms_per_step"], "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "bf16x3", "data": "synthetic",
            "config": {"workload": "512^3, p=8, L=6 (S=8), 1 + lognormal(sigma=1.5) + 4096 Plummer clumps; mixed form: "
                                   "tensor-core leaf-level M2L, bf16x6 level 5 (FP64 fields), double-float levels 2-4"
                                   + (", near zone by FFT" if args.near == "fft" else ""),
                       "forms": out}, "clocks": clk.summary()}
    print(json.dumps(line), flush=True)
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--n", type=int, default=256)
    ap.add_argument("--L", type=int, default=5)
    ap.add_argument("--p", type=int, default=6)
    ap.add_argument("--precision", choices=["fp32", "bf16", "bf16x3"], default="bf16x3")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-plain", action="store_true", help="skip timing the plain FP32 form")
    ap.add_argument("--workload", choices=["headline", "batch", "full512"], default="headline")
    ap.add_argument("--fields", type=int, default=64)
    ap.add_argument("--correction", default=None,
                    help="weights (.npz with 'w') of the learned table correction for the mixed form; "
                         "default: the trained order-6 weights shipped with the package, when p = 6")
    ap.add_argument("--no-correction", action="store_true", help="time the mixed form without the correction")
    ap.add_argument("--near", choices=["fft", "direct"], default="fft",
                    help="near zone of the timed form: FFT convolution on the doubled grid (Sec. 3; 8-cell "
                         "leaves) or the direct sum; the plain FP32 form always uses the direct sum")
    args = ap.parse_args()
    if args.impl == "reference":
        return run_reference(args)
    if args.workload == "batch":
        return run_batch(args)
    if args.workload == "full512":
        return run_full512(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
