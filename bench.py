#!/usr/bin/env python
"""Throughput of the GB300 sphere-GMRF sampler on its largest single-GPU workload.

Workload (default): 16384 x 32768 equiangular grid, C_l = 1/(l(l+1)+300^2) (p = 1), 4
realisations per step, FP32 tables (set up once in FP64 on the device), FP32 recursion + FFT.
A step is one smerf_sample call: the anchor kernel and the segment kernel that synthesises and
writes every ring.  Metric: sphere grid points per second, with the segment kernel's fraction
of the HBM roofline (the method's algorithmic bytes) and of the ALU issue roofline.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl gb300|reference] [--workload W]

Prints one JSON line (rank 0).  The CPU baseline, and --impl reference, time the oracle's
per-sample recursion of Alg. 2 (FP64, plain C, tables from the oracle's own Gaussian
conditioning, a plain radix-2 FFT per ring) on a bounded sample of the same workload.
"""
import argparse
import json
import math
import os
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

DEFAULT_WORKLOAD = "16384x32768-p1"
METRIC = "sphere grid points/s"
FLUSH_BYTES = 256 << 20


SMS, FP32_LANES, FP64_PER_SM = 152, 128, 2     # GB300: SMs, FP32 lanes per SM, FP64 FMAs per SM per clock


def alg_ops_per_item(p, Nc, fp64=False):
    """Algorithmic ALU operations of one (mode, realisation, ring) item of the method (an FMA
    counts as one): Philox4x32-10 (10 rounds x 2 widening multiplies + 2 three-input XORs per
    call of 4 normals), Box-Muller (12 per pair: 2 conversions, 2 scalings, log2, scaling,
    rsqrt, product, sin, cos, 2 products), the recursion x = A x + B xi on the Re and Im
    chains (Eq. (state_space)), and this item's share of the ring's C2R FFT (10 for the
    packing, 3.5 log2 Nc for a radix-4 complex FFT).  With fp64 only the floating-point part
    (Box-Muller, recursion, FFT)."""
    philox = 40.0 * (2 * p) / 4.0
    box_muller = 12.0 * p
    recursion = 2.0 * (p * p + p * (p + 1) / 2.0)
    fft = 10.0 + 3.5 * math.log2(Nc)
    return (box_muller + recursion + fft) if fp64 else (philox + box_muller + recursion + fft)


def fp64_pipe_ops_per_item(p, Nc):
    """The operations of an item that the FP64 recursion mode leaves on the FP64 pipe: the
    recursion; the noise is formed in 64-bit fixed point on the integer lanes, and so is the FFT
    of rings up to 2048 complex points (the in-place kernel's longer rings keep FP64 FFTs)."""
    recursion = 2.0 * (p * p + p * (p + 1) / 2.0)
    return recursion + (10.0 + 3.5 * math.log2(Nc) if Nc > 2048 else 0.0)


def sfu_ops_per_item(p):
    """Special-function operations of one item: Box-Muller's log2, rsqrt, sin and cos per pair
    of normals (p pairs per item)."""
    return 4.0 * p


SFU_LANES = 16  # special-function (MUFU) lanes per SM per clock


def alg_table_bytes(p, n_theta, n_phi, fp64):
    """The method's table bytes per launch: A (p x p) and the lower factor B (p(p+1)/2 values) per
    (mode, ring), read once, in the recursion precision (8 bytes per (mode, ring) for p = 1, 28
    for p = 2 in FP32)."""
    return (n_phi // 2 + 1) * n_theta * (p * p + p * (p + 1) // 2) * (8 if fp64 else 4)


def alu_peak(fp64, sm_mhz):
    """Lane operations per second: FP32 (and INT32) issue 128 lanes per SM per clock; FP64 2."""
    return SMS * (FP64_PER_SM if fp64 else FP32_LANES) * sm_mhz * 1e6


def _peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


class Clocks:
    """nvidia-smi sampler for the timed region."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), "--query-gpu=" + self.Q,
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except Exception:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            f = [x.strip() for x in ln.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx = float(f[2])
            except ValueError:
                continue
            for nm, v in zip(names, f[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        sm.sort()
        med = sm[len(sm) // 2] if sm else None
        return {"sm_mhz": med, "sm_max_mhz": mx, "reasons": sorted(reasons), "samples": len(sm)}


def csrc_digest():
    """Digest of the sources the sampling kernels are built from (their templates and their
    instantiation units); the committed DRAM-traffic record is valid while it matches."""
    import glob
    import hashlib
    h = hashlib.sha256()
    base = os.path.join(ROOT, "paper_1709_10314_gb300", "csrc")
    for f in sorted(glob.glob(os.path.join(base, "smerf_sample_*.cu")) +
                    [os.path.join(base, "smerf_sample_impl.cuh"), os.path.join(base, "smerf_internal.cuh"),
                     os.path.join(base, "smerf_ring.cuh")]):
        with open(f, "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


def cpu_cores():
    try:
        return len(os.sched_getaffinity(0))
    except Exception:
        return os.cpu_count()


class CpuBaseline:
    """The oracle's per-sample recursion (Alg. 2) on a bounded sample of a workload: the first
    h rings of the chain in Alg. 2's order (the start ring k0 and the next rings north) of R
    realisations, every mode, then a plain radix-2 FFT per ring (oracle.recursion_sample).  Its
    tables come from the oracle's Gaussian conditioning of its spectral-sum covariance
    (oracle.recursion_tables); on grids with more than 129 modes they are computed for every
    s-th mode and shared by the modes up to the next (the recursion's cost does not depend on
    the table values).  The set-up is not timed."""

    def __init__(self, kappa, A, n_theta, n_phi, h=4):
        import numpy as np
        import oracle
        self.oracle = oracle
        nm = n_phi // 2 + 1
        self.full = n_theta <= 64 and nm <= 129
        self.h = n_theta if self.full else min(h, n_theta)
        self.stride = 1 if nm <= 129 else (nm - 1) // 16
        modes = list(range(0, nm, self.stride))
        order = oracle.conditioning_order(n_theta, 0)[:self.h]
        o, par, T, B = oracle.recursion_tables(list(kappa), A, n_theta, n_phi, H=0, rings=order, modes=modes)
        idx = np.minimum(np.arange(nm) // self.stride, len(modes) - 1)
        self.args = (len(kappa), n_phi, o, par, np.ascontiguousarray(T[idx]), np.ascontiguousarray(B[idx]))
        self.n_phi = n_phi
        self.cores = cpu_cores()

    def run(self, seed, R, threads):
        t0 = time.perf_counter()
        self.oracle.recursion_sample(*self.args, seed=seed, n_samples=R, nthreads=threads)
        return time.perf_counter() - t0

    def calibrate(self, budget_s):
        """Realisations per sample so that one single-threaded sample takes about budget_s."""
        t = self.run(1, 1, 1)
        return max(1, int(budget_s / max(t, 1e-6)))

    def points(self, R):
        return R * self.h * self.n_phi

    def sample_text(self, R):
        what = ("the whole grid (%d rings), every mode's tables exact" % self.h) if self.full else \
            ("the first %d rings of the chain (start ring and the next rings north), every mode; tables "
             "computed for every %d-th mode and shared by the modes up to the next" % (self.h, self.stride))
        return ("Alg. 2 on the host: %s, %d realisation(s) per sample (%d points); FP64 recursion with the "
                "oracle's Philox/Box-Muller noise, plain radix-2 FFT per ring" % (what, R, self.points(R)))

    def measure(self, budget_s=1.5):
        R = self.calibrate(budget_s)
        t1 = self.run(2, R, 1)
        tn = self.run(3, R, self.cores)
        return {"value": self.points(R) / tn, "unit": "points/s", "cores": self.cores,
                "kind": "oracle recursion (Alg. 2)", "single_thread_value": self.points(R) / t1,
                "sample": self.sample_text(R)}


def workload_spec(wl):
    from paper_1709_10314_gb300.workloads import FIXED, uneven_requests
    if wl == "uneven-256":
        r = uneven_requests()[0]
        return dict(kappa=r["kappa"], A=r["A"], n_theta=r["n_theta"], n_phi=r["n_phi"]), "request 0 of the batch"
    c = FIXED[wl]
    return dict(kappa=c["kappa"], A=c["A"], n_theta=c["n_theta"], n_phi=c["n_phi"]), None


def run_reference(args, rank, world):
    if rank != 0:
        return
    spec, note = workload_spec(args.workload)
    cb = CpuBaseline(spec["kappa"], spec["A"], spec["n_theta"], spec["n_phi"])
    R = cb.calibrate(0.5)  # realisations per step: a few seconds of work per step on all cores
    R = max(1, R * min(cb.cores, 16) // 2)
    dts = []
    for i in range(args.warmup + args.steps):
        dt = cb.run(100 + i, R, cb.cores)
        if i >= args.warmup:
            dts.append(dt)
    ms = 1e3 * sum(dts) / len(dts)
    value = cb.points(R) / (ms / 1e3)
    sample = cb.sample_text(R) + ("; " + note if note else "")
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": "points/s", "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": workload_name(args.workload), "name": args.workload,
                       "n_theta": spec["n_theta"], "n_phi": spec["n_phi"]},
            "cpu_baseline": {"value": value, "unit": "points/s", "cores": cb.cores, "kind": "oracle recursion (Alg. 2)",
                             "sample": sample},
            "e2e": {"value": value, "unit": "points/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def workload_name(wl):
    from paper_1709_10314_gb300.workloads import FIXED
    if wl == "uneven-256":
        return ("uneven batch: 256 requests, n_theta in {128,256,512,1024}, n_phi=2 n_theta, kappa in [5,200], "
                "p in {1,2}, 1-8 realisations, FP32 recursion, one CUDA-graph replay per step")
    c = FIXED[wl]
    return "%dx%d equiangular grid, C_l=1/prod(l(l+1)+kappa^2) kappa=%s (p=%d), %d realisations, %s tables, %s recursion+FFT" % (
        c["n_theta"], c["n_phi"], "(" + ",".join("%g" % k for k in c["kappa"]) + ")", len(c["kappa"]), c["n"],
        c["tables"].upper(), c["recur"].upper())


def run_gb300(args, rank, world, local_rank):
    import torch
    import torch.distributed as dist
    from paper_1709_10314_gb300 import Batch, Plan, create_plans
    from paper_1709_10314_gb300.replicas import max_over_ranks, rank_seed
    from paper_1709_10314_gb300.workloads import FIXED, TUNED_LAUNCH, flags_for, uneven_requests

    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    wl = args.workload
    batch = None
    launch_cfg = None
    if wl == "uneven-256":
        reqs = uneven_requests()
        # all 256 plans made in one call, their set-ups overlapping on the GPU
        plans = create_plans([dict(kappa=r["kappa"], A=r["A"], n_theta=r["n_theta"], n_phi=r["n_phi"],
                                   flags=flags_for("fp32", args.tables or "fp32")) for r in reqs])
        counts = [r["n"] for r in reqs]
        base_seeds = [r["seed"] for r in reqs]
        # with --tune: launch configurations tuned once per request shape (set-up, untimed; by
        # default the built-in choice, which measured faster for the whole batch)
        if args.tune:
            shapes = {}
            for p_, n_ in zip(plans, counts):
                key = (p_.info()["p"], p_.n_theta, p_.n_phi)
                shapes.setdefault(key, []).append((p_, n_))
            for key, members in shapes.items():
                rep = max(members, key=lambda t: t[1])
                if rep[0].launch_candidates():
                    best = rep[0].autotune(rep[1])
                    for p_, _ in members:
                        p_.set_launch(best)
        outs = [torch.empty((n, p.n_theta, p.n_phi), dtype=torch.float32, device=dev) for p, n in zip(plans, counts)]
        batch = Batch(plans, counts)
        points = sum(n * p.n_theta * p.n_phi for p, n in zip(plans, counts))
        fp64_alu = False
        alg_ops = sum(n * p.n_theta * (p.n_phi // 2) * alg_ops_per_item(p.info()["p"], p.n_phi // 2)
                      for p, n in zip(plans, counts))
        table_bytes = sum(p.info()["table_bytes"] for p in plans)
        alg_tab = sum(alg_table_bytes(p.info()["p"], p.n_theta, p.n_phi, False) for p in plans)
        sfu_ops = sum(n * p.n_theta * (p.n_phi // 2) * sfu_ops_per_item(p.info()["p"]) for p, n in zip(plans, counts))
        out_bytes = points * 4
        workload = ("uneven batch: 256 requests, n_theta in {128,256,512,1024}, n_phi=2 n_theta, kappa in [5,200], "
                    "p in {1,2}, 1-8 realisations, FP32 recursion, FP%s tables, one CUDA-graph replay per step%s"
                    % ("64" if args.tables == "fp64" else "32",
                       ", one persistent launch" if args.single_launch else ", anchor launch + persistent launch"))
        batch.set_single_launch(args.single_launch)
        dtype = "f32"
        anchor = 16  # the plans' default anchor spacing
        setup_ms = plans[0].info()["setup_ms"]  # the wall time of the one call that made them all
        s_cap = torch.cuda.Stream(device=dev)

        def set_seeds(step):
            off = rank_seed(0, rank, 1 << 40) + (step << 20)
            batch.set([b_ + off for b_ in base_seeds], outs)

        set_seeds(0)
        with torch.cuda.stream(s_cap):
            batch.launch(stream=s_cap)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s_cap, capture_error_mode="relaxed"):
            batch.launch(stream=s_cap)
        launches = batch.info()["launches"]  # anchor launch + persistent launch, or one persistent launch

        def step(i, ev0=None, ev1=None):
            torch.cuda.synchronize()
            set_seeds(i)
            if ev0 is not None:
                ev0.record()
            graph.replay()
            if ev1 is not None:
                ev1.record()
    else:
        cfg = dict(FIXED[wl])
        recur = args.recur or cfg["recur"]
        tables = args.tables or cfg["tables"]
        from paper_1709_10314_gb300 import SMERF_ORDER_PAPER
        paper_order = cfg.get("order") == "paper"
        anchor = 0 if paper_order else (args.anchor or cfg.get("H", 16))
        plan = Plan(cfg["kappa"], cfg["A"], cfg["n_theta"], cfg["n_phi"],
                    flags=flags_for(recur, tables) | (SMERF_ORDER_PAPER if paper_order else 0),
                    anchor_spacing=anchor)
        info = plan.info()
        n = cfg["n"]
        # launch configuration of the segment kernel: timed candidates (set-up, untimed)
        ws_kernel = len(plan.launch_candidates()) > 0
        stored = TUNED_LAUNCH.get((wl, recur, tables))
        if args.launch and ws_kernel:
            launch_cfg = [int(v) for v in args.launch.split(",")]
            plan.set_launch(launch_cfg)
        elif ws_kernel and not args.no_tune and not args.tune and stored in plan.launch_candidates():
            launch_cfg = list(stored)
            plan.set_launch(launch_cfg)
        else:
            launch_cfg = list(plan.autotune(n)) if (ws_kernel and not args.no_tune) else None
        out = torch.empty((n, cfg["n_theta"], cfg["n_phi"]), dtype=plan.dtype, device=dev)
        points = n * cfg["n_theta"] * cfg["n_phi"]
        out_bytes = points * (8 if recur == "fp64" else 4)
        fp64_alu = recur == "fp64"
        item_ops = fp64_pipe_ops_per_item if fp64_alu else alg_ops_per_item
        alg_ops = n * cfg["n_theta"] * (cfg["n_phi"] // 2) * item_ops(len(cfg["kappa"]), cfg["n_phi"] // 2)
        table_bytes = info["table_bytes"]
        # what the segment kernel reads: the step tables and the anchor states
        seg_read_bytes = info["step_table_bytes"], n * info["scratch_bytes_per_sample"]
        setup_ms = info["setup_ms"]
        dtype = "f64" if recur == "fp64" else "f32"
        workload = "%dx%d equiangular grid, C_l=1/prod(l(l+1)+kappa^2) kappa=%s (p=%d), %d realisations, %s tables, %s recursion+FFT" % (
            cfg["n_theta"], cfg["n_phi"], "(" + ",".join("%g" % k for k in cfg["kappa"]) + ")", len(cfg["kappa"]), n,
            tables.upper(), recur.upper())
        p_ = len(cfg["kappa"])
        alg_tab = alg_table_bytes(p_, cfg["n_theta"], cfg["n_phi"], fp64_alu)
        sfu_ops = n * cfg["n_theta"] * (cfg["n_phi"] // 2) * sfu_ops_per_item(p_)
        launches = plan.launches(n)
        seed0 = rank_seed(cfg["seed"], rank, n * (args.warmup + args.steps + 8))

        def step(i, ev0=None, ev1=None):
            if ev0 is not None:
                ev0.record()
            plan.sample_timed(seed0 + i * n, n, out, s0[i], s1[i]) if ev0 is not None else plan.sample(seed0 + i * n, n, out)
            if ev1 is not None:
                ev1.record()

    flush = torch.empty(FLUSH_BYTES // 4, dtype=torch.float32, device=dev)
    ev = lambda: torch.cuda.Event(enable_timing=True)
    e0 = [ev() for _ in range(args.steps)]
    e1 = [ev() for _ in range(args.steps)]
    s0 = [ev() for _ in range(args.steps)]
    s1 = [ev() for _ in range(args.steps)]
    # the clock sampler starts first, so that the warm-up steps (not an idle pause) directly
    # precede the timed ones
    clk = Clocks(local_rank)
    clk.start()
    time.sleep(0.3)
    for w in range(args.warmup):
        step(args.steps + w)
        flush.fill_(float(w))
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    for i in range(args.steps):
        step(i, e0[i], e1[i])
        flush.fill_(float(i))  # L2 flush between timed steps (outside the step events)
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    clocks = clk.stop()
    step_ms = sum(a.elapsed_time(b) for a, b in zip(e0, e1)) / args.steps
    if batch is None:
        seg_ms = sum(a.elapsed_time(b) for a, b in zip(s0, s1)) / args.steps
        ring = (not ws_kernel) and len(FIXED[wl]["kappa"]) == 1 and (args.recur or FIXED[wl]["recur"]) == "fp32" \
            and FIXED[wl]["n_phi"] in (16384, 32768)
        kernel = "segment_ws_kernel (small requests: segment_band_kernel)" if ws_kernel else ("ring_kernel" if ring else "segment_kernel")
    else:
        seg_ms = step_ms  # the graph replay: all groups' anchor + segment launches
        kernel = "batched graph replay (anchor + segment launches of every group)"
    step_ms, seg_ms = max_over_ranks([step_ms, seg_ms], device=dev)
    value = world * points / (step_ms / 1e3)

    # Rooflines of the segment kernel (the kernel that synthesises and writes the field).
    # HBM: the method's algorithmic bytes per launch -- the field written once plus the tables
    # read once at the method's bytes per (mode, ring) (A and the lower factor B) -- against the
    # measured copy bandwidth.  The bytes this design adds (bridge C blocks and row padding of
    # the step tables, anchor states) are reported beside it, not counted as algorithmic.  ALU:
    # algorithmic operations / kernel time against the FP32/INT32 lane rate at the maximum SM
    # clock; the kernel is bound by instruction issue (noise, recursion and FFT arithmetic).
    # SFU: Box-Muller's special functions against the 16 MUFU lanes per SM.  The batched graph
    # replay (anchor and segment launches of every group) counts the field and all of its
    # plans' tables.
    staged = batch is None and (args.recur or FIXED[wl]["recur"]) == "fp32" and \
        (args.tables or FIXED[wl]["tables"]) == "fp64" and FIXED[wl]["n"] >= 4
    alg_bytes = out_bytes + alg_tab
    if batch is None:
        step_b, anc_b = seg_read_bytes
        step_read = step_b // 2 if staged else step_b
        design = {"step_tables_as_read": step_read, "anchor_states": anc_b,
                  "extra_over_algorithmic": step_read - alg_tab + anc_b}
    else:
        design = {"tables_stored": table_bytes, "extra_over_algorithmic": table_bytes - alg_tab}
    peak, peak_kind = _peaks()
    achieved = alg_bytes / (seg_ms / 1e3) / 1e9
    sm_max = float(clocks.get("sm_max_mhz") or 2070.0) if isinstance(clocks, dict) else 2070.0
    alu_pk = alu_peak(fp64_alu, sm_max) / 1e9
    alu_ach = alg_ops / (seg_ms / 1e3) / 1e9
    sfu_pk = SMS * SFU_LANES * sm_max * 1e6 / 1e9
    sfu_ach = sfu_ops / (seg_ms / 1e3) / 1e9
    # DRAM traffic of one segment-kernel launch from the committed ncu record, only while the
    # kernel sources still hash to what was profiled (null otherwise)
    traffic = None
    prof = os.path.join(ROOT, "profiles", "segment_kernel_traffic.json")
    if os.path.exists(prof) and not args.recur and args.tables is None and batch is None:
        try:
            rec = json.load(open(prof))
            w = rec.get("workloads", {}).get(wl)
            if w and rec.get("csrc_sha256_16") == csrc_digest() and w.get("launch") == launch_cfg \
                    and w.get("anchor_spacing", 16) == anchor:
                traffic = w.get("traffic_bytes_per_launch")
        except Exception:
            traffic = None

    # end to end through the C ABI with host buffers (the field crosses the CPU-GPU link inside
    # the timed region): smerf_sample_host, or the batch writing page-locked host outputs.  The
    # link's own rate is measured beside it: one device-to-host copy of the same field into
    # page-locked memory.
    e2e = None
    if batch is not None:
        host_outs = [torch.empty(tuple(o.shape), dtype=o.dtype, pin_memory=True) for o in outs]
        off = rank_seed(0, rank, 1 << 40) + ((args.steps + args.warmup + 1) << 20)
        batch.sample([b_ + off for b_ in base_seeds], host_outs)
        torch.cuda.synchronize()
        ne = 3
        t0 = time.perf_counter()
        for i in range(ne):
            batch.sample([b_ + off + ((i + 1) << 20) for b_ in base_seeds], host_outs)
            torch.cuda.synchronize()
        e2e_s = (time.perf_counter() - t0) / ne
        e2e = {"value": world * points / e2e_s, "unit": "points/s", "h2d_bytes_per_step": 0,
               "d2h_bytes_per_step": out_bytes}
        del host_outs
    else:
        host = torch.empty(tuple(out.shape), dtype=out.dtype, pin_memory=True)
        plan.sample_host(seed0, n, host)
        ne = 3
        t0 = time.perf_counter()
        for i in range(ne):
            plan.sample_host(seed0 + i * n, n, host)
        e2e_s = (time.perf_counter() - t0) / ne
        e2e = {"value": world * points / e2e_s, "unit": "points/s", "h2d_bytes_per_step": 0,
               "d2h_bytes_per_step": out_bytes}
        # link ceiling: cudaMemcpyAsync of the device field into the same page-locked buffer
        torch.cuda.synchronize()
        c0, c1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        host.copy_(out, non_blocking=True)
        c0.record()
        for _ in range(2):
            host.copy_(out, non_blocking=True)
        c1.record()
        torch.cuda.synchronize()
        link_s = c0.elapsed_time(c1) / 2 / 1e3
        e2e["link"] = {"d2h_copy_gbs": out_bytes / link_s / 1e9, "host_path_gbs": out_bytes / e2e_s / 1e9,
                       "what": "cudaMemcpyAsync of the field into page-locked host memory (CUDA events) vs "
                               "the host-output sampling path (wall clock, synchronised per call)"}
        del host

    if rank != 0:
        return
    cpu = None
    if world == 1 and not args.no_cpu_baseline:
        spec, note = workload_spec(wl)
        cb = CpuBaseline(spec["kappa"], spec["A"], spec["n_theta"], spec["n_phi"])
        cpu = cb.measure()
        if note:
            cpu["sample"] += "; " + note
    line = {"metric": METRIC, "value": value, "unit": "points/s", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": step_ms, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": dtype, "data": "synthetic",
            "config": {"workload": workload, "name": wl, "points_per_gpu": points, "anchor_spacing": anchor,
                       "launch": launch_cfg, "parallelism": "replicas" if world > 1 else "single",
                       "l2": "flushed between timed steps (256 MiB write outside the step events)"},
            "hbm_roofline_frac": achieved / peak,
            "roofline": {"bound": "alu", "achieved": alu_ach, "peak": alu_pk, "unit": "Gop/s",
                         "frac": alu_ach / alu_pk, "traffic": traffic,
                         "peak_kind": "derived: %d SMs x %d %s lanes x %.0f MHz" % (
                             SMS, FP64_PER_SM if fp64_alu else FP32_LANES, "FP64" if fp64_alu else "FP32/INT32", sm_max),
                         "algorithmic_ops": alg_ops, "kernel": kernel, "kernel_ms": seg_ms,
                         "hbm": {"achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
                                 "peak_kind": peak_kind, "algorithmic_bytes": alg_bytes,
                                 "algorithmic": "field written once + tables A, B read once per (mode, ring)",
                                 "design_bytes": design, "tables_staged_fp32": staged,
                                 "target_frac": 0.6},
                         "sfu": {"achieved": sfu_ach, "peak": sfu_pk, "unit": "Gop/s", "frac": sfu_ach / sfu_pk,
                                 "peak_kind": "derived: %d SMs x %d MUFU lanes x %.0f MHz" % (SMS, SFU_LANES, sm_max),
                                 "ops": "log2, rsqrt, sin, cos per pair of normals"}},
            "cpu_baseline": cpu,
            "e2e": e2e,
            "gpu_launches": launches * args.steps,
            "clocks": clocks,
            "setup_ms": setup_ms, "table_bytes": table_bytes}
    print(json.dumps(line), flush=True)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="gb300", choices=["gb300", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--tables", default=None, choices=["fp64", "fp32"],
                    help="override the workload's table storage precision")
    ap.add_argument("--recur", default=None, choices=["fp64", "fp32"],
                    help="override the workload's recursion precision")
    ap.add_argument("--tune", action="store_true",
                    help="time the launch candidates (smerf_plan_autotune) instead of the stored choice")
    ap.add_argument("--no-tune", action="store_true",
                    help="keep the built-in segment-kernel launch configuration (no autotuning)")
    ap.add_argument("--launch", default=None,
                    help="fix the segment-kernel launch configuration: units/thread,realisations/CTA,"
                         "producer threads,FFT threads (one of the plan's candidates)")
    ap.add_argument("--single-launch", action="store_true",
                    help="uneven batch: anchors and segments in one persistent launch")
    ap.add_argument("--anchor", type=int, default=0,
                    help="anchor spacing H of the plan (0: the workload's default)")
    ap.add_argument("--workload", default=DEFAULT_WORKLOAD,
                    choices=["1024x2048-p2", "1024x2048-p3", "plain-64x128-p1-fp64", "4096x8192-p1", "16384x32768-p1",
                             "4096x32768-p1", "uneven-256"])
    args = ap.parse_args()
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))
    if args.impl == "reference":
        run_reference(args, rank, world)
        return
    if world > 1:
        import torch
        import torch.distributed as dist
        torch.cuda.set_device(local_rank)
        dist.init_process_group("nccl")
    run_gb300(args, rank, world, local_rank)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
