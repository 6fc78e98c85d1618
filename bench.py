#!/usr/bin/env python
"""Benchmark of the HELIOS-K hot path on GB300: one step = one (T, P)
condition through the whole path -- line preparation, Voigt opacity on the
grid (Sec. 2.3-2.4) and the per-bin k-distribution tables (sort + Chebyshev
fit, Sec. 2.6) -- on the "medium" synthetic workload: 1e5 lines over
0-30000 cm^-1, 3e6-point grid at 0.01 cm^-1, cutoff 100 cm^-1, 300 bins x 20
coefficients, T = 1500 K, P = 1 atm, 18 amu.

  python bench.py [--gpus N --steps K --warmup W] [--impl ours|reference]

Prints one JSON line.  `value` is Voigt evaluations per second of the whole
step with the line list resident in HBM; `e2e` is the same metric through the
C ABI from pinned host buffers (upload, opacity, tables back to the host).
The reference arm (--impl reference) times the FP64 CPU oracle on the host
cores on a bounded sample of the same workload.  Under torchrun each rank
runs its own condition (weak scaling, no data-path collective).
"""
import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "Voigt evals/s and opacity+k-table time/(T,P) vs plain FP64 GPU at stated rel err"
UNIT = "Voigt evals/s"
WORKLOAD = "medium"
L2_FLUSH_BYTES = 256 << 20

# Algorithmic floating-point operations per evaluation (add/sub/mul/div = 1,
# fma = 2), per method, as written in the kernels' formulas:
#   FP64 GH1  u, r^2, one division, accumulate                      -> 6
#   FP64 GH3  u, r^2, u-+t, d1, d2, d1+d2, d1 d2, num, den, /, *, + -> 19
#   FP64 916  33 per evaluation + 10 per series term
#   FP32 forms add the grid offset (1) and replace the accumulate by the
#   4 additions of the Kahan step: GH1 10, GH3 23, 916 37 + 10 per term.
FLOPS = {"f64": (6, 19, 33, 10), "f32": (10, 23, 37, 10)}
# FP64 pipe of GB300: 2 FP64 FMA / clock / SM (1.25 TFLOP/s nominal at the
# 2.07 GHz maximum clock over 152 SMs); FP32: 128 FMA lanes / SM.  These unit
# counts give the derived peaks reported beside the measured ones.
FMA_PER_CLK_SM = {"f64": 2, "f32": 128}


def probe_peaks(ctx, helk, device_index):
    """Measured throughput of the units that bound the Voigt stage (the
    library's probe kernels, timed with CUDA events), with the SM clock
    sampled while they run: the denominators of the roofline fractions."""
    kinds = (("fp32_tflops", helk.HELK_PROBE_FFMA), ("fp64_tflops", helk.HELK_PROBE_DFMA),
             ("mufu_rcp_tops", helk.HELK_PROBE_MUFU_RCP), ("mufu_ex2_tops", helk.HELK_PROBE_MUFU_EX2))
    ctx.peak_probe(helk.HELK_PROBE_FFMA)  # warm-up (clocks ramp)
    out = {}
    with Clocks(device_index) as clk:
        for name, kind in kinds:
            ops, ms = ctx.peak_probe(kind)
            out[name] = ops / 1e12
            out[name.rsplit("_", 1)[0] + "_ms_per_launch"] = ms
    out["clocks"] = clk.summary()
    out["how"] = ("helk_peak_probe: every SM filled with 8 independent chains a thread of one instruction "
                  "(FP32 FMA, FP64 FMA, rcp.approx after an FP32 add, ex2.approx), loop calibrated to ~20 ms a launch, mean of "
                  "3 launches by CUDA events; FMA counted as 2 flops; burst figure (kernel timed alone)")
    return out


def workload_desc(w):
    return ("medium: %d lines over 0-30000 cm^-1, %d-point grid at %g cm^-1, cutoff %g cm^-1, "
            "%d k-bins x %d Chebyshev coefficients, T=%g K, P=%g atm, %g amu"
            % (w["nlines"], w["ngrid"], w["dnu"], w["cut"][1], w["nbins"], w["ncheb"], w["T"][0],
               w["P_atm"][0], w["mass"]))


def dist_env():
    return (int(os.environ.get("RANK", "0")), int(os.environ.get("LOCAL_RANK", "0")),
            int(os.environ.get("WORLD_SIZE", "1")))


def rank_temperature(w, rank, world):
    """The condition rank `rank` of `world` runs (weak scaling: every rank
    runs the full workload at its own temperature; one rank runs the
    workload's own)."""
    import numpy as np
    return w["T"][0] if world == 1 else float(np.linspace(500.0, 3000.0, world)[rank])


def max_over_ranks(value, dist, device):
    """Max of a per-rank scalar (step times are reported as the slowest
    rank's); the one collective of the benchmark, outside the data path."""
    if dist is None:
        return value
    import torch
    t = torch.tensor([float(value)], device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def kdist_hbm(ms, n, peaks):
    """HBM view of the k-table stage: its algorithmic bytes (each opacity
    read once, 8 B a point; the pseudo-inverse comes from L2) over its time,
    against the measured copy bandwidth."""
    if not ms:
        return None
    gbs = 8.0 * n / (ms * 1e-3) / 1e9
    peak = peaks.get("hbm_gbs")
    return {"bytes_per_launch": 8 * n, "achieved": gbs, "unit": "GB/s", "peak": peak,
            "frac": gbs / peak if peak else None,
            "note": "latency-bound per-bin sort (one 512-thread CTA per bin, two per SM) and fit; not HBM-bound at 1e4-point bins"}


def measured_peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return json.load(f)
    except Exception:
        return {}


class Clocks:
    """nvidia-smi sampling during the timed region."""

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.path = None

    def __enter__(self):
        q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index), "--query-gpu=" + q,
                 "--format=csv,noheader,nounits", "-lms", "100"],
                stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None
        time.sleep(0.3)
        return self

    def __exit__(self, *a):
        if self.proc:
            time.sleep(0.2)
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()

    def summary(self):
        if not self.proc or not self.path:
            return None
        rows = []
        with open(self.path) as f:
            for line in f:
                p = [x.strip() for x in line.split(",")]
                if len(p) >= 9:
                    rows.append(p)
        os.unlink(self.path)
        if not rows:
            return None
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        reasons = set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for r in rows:
            for n, v in zip(names, r[5:9]):
                if v.lower() == "active":
                    reasons.add(n)
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(mx) if mx else None, "reasons": sorted(reasons),
                "samples": len(rows)}


# The Voigt kernels' translation unit: the kernel file and the headers of
# csrc/ it includes; the profile summaries record a hash of these sources.
KERNEL_HEADERS = ("wings.cuh", "voigt_f32.cuh", "voigt_core.cuh", "voigt_common.cuh", "helk_internal.cuh",
                  "route.cuh", "sort_runs.cuh")


def kernel_source_hash(kernel_src):
    d = os.path.dirname(kernel_src)
    h = hashlib.sha256()
    for f in (kernel_src,) + tuple(os.path.join(d, x) for x in KERNEL_HEADERS):
        h.update(open(f, "rb").read())
    return h.hexdigest()[:16]


def traffic_from_profile(kernel_src, profile_txt):
    """Per-launch DRAM bytes recorded by an ncu capture, if the kernel's
    sources are unchanged since (hash recorded in the summary)."""
    try:
        h = kernel_source_hash(kernel_src)
        vals = {}
        with open(profile_txt) as f:
            for line in f:
                if ":" in line:
                    k, v = line.split(":", 1)
                    vals[k.strip()] = v.strip()
        if vals.get("kernel_source_sha256_16") != h:
            return None
        return float(vals["dram_bytes_per_launch_full_workload"])
    except Exception:
        return None


# --------------------------------------------------------------- oracle --
def oracle_sample(w, lines, target_s, nthreads):
    """Time the FP64 oracle on a contiguous slab of k-bins (all their lines):
    opacity on the slab's grid + sort + Chebyshev fit.  Returns
    (evals, seconds, nbins_used)."""
    import oracle
    nb = w["ngrid"] // w["nbins"]

    def run(nbins_s, b0):
        cond = oracle.Condition(w["T"][0], w["P_atm"][0], w["mass"],
                                w["nu_min"] + b0 * nb * w["dnu"], w["dnu"], nbins_s * nb,
                                oracle.CUT_ABS, w["cut"][1])
        t = time.perf_counter()
        k, ev, _ = oracle.opacity(lines, cond, nthreads=nthreads)
        oracle.kdist(k, nbins_s, w["ncheb"])
        return ev, time.perf_counter() - t

    b0 = w["nbins"] // 2
    ev, dt = run(1, b0)
    nbins_s = max(1, min(w["nbins"] - b0, int(target_s / max(dt, 1e-3))))
    if nbins_s > 1:
        ev, dt = run(nbins_s, b0)
    return ev, dt, nbins_s


def run_reference(args):
    rank, local_rank, world = dist_env()
    if rank != 0:
        return
    from paper_1503_03806_gb300 import synth
    import oracle
    oracle.lib()
    w = synth.WORKLOADS[WORKLOAD]
    lines = synth.workload_lines(WORKLOAD)
    cores = os.cpu_count() or 1
    # size one step at ~1/(K+W) of a ~60 s budget
    per_step = max(2.0, 60.0 / (args.steps + args.warmup))
    ev1, dt1, nbs = oracle_sample(w, lines, per_step, cores)
    for _ in range(max(0, args.warmup - 1)):
        oracle_sample(w, lines, per_step, cores)
    evs, dts = [], []
    for _ in range(args.steps):
        ev, dt, nbs = oracle_sample(w, lines, per_step, cores)
        evs.append(ev)
        dts.append(dt)
    value = sum(evs) / sum(dts)
    sample = "%d contiguous k-bins (%d grid points, all overlapping lines) per step" % (
        nbs, nbs * (w["ngrid"] // w["nbins"]))
    out = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus, "steps": args.steps,
           "warmup": args.warmup, "ms_per_step": 1e3 * sum(dts) / len(dts),
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
           "data": "synthetic", "impl": "reference",
           "config": {"workload": workload_desc(w), "sample": sample},
           "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle",
                            "sample": sample},
           "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(out), flush=True)


# ------------------------------------------------------------------ ours --
def run_ours(args):
    import numpy as np
    import torch
    rank, local_rank, world = dist_env()
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl" if torch.cuda.is_available() else "gloo")
    torch.cuda.set_device(local_rank)
    import __graft_entry__
    __graft_entry__.build()
    from paper_1503_03806_gb300 import helk, synth

    w = synth.WORKLOADS[WORKLOAD]
    T = rank_temperature(w, rank, world)
    P, mass, cut = w["P_atm"][0], w["mass"], w["cut"]
    grid = (w["nu_min"], w["dnu"], w["ngrid"])
    nbins, ncheb = w["nbins"], w["ncheb"]
    lines = synth.workload_lines(WORKLOAD)
    PREC = {"f64": helk.HELK_PREC_F64, "f32": helk.HELK_PREC_F32_KAHAN}
    peaks = measured_peaks()
    max_mhz = float(peaks.get("sm_max_mhz", 2070.0))
    nsm = torch.cuda.get_device_properties(local_rank).multi_processor_count

    ctx = helk.Context(local_rank)
    peaks_meas = probe_peaks(ctx, helk, local_rank)
    ctx.upload(lines)
    kappa = torch.empty(grid[2], dtype=torch.float64, device="cuda")
    flush = torch.empty(L2_FLUSH_BYTES, dtype=torch.uint8, device="cuda")

    def measure(form, clocks=False):
        prec = PREC[form]
        # work of one step (exact counts from the counting variant, which evaluates point by point)
        ctx.opacity(T, P, mass, cut, grid, out=kappa, precision=prec, count_regions=True)
        evals, reg = ctx.stats(with_regions=True)
        f = FLOPS[form]
        flops = int(reg[2] * f[0] + reg[1] * f[1] + reg[0] * f[2] + reg[3] * f[3])

        def step():
            ctx.opacity(T, P, mass, cut, grid, out=kappa, precision=prec)
            ctx.kdist(kappa, nbins, ncheb)

        for _ in range(args.warmup):
            step()
        torch.cuda.synchronize()
        starts = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
        ends = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
        if dist:
            dist.barrier()
        torch.cuda.synchronize()
        clk = Clocks(local_rank) if clocks else None
        if clk:
            clk.__enter__()
        t0 = time.perf_counter()
        nl0 = ctx.launch_count()
        for i in range(args.steps):
            flush.zero_()                      # L2 flush, outside the timed events
            starts[i].record()
            step()
            ends[i].record()
        torch.cuda.synchronize()
        launches = ctx.launch_count() - nl0   # the library's kernels in the timed steps
        wall = time.perf_counter() - t0
        if clk:
            clk.__exit__()
        if dist:
            dist.barrier()
        # per-stage times from a separate pass (the stage events stay out of
        # the timed steps)
        ctx.set_profiling(True)
        for _ in range(max(3, min(args.steps, 10))):
            flush.zero_()
            step()
        torch.cuda.synchronize()
        stage = ctx.stage_times()
        ctx.set_profiling(False)
        ms = [a.elapsed_time(b) for a, b in zip(starts, ends)]
        ms_step = max_over_ranks(sum(ms) / len(ms), dist, "cuda")
        voigt_ms, voigt_n = stage["voigt"]
        voigt_s = voigt_ms / max(1, voigt_n) * 1e-3
        peak_derived = FMA_PER_CLK_SM[form] * 2 * nsm * max_mhz * 1e6 / 1e12
        peak = peaks_meas["fp32_tflops" if form == "f32" else "fp64_tflops"]
        achieved = flops / voigt_s / 1e12
        src = os.path.join(ROOT, "paper_1503_03806_gb300", "csrc",
                           "k_wings.cu" if form == "f32" else "k_wings64.cu")
        # `achieved` is the work of the point-by-point sums over the time of the
        # stage.  The stage interpolates most of it (wings.cuh), so this is no rate
        # of the pipe and may exceed its peak: frac is against what no kernel can
        # do without, the line list read and kappa written once.
        hbm_bytes = 8 * (len(lines) * lines["nu0"].shape[0] + grid[2])
        hbm_peak = peaks.get("hbm_gbs")
        hbm_gbs = hbm_bytes / voigt_s / 1e9
        roof = {"bound": "alu", "achieved": achieved, "peak": peak,
                "unit": "TFLOP/s of point-by-point work (most of it interpolated)",
                "frac": hbm_gbs / hbm_peak if hbm_peak else None,
                "frac_basis": "of measured copy bandwidth, for the line list read and kappa written once",
                "hbm_floor_bytes": hbm_bytes, "hbm_floor_gbs": hbm_gbs, "hbm_peak_gbs": hbm_peak,
                "point_by_point_over_peak": achieved / peak,
                "traffic": traffic_from_profile(src, os.path.join(ROOT, "profiles",
                                                                  "wings_%s_medium.txt" % form)),
                "kernel": ("k_wing_far32 + k_core_f32 + k_wing_near32" if form == "f32"
                           else "k_wing_far64 + k_wing_near64") + " (the Voigt stage)",
                "peak_basis": "measured: %s FMA probe of this run (peaks_measured, helk_peak_probe), burst"
                              % form.upper(),
                "peak_derived": peak_derived,
                "peak_derived_basis": "%s pipe: %d FMA/clk/SM x %d SMs x %.0f MHz max clock"
                                      % (form.upper(), FMA_PER_CLK_SM[form], nsm, max_mhz),
                "flops_per_launch": flops, "voigt_ms_per_launch": voigt_s * 1e3}
        return {"form": form, "evals": evals, "reg": [int(x) for x in reg], "ms_step": ms_step,
                "launches": launches,
                "value": world * evals / (ms_step * 1e-3), "roofline": roof, "wall": wall,
                "stages": {k: v[0] / max(1, v[1]) for k, v in stage.items() if v[1]},
                "clocks": clk.summary() if clk else None}

    r64 = measure("f64")
    k64 = kappa.clone()
    r32 = measure("f32", clocks=True)
    # accuracy of the FP32 form on this workload, against the FP64 form
    # (itself held to the FP64 oracle at 1e-9 by the tests)
    g = kappa.view(nbins, -1)
    r = k64.view(nbins, -1)
    sel = r > 1e-8 * r.max(dim=1, keepdim=True).values
    err32 = float(((g - r).abs() / r)[sel].max().item())
    clocks = r32["clocks"]

    # end to end through the C ABI from pinned host memory (FP32 form)
    e2e = None
    if not args.no_e2e:
        pinned = {k: torch.from_numpy(v).pin_memory() for k, v in lines.items()}
        h2d = sum(v.numel() * 8 for v in pinned.values())
        d2h = nbins * ncheb * 8 + nbins * 8

        def e2e_step():
            ctx.upload(pinned)
            ctx.opacity(T, P, mass, cut, grid, out=kappa, precision=PREC["f32"])
            ctx.kdist(kappa, nbins, ncheb, on_host=True)

        for _ in range(max(1, args.warmup)):
            e2e_step()
        torch.cuda.synchronize()
        tt = []
        for _ in range(args.steps):
            flush.zero_()
            torch.cuda.synchronize()
            t1 = time.perf_counter()
            e2e_step()
            torch.cuda.synchronize()
            tt.append(time.perf_counter() - t1)
        e2e_s = max_over_ranks(sum(tt) / len(tt), dist, "cuda")
        e2e = {"value": world * r32["evals"] / e2e_s, "unit": UNIT, "h2d_bytes_per_step": h2d,
               "d2h_bytes_per_step": d2h, "ms_per_step": e2e_s * 1e3}

    # batched conditions: the 8 T x 8 P workload (1e6 lines) in one captured
    # graph per call, k-tables of all 64 in one call
    tpg = None
    if not args.no_tp_grid:
        wt = synth.WORKLOADS["tp_grid"]
        tl = synth.workload_lines("tp_grid")
        Ts = np.repeat(np.asarray(wt["T"]), len(wt["P_atm"]))
        Ps = np.tile(np.asarray(wt["P_atm"]), len(wt["T"]))
        qs = (296.0 / Ts) ** 1.5
        gt = (wt["nu_min"], wt["dnu"], wt["ngrid"])
        ctx.upload(tl)
        kb = torch.empty((len(Ts), gt[2]), dtype=torch.float64, device="cuda")
        ctx.opacity_batch(Ts, Ps, wt["mass"], wt["cut"], gt, out=kb, precision=PREC["f32"], q_ratio=qs,
                          count_regions=True)
        ev_b, _ = ctx.batch_stats(len(Ts))
        nsteps = max(1, min(args.steps, 3))
        for _ in range(max(1, min(args.warmup, 2))):
            ctx.opacity_batch(Ts, Ps, wt["mass"], wt["cut"], gt, out=kb, precision=PREC["f32"], q_ratio=qs)
            ctx.kdist(kb.view(-1), len(Ts) * wt["nbins"], wt["ncheb"])
        torch.cuda.synchronize()
        ctx.set_profiling(True)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(nsteps):
            ctx.opacity_batch(Ts, Ps, wt["mass"], wt["cut"], gt, out=kb, precision=PREC["f32"], q_ratio=qs)
            ctx.kdist(kb.view(-1), len(Ts) * wt["nbins"], wt["ncheb"])
        e1.record()
        torch.cuda.synchronize()
        st_b = ctx.stage_times()
        ctx.set_profiling(False)
        ms_b = e0.elapsed_time(e1) / nsteps
        tpg = {"workload": "tp_grid: %d lines, %d conditions (T %g-%g K x P %g-%g atm), %d-point grid, "
                           "cutoff min(500 Gamma_L, 100 cm^-1), %d bins x %d coefficients"
                           % (wt["nlines"], len(Ts), min(Ts), max(Ts), min(Ps), max(Ps), gt[2],
                              wt["nbins"], wt["ncheb"]),
               "form": "FP32 + Kahan, one captured graph per call",
               "ms_per_call": ms_b, "ms_per_condition": ms_b / len(Ts),
               "evals_per_call": int(ev_b.sum()), "value": int(ev_b.sum()) / (ms_b * 1e-3),
               "unit": UNIT,
               "stages_ms_per_call": {k: v[0] / max(1, v[1]) for k, v in st_b.items() if v[1]}}
        del kb
        ctx.upload(lines)

    # the learned surrogate for Algorithm 916: trained on the GPU by the
    # library's own kernels, validated cell by cell, then routed in the FP32
    # form; timed against the FP32 and FP64 forms on a core-dominated case
    surr = None
    if not args.no_surrogate:
        t0 = time.perf_counter()
        ctx.surrogate_init(7)
        sloss = ctx.surrogate_train(10_000_000, 11, 100, batch=4096, lr=2e-3)
        train_s = time.perf_counter() - t0
        mask, serr = ctx.surrogate_validate(32, 32, 8, 5e-5)
        sl = synth.random_lines(3000, 601, 10000.0, 10300.0)
        sgrid, scut = (10000.0, 0.001, 300_000), ("abs", 0.3)
        ctx.upload(sl)
        ks = torch.empty(sgrid[2], dtype=torch.float64, device="cuda")
        forms = {"fp64": dict(precision=PREC["f64"]), "fp32": dict(precision=PREC["f32"]),
                 "fp32_surrogate": dict(precision=PREC["f32"], surrogate=True)}
        sms, outs = {}, {}
        for name, kw in forms.items():
            ctx.opacity(1500.0, 0.01, 18.0, scut, sgrid, out=ks, **kw)
            torch.cuda.synchronize()
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(5):
                ctx.opacity(1500.0, 0.01, 18.0, scut, sgrid, out=ks, **kw)
            b.record()
            torch.cuda.synchronize()
            sms[name] = a.elapsed_time(b) / 5
            outs[name] = ks.clone()
        ctx.opacity(1500.0, 0.01, 18.0, scut, sgrid, out=ks, precision=PREC["f32"], count_regions=True)
        sev, sreg = ctx.stats(with_regions=True)
        r = outs["fp64"].view(30, -1)
        selm = r > 1e-8 * r.max(dim=1, keepdim=True).values
        serr_s = float(((outs["fp32_surrogate"].view(30, -1) - r).abs() / r)[selm].max().item())
        checked = serr >= 0
        surr = {"network": "2-64-64-64-1 SiLU, BF16 mma.sync m16n8k16 (hi/lo split forward), FP32 accumulate",
                "training": "1e7 samples x 100 epochs, Adam, batch 4096, targets from FP64 Algorithm 916",
                "train_s": train_s, "final_loss": sloss,
                "validated_cells": int(mask.sum()), "checked_cells": int(checked.sum()),
                "validation_tol": 5e-5, "stated_error": 1e-4,
                "workload": "core-dominated: 3000 lines over 10000-10300 cm^-1, P 0.01 atm, 1500 K, "
                            "3e5-point grid at 0.001 cm^-1, cutoff 0.3 cm^-1",
                "evals": int(sev), "alg916_share": float(sreg[0]) / max(1, int(sev)),
                "ms": sms, "gain_vs_fp64": sms["fp64"] / sms["fp32_surrogate"],
                "gain_vs_fp32": sms["fp32"] / sms["fp32_surrogate"],
                "max_rel_err_vs_fp64": serr_s}
        del ks
        ctx.upload(lines)
        # the benchmark's own spectrum (opacity + k-tables, one (T,P)) with
        # the surrogate routed, beside the FP32 and FP64 steps timed above
        km = torch.empty(w["ngrid"], dtype=torch.float64, device="cuda")
        mgrid = (w["nu_min"], w["dnu"], w["ngrid"])

        def sstep():
            ctx.opacity(w["T"][0], w["P_atm"][0], w["mass"], w["cut"], mgrid, out=km, precision=PREC["f32"],
                        surrogate=True)
            ctx.kdist(km, w["nbins"], w["ncheb"])
        for _ in range(3):
            sstep()
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(5):
            sstep()
        b.record()
        torch.cuda.synchronize()
        ms_sur = a.elapsed_time(b) / 5
        surr["medium_spectra_per_s"] = {"fp32_surrogate": 1e3 / ms_sur, "fp32": 1e3 / r32["ms_step"],
                                        "fp64": 1e3 / r64["ms_step"],
                                        "note": "opacity + k-tables of the medium workload per second; "
                                                "surrogate step without the L2 flush"}
        del km

    # the paper's Transmission stage (Sec. 3.5: 1000 column masses per bin) on
    # the medium workload's k-tables: from the sorted values and from the fit
    trans = None
    if not args.no_transmission:
        trans = leg_transmission(ctx, w, T, P, mass, cut, grid, PREC["f32"])

    # the 1e7-line workload at 1500 K, 1 atm: opacity + k-tables per (T, P),
    # FP32 with and without the surrogate (when its leg trained one)
    surrw = None
    if not args.no_surrogate_workload:
        surrw = leg_surrogate_workload(ctx, args, PREC["f32"], trained=surr is not None, flush=flush)
        ctx.upload(lines)

    # the mixed workload: 1e8 lines of 4 species, 16 conditions in one batch
    # call, then the k-tables of all of them in one call
    mixed = None
    if not args.no_mixed:
        mixed = leg_mixed(ctx, PREC["f32"], local_rank, peaks)
        ctx.upload(lines)

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        cores = os.cpu_count() or 1
        ev_c, dt_c, nbs = oracle_sample(w, lines, 10.0, cores)
        cpu = {"value": ev_c / dt_c, "unit": UNIT, "cores": cores, "kind": "oracle",
               "sample": "%d contiguous k-bins (%d grid points, all overlapping lines): opacity + "
                         "sort + fit, FP64, %.1f s" % (nbs, nbs * (grid[2] // nbins), dt_c)}

    if rank == 0:
        reg = r32["reg"]
        out = {"metric": METRIC, "value": r32["value"], "unit": UNIT, "n_gpus": world,
               "steps": args.steps, "warmup": args.warmup, "ms_per_step": r32["ms_step"],
               "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
               "dtype": "f32 (Voigt, Kahan) / float-float + exact integer (k-tables)", "data": "synthetic",
               "config": {"workload": workload_desc(w),
                          "form": "FP32 Voigt + Kahan; k-tables: float-float log and fit (~2^-46 relative), "
                                  "exact 128-bit integer mean, FP64 pseudo-inverse",
                          "l2": "flushed between steps (256 MB write)",
                          "evals_per_step": r32["evals"],
                          "evals_by_method": {"alg916": reg[0], "gh3": reg[1], "gh1": reg[2]}},
               "rel_err_f32_vs_f64": err32,
               "stages_ms_per_step": r32["stages"],
               "kdist_hbm": kdist_hbm(r32["stages"].get("kdist"), grid[2], peaks),
               "roofline": r32["roofline"], "peaks_measured": peaks_meas,
               "cpu_baseline": cpu, "e2e": e2e, "clocks": clocks,
               "gpu_launches": r32["launches"],
               "fp64": {"value": r64["value"], "ms_per_step": r64["ms_step"],
                        "stages_ms_per_step": r64["stages"], "roofline": r64["roofline"],
                        "gpu_launches": r64["launches"]},
               "speedup_f32_vs_f64": r32["value"] / r64["value"],
               "tp_grid": tpg, "surrogate": surr, "surrogate_workload": surrw, "mixed": mixed,
               "transmission": trans}
        print(json.dumps(out), flush=True)
    ctx.close()
    if dist:
        dist.destroy_process_group()


def leg_transmission(ctx, w, T, P, mass, cut, grid, prec):
    """Transmission of every bin of the medium workload for 1000 column
    masses (log-spaced), from the sorted k(g) and from the 20-coefficient fit
    resampled on 1000 points: the paper's last stage, timed by CUDA events."""
    import numpy as np
    import torch
    nbins, ncheb = w["nbins"], w["ncheb"]
    kap = ctx.opacity(T, P, mass, cut, grid, precision=prec)
    coef, _, srt = ctx.kdist(kap, nbins, ncheb, want_sorted=True)
    m = np.logspace(14.0, 30.0, 1000)  # molecules cm^-2 (kappa is per molecule)
    out = {}
    for name, kw in (("direct", dict(sorted_k=srt)), ("fit", dict(coeffs=coef, ng=1000))):
        ctx.transmission(nbins, m, **kw)
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(3):
            ctx.transmission(nbins, m, **kw)
        b.record()
        torch.cuda.synchronize()
        out[name + "_ms"] = a.elapsed_time(b) / 3
    out["what"] = ("T_b(m) for %d bins x 1000 column masses: direct = midpoint rule over the %d sorted "
                   "values of each bin, fit = midpoint rule over 1000 points of the resampled k(g); "
                   "e^{-k_0 m} factored out, terms below e^-87 of it skipped, the rest by a float-float "
                   "exponential on the FP32 pipe" % (nbins, grid[2] // nbins))
    return out


def timed_steps(step, steps, warmup, flush):
    """Mean device time of `steps` calls of step() after `warmup` untimed
    ones, the L2 flushed before each (outside the events)."""
    import torch
    for _ in range(warmup):
        step()
    torch.cuda.synchronize()
    ms = []
    for _ in range(steps):
        if flush is not None:
            flush.zero_()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        step()
        b.record()
        torch.cuda.synchronize()
        ms.append(a.elapsed_time(b))
    return sum(ms) / len(ms)


def leg_surrogate_workload(ctx, args, prec, trained, flush):
    """The 1e7-line workload (log-normal strengths, lower-state energies) at
    1500 K, 1 atm on the 3e6-point grid: opacity + 300 x 20 k-tables per
    (T, P) in the FP32 form, and with the surrogate routed when a network was
    trained and validated in this run."""
    import torch
    from paper_1503_03806_gb300 import helk, synth
    ws = synth.WORKLOADS["surrogate"]
    ls = synth.workload_lines("surrogate")
    g = (ws["nu_min"], ws["dnu"], ws["ngrid"])
    Tq, Pq, q = ws["T"][0], ws["P_atm"][0], (296.0 / ws["T"][0]) ** 1.5
    ctx.upload(ls)
    del ls
    k = torch.empty(g[2], dtype=torch.float64, device="cuda")
    ctx.opacity(Tq, Pq, ws["mass"], ws["cut"], g, out=k, precision=prec, q_ratio=q, count_regions=True)
    evals, reg = ctx.stats(with_regions=True)
    out = {"workload": "surrogate: %d lines, %d-point grid, cutoff min(500 Gamma_L, 100 cm^-1), T %g K, "
                       "P %g atm, %d bins x %d coefficients"
                       % (ws["nlines"], g[2], Tq, Pq, ws["nbins"], ws["ncheb"]),
           "evals_per_step": int(evals), "alg916_share": float(reg[0]) / max(1, int(evals))}
    forms = {"fp32": False}
    if trained:
        forms["fp32_surrogate"] = True
    for name, sur in forms.items():
        def step():
            ctx.opacity(Tq, Pq, ws["mass"], ws["cut"], g, out=k, precision=prec, q_ratio=q, surrogate=sur)
            ctx.kdist(k, ws["nbins"], ws["ncheb"])
        ms = timed_steps(step, max(3, min(args.steps, 10)), max(3, args.warmup), flush)
        out[name] = {"ms_per_step": ms, "spectra_per_s": 1e3 / ms, "value": evals / (ms * 1e-3),
                     "unit": UNIT}
    if trained:
        out["gain_vs_fp32"] = out["fp32"]["ms_per_step"] / out["fp32_surrogate"]["ms_per_step"]
    del k
    return out


def leg_mixed(ctx, prec, device_index, peaks):
    """The mixed workload: 1e8 lines of 4 species (per-line mass and
    abundance weight), all 4 T x 4 P conditions in one helk_opacity_batch call
    (FP32 form, records in chunks under the batch record budget) on the
    3e7-point grid, then the k-tables of all 16 conditions (16000 bins of
    30000 points, 20 coefficients) in one helk_kdist call.  One timed call of
    each (a call is tens of seconds), clocks sampled."""
    import numpy as np
    import torch
    from paper_1503_03806_gb300 import synth
    wm = synth.WORKLOADS["mixed"]
    parts = []
    for sp, (m, x) in enumerate(zip(wm["species_mass"], wm["mixing"])):
        L = synth.workload_lines("mixed", species=sp)
        L["mass"] = np.full(L["nu0"].shape[0], m)
        L["weight"] = np.full(L["nu0"].shape[0], x)
        parts.append(L)
    lm = {k: np.concatenate([p[k] for p in parts]) for k in parts[0]}
    del parts
    order = np.argsort(lm["nu0"], kind="stable")
    lm = {k: np.ascontiguousarray(v[order]) for k, v in lm.items()}
    del order
    g = (wm["nu_min"], wm["dnu"], wm["ngrid"])
    Ts = np.repeat(np.asarray(wm["T"]), len(wm["P_atm"]))
    Ps = np.tile(np.asarray(wm["P_atm"]), len(wm["T"]))
    qs = (296.0 / Ts) ** 1.5
    nc = len(Ts)
    ctx.upload(lm)
    nlines = lm["nu0"].shape[0]
    del lm
    kb = torch.empty((nc, g[2]), dtype=torch.float64, device="cuda")
    # one-time set-up of this bin size (the pseudo-inverse), outside the timing
    nbp = g[2] // wm["nbins"]
    ctx.kdist(torch.ones(nbp, dtype=torch.float64, device="cuda"), 1, wm["ncheb"])
    torch.cuda.synchronize()
    with Clocks(device_index) as clk:
        ctx.set_profiling(True)
        a, b, c2 = (torch.cuda.Event(enable_timing=True) for _ in range(3))
        a.record()
        ctx.opacity_batch(Ts, Ps, 18.0, wm["cut"], g, out=kb, precision=prec, q_ratio=qs)
        b.record()
        ctx.kdist(kb.view(-1), nc * wm["nbins"], wm["ncheb"])
        c2.record()
        torch.cuda.synchronize()
        st = ctx.stage_times()
        ctx.set_profiling(False)
    ev, _ = ctx.batch_stats(nc)
    ms_op, ms_kd = a.elapsed_time(b), b.elapsed_time(c2)
    total = ms_op + ms_kd
    n_all = nc * g[2]
    kd_gbs = 8.0 * n_all / (ms_kd * 1e-3) / 1e9
    out = {"workload": "mixed: %d lines (4 species, masses %s amu, mixing 1/4), %d conditions (T %g-%g K x P "
                       "%g-%g atm), %d-point grid at %g cm^-1, cutoff min(500 Gamma_L, 100 cm^-1), %d bins x %d "
                       "coefficients per condition" % (nlines, wm["species_mass"], nc, min(Ts), max(Ts), min(Ps),
                                                       max(Ps), g[2], g[1], wm["nbins"], wm["ncheb"]),
           "form": "FP32 + Kahan, one helk_opacity_batch call (records in chunks under the 64 GiB budget) + "
                   "one helk_kdist call",
           "evals_per_call": int(ev.sum()), "evals_per_condition": [int(x) for x in ev],
           "opacity_ms": ms_op, "kdist_ms": ms_kd, "ms_per_condition": total / nc,
           "spectra_per_s": nc / (total * 1e-3), "value": float(ev.sum()) / (ms_op * 1e-3), "unit": UNIT,
           "kdist_hbm": {"bytes": 8 * n_all, "achieved": kd_gbs, "unit": "GB/s",
                         "peak": peaks.get("hbm_gbs"),
                         "frac": kd_gbs / peaks["hbm_gbs"] if peaks.get("hbm_gbs") else None,
                         "note": "bins of 30000 points: split by value into parts sorted in shared memory; the "
                                 "one-time pseudo-inverse of this bin size is built before the timing"},
           "stages_ms": {k: v[0] for k, v in st.items() if v[1]},
           "clocks": clk.summary(), "timed_calls": 1}
    del kb
    torch.cuda.empty_cache()
    return out


def run_profile_surrogate():
    """Short fixed run for profilers: train the surrogate briefly (1e6
    samples x 2 epochs), validate it, and run the core-dominated opacity case
    with routing twice."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_1503_03806_gb300 import helk, synth
    ctx = helk.Context(0)
    ctx.surrogate_init(7)
    ctx.surrogate_train(1_000_000, 11, 2, batch=4096, lr=3e-3)
    ctx.surrogate_validate(32, 32, 8, 1e-3)
    ctx.upload(synth.random_lines(3000, 601, 10000.0, 10300.0))
    k = torch.empty(300_000, dtype=torch.float64, device="cuda")
    for _ in range(2):
        ctx.opacity(1500.0, 0.01, 18.0, ("abs", 0.3), (10000.0, 0.001, 300_000), out=k,
                    precision=helk.HELK_PREC_F32_KAHAN, surrogate=True)
    ctx.sync()
    ctx.close()


def run_profile_case(form):
    """Short fixed run for profilers: upload the workload, then two passes of
    opacity (FP32 or FP64 form) + k-tables."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_1503_03806_gb300 import helk, synth
    w = synth.WORKLOADS[WORKLOAD]
    prec = helk.HELK_PREC_F32_KAHAN if form == "f32" else helk.HELK_PREC_F64
    ctx = helk.Context(0)
    ctx.upload(synth.workload_lines(WORKLOAD))
    grid = (w["nu_min"], w["dnu"], w["ngrid"])
    kappa = torch.empty(w["ngrid"], dtype=torch.float64, device="cuda")
    for _ in range(2):
        ctx.opacity(w["T"][0], w["P_atm"][0], w["mass"], w["cut"], (w["nu_min"], w["dnu"], w["ngrid"]),
                    out=kappa, precision=prec)
        ctx.kdist(kappa, w["nbins"], w["ncheb"])
    ctx.sync()
    ctx.close()


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-tp-grid", action="store_true", help="skip the batched 64-condition leg")
    ap.add_argument("--no-surrogate", action="store_true", help="skip the surrogate leg")
    ap.add_argument("--no-surrogate-workload", action="store_true", help="skip the 1e7-line workload leg")
    ap.add_argument("--no-mixed", action="store_true", help="skip the 1e8-line 16-condition leg")
    ap.add_argument("--no-transmission", action="store_true", help="skip the transmission leg")
    ap.add_argument("--profile-case", choices=["f32", "f64", "surrogate"], default=None,
                    help="run a short fixed case for ncu and exit")
    args = ap.parse_args()
    if args.profile_case == "surrogate":
        run_profile_surrogate()
    elif args.profile_case:
        run_profile_case(args.profile_case)
    elif args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
