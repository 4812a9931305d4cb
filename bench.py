"""Benchmark of the approximate-region hot path on GB300.

Headline workload (the large hydro configuration): a 256^3-element hexahedral
Lagrangian-hydro mesh (node coordinates jittered +-5%, energy 3.9e6 in the
corner element), FP64, 200 time steps, whose equation-of-state (EOS) call is
the approximated region. Before timing, every candidate form of the EOS
(TAF and iACT with state scoped to one launch, and with windows / tables kept
across time steps) runs once and is scored against the exact run: the error
of the final origin energy (the paper's LULESH quantity of interest) and the
normalised RMSE of the final pressure field, ||p - p_exact|| / ||p_exact||
(the exact pressure is zero outside the blast, so this is the error on the
elements the blast reached). A form qualifies when both are <= 1% and it
approximates at least 10% of the active invocations: the EOS calls of
elements that carry energy at that step in the exact run (elsewhere the EOS
returns zero, and predicting there says nothing about the method). The
fastest qualifying form is the headline.

One benchmark step is one run of that form from the initial state (200 time
steps: nodal update, element volume / gradient / viscosity, the EOS region
under the technique, energy update) plus its quality against the stored exact
result. `value` is element updates per second of the whole run (E x 200 per
step); `speedup_vs_exact` gives the run-level and EOS-region-level speedup
against the exact run on the same GPU; `roofline` covers the dominant kernel
(the element kernel) and `kernels` every exact kernel's roofline
fraction; `cpu_baseline` is the CPU oracle on a bounded sample of the same run.
Every other configuration (Black-Scholes at 65,536 and 2^24 options, the
64^3 hydro run, the batched knob sweep, the surrogate, Binomial Options,
K-Means, the LavaMD-style forces and the other added workloads) is a section
printed on its own line
before the final one, and the whole record is written to the --detail file
(by default _build/bench_detail.json at the repository root, which git
ignores).

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]

Under torchrun (N > 1) every rank runs an independent replica (the path has
no exchange between regions); `value` sums the ranks' element updates over the
slowest rank's time.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

from paper_2308_16877_gb300 import workloads as W  # noqa: E402

METRIC = "region elements/s and speedup vs exact kernel on 1 GB300 at <=1% quality loss"
GAMMA = 5.0 / 3.0

HEAD_N = 256                                    # headline mesh: 256^3 elements
HEAD_STEPS = 200
HYDRO_N = 64                                    # the 64^3 x 100-step configuration
HYDRO_STEPS = 100
HYDRO_IPT = 8                                   # EOS items per logical thread (kernel-scoped state)
QUALITY_BOUND = 0.01                            # <= 1% quality loss
MIN_ACTIVE_APPROX = 0.10                        # share of active invocations a headline form approximates
TAF = dict(hsize=4, psize=8, thresh=0.005, level=0)
IACT = dict(tsize=8, tperwarp=32, thresh=1e-3, level=0)
# iACT input normalisation: energy by the initial corner energy, relative
# volume as is, volume change by the CFL number, viscosity by the initial
# corner pressure.
IACT_SCALE = (1.0 / W.HYDRO_E0, 1.0, 10.0, 1.0 / ((GAMMA - 1.0) * W.HYDRO_E0))

# Candidate forms of the EOS region for the headline: (name, technique
# (1 TAF, 2 iACT), state kept across time steps, knobs). Kept state uses one
# logical thread per element (T = E), so a thread's window or a warp's tables
# follow the same elements from step to step; launch-scoped state uses
# T = E / 8 (8 elements per thread within a step).
HEAD_FORMS = [
    ("taf h4 p8 0.5%", 1, False, dict(hsize=4, psize=8, thresh=0.005, level=0)),
    ("iact t8 g32 1e-3", 2, False, dict(tsize=8, tperwarp=32, thresh=1e-3, level=0)),
    ("taf kept h2 p2 0.1%", 1, True, dict(hsize=2, psize=2, thresh=0.001, level=0)),
    ("taf kept h4 p8 0.5%", 1, True, dict(hsize=4, psize=8, thresh=0.005, level=0)),
    ("iact kept t8 g1 1e-3", 2, True, dict(tsize=8, tperwarp=1, thresh=1e-3, level=0)),
    ("iact kept t4 g4 1e-3", 2, True, dict(tsize=4, tperwarp=4, thresh=1e-3, level=0)),
    ("iact kept t2 g32 1e-4", 2, True, dict(tsize=2, tperwarp=32, thresh=1e-4, level=0)),
    ("iact kept t8 g32 1e-3", 2, True, dict(tsize=8, tperwarp=32, thresh=1e-3, level=0)),
]

# Bytes of the element kernel per element: the three coordinates of a node (a
# node per element), e, the relative volume, V0 and 1 / V0 read; 24 gradient
# values, the four EOS inputs and q written. Its gradients and volume run in
# 64-bit fixed point, so what bounds it is the issue of integer instructions
# (a rate no published peak covers) and its ceiling here is HBM.
ELEM_BYTES = 24 + 32 + 192 + 32 + 8
# The FP64 issue rate of the part, in FP64 instructions per lane per second
# (each add, multiply or FMA one): the nominal 1.25 TFLOP/s of GB300 at 152 SMs
# and 2070 MHz is 1.25e12 / (2 x 152 x 2.07e9) = 1.99, i.e. 2 FP64 FMA per SM
# per clock, taken at the SM count of the device and the median SM clock sampled
# under load. The FMA rate that the library's probe measures in the same run is
# reported beside it.
FP64_FMA_PER_SM_CLK = 2
# The node kernel's FP64 work per node: 24 corner-force FMAs and 6 for the
# velocity and position updates (30.4 measured per node, boundary nodes having
# fewer elements); it runs the FP64 pipe and HBM near their limits at once.
NODE_OPS = 30

BS_N = 1 << 24
BS_CFG0_N = 65536
BS_TAF = dict(hsize=4, psize=8, thresh=0.005, level=0)
BS_PERFO = dict(kind=0, m_or_percent=4, herded=True)
BS_IACT = dict(tsize=8, tperwarp=32, thresh=0.05, level=1)

KERNEL_SOURCES = {"map_kernel": ["exact_perfo.cu", "regions.cuh"], "taf_kernel": ["taf.cu", "regions.cuh"],
                  "iact_kernel": ["iact.cu", "regions.cuh"], "elem_kernel": ["hydro.cu"],
                  "node_kernel": ["hydro.cu"]}


def sig(x, k=4):
    """x rounded to k significant digits (floats), for the compact line."""
    if isinstance(x, float):
        return float(f"{x:.{k}g}") if np.isfinite(x) else None
    if isinstance(x, dict):
        return {a: sig(b, k) for a, b in x.items()}
    if isinstance(x, (list, tuple)):
        return [sig(b, k) for b in x]
    return x


def aggregate(total_ms, units_per_rank, world, device=None):
    """Whole-job throughput of `world` replicas: the slowest rank's time (max
    over ranks with an all-reduce when world > 1) and the units all ranks
    processed. Returns (max_ms, units per second)."""
    if world > 1:
        import torch
        import torch.distributed as dist
        t = torch.tensor([float(total_ms)], dtype=torch.float64, device=device)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        total_ms = float(t.item())
    return total_ms, world * units_per_rank / (total_ms * 1e-3)


def env_rank():
    return (int(os.environ.get("RANK", 0)), int(os.environ.get("WORLD_SIZE", 1)),
            int(os.environ.get("LOCAL_RANK", 0)))


class ClockSampler:
    """nvidia-smi samples of SM clock and throttle reasons while running."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index, self.proc, self.lines = index, None, []

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            threading.Thread(target=self._read, daemon=True).start()
        except Exception:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()

    def summary(self):
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for l in self.lines:
            f = [c.strip() for c in l.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx = float(f[2])
            except ValueError:
                continue
            for nm, v in zip(names, f[5:9]):
                if v.lower() == "active":
                    reasons.add(nm)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unsampled"], "samples": 0}
        return {"sm_mhz": float(np.median(sm)), "sm_max_mhz": mx, "reasons": sorted(reasons),
                "samples": len(sm)}


def source_digest(tag):
    h = hashlib.sha1()
    for f in KERNEL_SOURCES[tag.split("<")[0]]:
        with open(os.path.join(ROOT, "paper_2308_16877_gb300", "csrc", f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:12]


def dram_traffic(tag, units):
    """DRAM bytes (read + write) per launch from the ncu record in
    profiles/dram_traffic.txt (bytes per unit, scaled to `units`); None when
    the kernel's sources changed since the capture or no record exists."""
    p = os.path.join(ROOT, "profiles", "dram_traffic.txt")
    if not os.path.exists(p):
        return None
    for line in open(p):
        f = line.split()
        if len(f) >= 3 and not line.startswith("#") and f[0] == tag:
            return float(f[1]) * units if f[2] == source_digest(tag) else None
    return None


def measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        return float(d.get("hbm_gbs", 6800.0)), "measured"
    return 6800.0, "fallback"


def measured_hbm():
    return measured_peaks()


def timed_ms(torch, stream, f, reps):
    """Mean CUDA-event time of f() on `stream` over reps calls after one warm call."""
    f()
    torch.cuda.synchronize()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record(stream)
    for _ in range(reps):
        f()
    b.record(stream)
    torch.cuda.synchronize()
    return a.elapsed_time(b) / reps


# ---------------------------------------------------------------- CPU oracle

def form_oracle_knobs(oracle, form, n):
    """The oracle's EOS knobs for a headline form (None: exact)."""
    if form is None:
        return None
    name, tech, kept, kn = form
    E = n ** 3
    T = E if kept else E // HYDRO_IPT
    if tech == 1:
        return oracle.eos_knobs(oracle.EOS_TAF, hsize=kn["hsize"], psize=kn["psize"], thresh=kn["thresh"],
                                level=kn["level"], threads=T, block=256, persistent=kept, n=n)
    return oracle.eos_knobs(oracle.EOS_IACT, tsize=kn["tsize"], tperwarp=kn["tperwarp"], thresh=kn["thresh"],
                            level=kn["level"], threads=T, block=256, in_scale=IACT_SCALE, persistent=kept, n=n)


_INITIAL = {}                                   # initial meshes by size (generated once)


def hydro_cpu(form, n=HEAD_N, steps=4, single_steps=0):
    """The oracle on the same mesh and EOS form: `steps` time steps from the
    initial state (a bounded sample of the 200-step run); element updates per
    second on all host cores, and on one core for `single_steps` steps."""
    import oracle
    if n not in _INITIAL:
        _INITIAL[n] = W.hydro_initial(n)
    x, y, z, e = _INITIAL[n]
    dt = W.hydro_dt(n)
    E = n ** 3

    def timed(nsteps):
        S = oracle.HydroState(n, x, y, z, e)
        k = form_oracle_knobs(oracle, form, n)
        t0 = time.perf_counter()
        for _ in range(nsteps):
            S.step(dt, k)
        return time.perf_counter() - t0

    cores = oracle.num_threads()
    dt_s = timed(steps)
    label = form[0] if form is not None else "exact EOS"
    out = {"value": E * steps / dt_s, "unit": "elements/s", "cores": cores, "kind": "oracle",
           "sample": f"{n}^3, first {steps} steps", "seconds": dt_s}
    if single_steps:
        oracle.set_threads(1)
        try:
            t1 = timed(single_steps)
        finally:
            oracle.set_threads(cores)
        out["single_thread"] = {"value": E * single_steps / t1, "unit": "elements/s",
                                "sample": f"first {single_steps} time step(s), one core"}
    return out


def workload_name(n, time_steps, form):
    """The headline workload as the bench line's config names it."""
    return (f"hydro {n}^3, {time_steps} steps, EOS under {form} (fastest within 1% loss, "
            f">={MIN_ACTIVE_APPROX:.0%} of active calls approximated)")


def run_reference(args):
    """The reference arm: the CPU oracle (there is no reference implementation
    of this paper to install) on bounded samples of the headline workload."""
    rank, world, _ = env_rank()
    if rank != 0:
        return 0
    import oracle
    oracle.lib()
    form = next(f for f in HEAD_FORMS if f[0] == args.reference_form)
    times, per, cores = [], None, oracle.num_threads()
    for i in range(args.warmup + args.steps):
        cb = hydro_cpu(form, n=args.n, steps=1)
        per = args.n ** 3
        if i >= args.warmup:
            times.append(cb["seconds"])
    v = per * len(times) / sum(times)
    line = {"impl": "reference", "metric": METRIC, "value": v, "unit": "elements/s",
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * sum(times) / len(times), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": workload_name(args.n, args.time_steps, form[0]),
                       "l2": "inputs > L2 (6.5 GB state)", "parallelism": "oracle on host cores"},
            "cpu_baseline": {"value": v, "unit": "elements/s", "cores": cores, "kind": "oracle",
                             "sample": f"first time step of the {args.n}^3 run, {form[0]}"},
            "e2e": {"value": v, "unit": "elements/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line))
    return 0


# ---------------------------------------------------------------- GPU sections

def bench_blackscholes(hpac, torch, dev, stream, reps=20):
    """Single-precision Black-Scholes region passes on 2^24 options (inputs
    larger than L2): exact, perforation small:4, TAF, iACT."""
    n = BS_N
    T = n // 8
    xh = W.blackscholes_inputs(n)
    x = torch.from_numpy(xh).to(dev)
    sc = W.iact_scale(xh, n)
    out = {k: torch.zeros(n, dtype=torch.float32, device=dev) for k in ("exact", "perfo", "taf", "iact")}
    R = hpac.Region(hpac.HPAC_REGION_BLACKSCHOLES, x, param=W.BS_RATE, logical_threads=T,
                    block_threads=256, stream=stream)
    x64 = x.double().contiguous()
    ref = torch.zeros(n, dtype=torch.float64, device=dev)
    with hpac.Region(hpac.HPAC_REGION_BLACKSCHOLES, x64, param=W.BS_RATE, stream=stream) as R64:
        R64.run_exact(x64, ref)
    del x64
    calls = {"exact": lambda: R.run_exact(x, out["exact"]),
             "perfo": lambda: R.run_perfo(x, out["perfo"], BS_PERFO["kind"], BS_PERFO["m_or_percent"],
                                          herded=True),
             "taf": lambda: R.run_taf(x, out["taf"], **BS_TAF),
             "iact": lambda: R.run_iact(x, out["iact"], in_scale=sc, **BS_IACT)}
    ms = {}
    for k, f in calls.items():
        for _ in range(3):
            f()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(reps):
            f()
        e1.record(stream)
        torch.cuda.synchronize()
        ms[k] = e0.elapsed_time(e1) / reps
    stats = {"perfo": R.run_perfo(x, out["perfo"], 0, 4, herded=True, stats=True),
             "taf": R.run_taf(x, out["taf"], stats=True, **BS_TAF),
             "iact": R.run_iact(x, out["iact"], in_scale=sc, stats=True, **BS_IACT)}
    rms = float(torch.sqrt(torch.mean(ref * ref)).item())
    q = {k: {"mape": hpac.quality(ref, out[k], hpac.HPAC_METRIC_MAPE, stream=stream)["value"],
             "nrmse": hpac.quality(ref, out[k], hpac.HPAC_METRIC_RMSE, stream=stream)["value"] / rms}
         for k in out}
    peak, src = measured_hbm()
    gbs = 20 * n / (ms["exact"] * 1e-3) / 1e9
    R.close()
    return {"options": n, "pass_ms": ms, "speedup_vs_exact": {k: ms["exact"] / v for k, v in ms.items()},
            "exact_gbs": gbs, "exact_hbm_frac": gbs / peak, "hbm_peak_source": src,
            "kernel_row": {"bound": "hbm", "ms": ms["exact"], "bytes": 20 * n, "peak": peak * 1e9,
                           "unit": "B/s", "achieved": gbs * 1e9, "frac": gbs / peak},
            "quality": q, "approximated": stats,
            "note": "MAPE is dominated by options whose exact price is below single-precision "
                    "resolution; NRMSE = RMSE / RMS(exact price)"}


def bench_sweep(hpac, torch, dev, stream, baseline=True):
    """The batched knob sweep: 256 configurations x 32 Black-Scholes regions of
    2^12..2^22 options in one graph launch (autotuned schedule), against the
    same work as 8192 separate region-API runs each followed by its quality."""
    from paper_2308_16877_gb300 import autotune
    sizes = W.sweep_region_sizes()
    configs = W.sweep_configs()
    x, regions = W.sweep_inputs(sizes)
    xd = torch.from_numpy(x).to(dev)
    x64 = xd.double().contiguous()
    ref = torch.zeros(x.shape[1], dtype=torch.float64, device=dev)
    with hpac.Region(hpac.HPAC_REGION_BLACKSCHOLES, x64, param=W.BS_RATE, stream=stream) as R:
        R.run_exact(x64, ref)
    del x64
    make = lambda bt, bps, tb: hpac.Sweep(configs, regions, xd, ref, W.BS_RATE, bt, bps, tb, stream=stream)
    best, tune_ms = autotune.tune_sweep(make, regions, len(configs))
    sw = make(*best)
    sw.run()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    reps = 5
    e0.record(stream)
    for _ in range(reps):
        sw.run()
    e1.record(stream)
    torch.cuda.synchronize()
    graph_ms = e0.elapsed_time(e1) / reps
    res = sw.results()
    sw.close()
    work = len(configs) * int(sum(sizes))
    out = {"configs": len(configs), "regions": len(sizes), "options": int(sum(sizes)),
           "schedule": {"block_threads": best[0], "blocks_per_sm": best[1], "tile_blocks": best[2]},
           "tuner_evaluations": len(tune_ms), "tuner_worst_ms": max(tune_ms.values()),
           "graph_ms": graph_ms, "config_elements_per_s": work / (graph_ms * 1e-3),
           "approximated_total": int(res["approximated"].sum()), "skipped_total": int(res["skipped"].sum())}
    if baseline:
        # separate launches: one region call per (configuration, region) on a
        # column view of the concatenated inputs, then its quality
        regs = []
        for (n, off, T) in regions:
            xs = xd[:, off:off + n].contiguous()
            regs.append((hpac.Region(hpac.HPAC_REGION_BLACKSCHOLES, xs, param=W.BS_RATE,
                                     logical_threads=T, stream=stream), xs, ref[off:off + n].contiguous(),
                         torch.zeros(n, dtype=torch.float32, device=dev)))
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for cfg in configs:
            for R, xs, rs, o in regs:
                if cfg["tech"] == "taf":
                    R.run_taf(xs, o, cfg["hsize"], cfg["psize"], cfg["thresh"], 0)
                else:
                    o.zero_()
                    R.run_perfo(xs, o, cfg["kind"], cfg["m"], cfg.get("rate", 0.0), cfg.get("seed", 0),
                                bool(cfg["herded"]))
                hpac.quality(rs, o, hpac.HPAC_METRIC_MAPE, stream=stream)
        torch.cuda.synchronize()
        sep_s = time.perf_counter() - t0
        for R, *_ in regs:
            R.close()
        out.update({"separate_launches": len(configs) * len(regions), "separate_ms": sep_s * 1e3,
                    "separate_config_elements_per_s": work / sep_s,
                    "graph_speedup_vs_separate": sep_s * 1e3 / graph_ms})
    return out


def bench_search(hpac, torch, dev, stream, bound=0.01, reps=5):
    """Genetic knob search (population 32, 12 generations: 384 evaluations, one
    sweep launch per generation) against the exhaustive 256-configuration grid
    on the same 32 Black-Scholes regions: the best feasible saved share (TAF
    predictions + perforated invocations over all invocations at normalised
    RMSE <= bound) of each, and the measured speedup of each best configuration
    over the exact kernel through the region API, summed over the regions."""
    from paper_2308_16877_gb300 import search as S
    sizes = W.sweep_region_sizes()
    x, regions = W.sweep_inputs(sizes)
    xd = torch.from_numpy(x).to(dev)
    x64 = xd.double().contiguous()
    ref = torch.zeros(x.shape[1], dtype=torch.float64, device=dev)
    with hpac.Region(hpac.HPAC_REGION_BLACKSCHOLES, x64, param=W.BS_RATE, stream=stream) as R:
        R.run_exact(x64, ref)
    del x64
    t0 = time.perf_counter()
    ev = S.sweep_evaluator(hpac, regions, xd, ref, W.BS_RATE, stream=stream)
    best, best_r, hist = S.genetic_search(ev, bound=bound)
    torch.cuda.synchronize()
    search_s = time.perf_counter() - t0
    grid = W.sweep_configs()
    t0 = time.perf_counter()
    gev = S.sweep_evaluator(hpac, regions, xd, ref, W.BS_RATE, stream=stream)
    gres = gev(grid)
    grid_s = time.perf_counter() - t0
    gi = max(range(len(grid)), key=lambda i: S.score(*gres[i], bound))

    regs = []
    for (n, off, T) in regions:
        xs = xd[:, off:off + n].contiguous()
        regs.append((hpac.Region(hpac.HPAC_REGION_BLACKSCHOLES, xs, param=W.BS_RATE, logical_threads=T,
                                 stream=stream), xs, torch.zeros(n, dtype=torch.float32, device=dev)))

    def call(cfg):
        for R, xs, o in regs:
            if cfg is None:
                R.run_exact(xs, o)
            elif cfg["tech"] == "taf":
                R.run_taf(xs, o, cfg["hsize"], cfg["psize"], cfg["thresh"], 0)
            else:
                R.run_perfo(xs, o, cfg["kind"], cfg["m"], cfg.get("rate", 0.0), cfg.get("seed", 0),
                            bool(cfg["herded"]))

    def timed(cfg):
        call(cfg)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(reps):
            call(cfg)
        e1.record(stream)
        torch.cuda.synchronize()
        return e0.elapsed_time(e1) / reps

    exact_ms = timed(None)
    s_ms, g_ms = timed(best), timed(grid[gi])
    for R, *_ in regs:
        R.close()
    return {"bound_nrmse": bound, "evaluations": ev.calls["configs"], "launches": ev.calls["launches"],
            "search_s": search_s, "grid_s": grid_s,
            "search_best": {"config": best, "saved": best_r[0], "nrmse": best_r[1],
                            "speedup_vs_exact": exact_ms / s_ms},
            "grid_best": {"config": grid[gi], "saved": gres[gi][0], "nrmse": gres[gi][1],
                          "speedup_vs_exact": exact_ms / g_ms},
            "history_best_saved": hist, "exact_ms_all_regions": exact_ms}


def bench_binomial(hpac, torch, dev, stream, members=4096, time_points=64, steps=1024, reps=3):
    """Binomial Options (Table 1): a portfolio of American calls priced at
    successive time points on 1024-step trees, one option per team of 32
    lanes, one team per member (T = members). TAF and iACT decide per team
    (the paper's block level), perforation drops whole options; each
    configuration is timed against the exact kernel and scored by the MAPE of
    its prices against the exact ones (the paper's highest speedup at a
    quality bound)."""
    x = W.binomial_portfolio(members, time_points)
    n = x.shape[1]
    xd = torch.from_numpy(x).to(dev)
    sc = W.iact_scale(x, n)
    exact = torch.zeros(n, dtype=torch.float32, device=dev)
    out = torch.zeros(n, dtype=torch.float32, device=dev)
    R = hpac.Region(hpac.HPAC_REGION_BINOMIAL, xd, param=W.BS_RATE, arg=steps, logical_threads=members,
                    stream=stream)

    def timed(f):
        f()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(reps):
            f()
        e1.record(stream)
        torch.cuda.synchronize()
        return e0.elapsed_time(e1) / reps

    exact_ms = timed(lambda: R.run_exact(xd, exact))
    ref = exact.double()
    rows = []

    def add(tech, knobs, f):
        ms = timed(f)
        mape = hpac.quality(ref, out, hpac.HPAC_METRIC_MAPE, stream=stream)["value"]
        rows.append(dict(technique=tech, **knobs, ms=ms, speedup=exact_ms / ms, mape=mape))

    for h in (1, 2, 4):
        for p in (2, 4, 8, 16):
            for thr in (0.005, 0.01, 0.02, 0.05):
                add("taf", dict(h=h, p=p, thr=thr),
                    lambda: R.run_taf(xd, out, h, p, thr, hpac.HPAC_LEVEL_BLOCK))
    for ts in (4, 8):
        for thr in (0.005, 0.01, 0.02, 0.05):
            add("iact", dict(tsize=ts, thr=thr),
                lambda: R.run_iact(xd, out, ts, 32, thr, hpac.HPAC_LEVEL_BLOCK, in_scale=sc))
    for m in (2, 3, 4, 8):
        def perf(m=m):
            out.zero_()                # a dropped option keeps the caller's (zero) prefill
            R.run_perfo(xd, out, hpac.HPAC_PERFO_SMALL, m, herded=True)
        add("perfo_small", dict(m=m), perf)
    R.close()

    def best(tech_prefix, bound):
        ok = [r for r in rows if r["technique"].startswith(tech_prefix) and r["mape"] <= bound]
        return max(ok, key=lambda r: r["speedup"]) if ok else None

    # the exact kernel against the FP32 issue rate: 5 single-precision
    # instructions per node update (multiply, fused multiply-add, multiply,
    # subtract, max), N (N + 1) / 2 updates per option
    instr = 5.0 * steps * (steps + 1) / 2 * n
    peak = 152 * 128 * 2.07e9
    return {"options": n, "members": members, "time_points": time_points, "steps": steps,
            "exact_ms": exact_ms, "options_per_s": n / (exact_ms * 1e-3),
            "exact_fp32_issue_frac": instr / (exact_ms * 1e-3) / peak,
            "best_at_1pct_mape": {t: best(t, 0.01) for t in ("taf", "iact", "perfo")},
            "best_at_10pct_mape": {t: best(t, 0.10) for t in ("taf", "iact", "perfo")},
            "table": rows}


def bench_kmeans(hpac, torch, dev, stream, n=1 << 22, clusters=16, max_iter=300):
    """K-Means (Table 1; the distance kernel is the approximated region,
    Section 4.2): 4M observations of 8 features from 16 overlapping blobs,
    started from the first 16 observations, iterated until no observation
    changes cluster. Exact, TAF and iACT with kernel-scoped state (T = N/8),
    TAF and iACT with state kept across iterations (T = N: one logical thread
    per observation, so a window holds that observation's recent ids), and
    herded perforation (a skipped observation keeps its previous id). Reported:
    iterations, time to convergence (assignment + update + the changed-count
    read every iteration), and MCR of the final ids against the exact run's."""
    x, labels, _ = W.kmeans_blobs(n, clusters, spread=2.0)
    xd = torch.from_numpy(x).to(dev)
    init = torch.from_numpy(np.ascontiguousarray(x[:, :clusters].T)).to(dev)
    sc = W.iact_scale(x, n)
    work = hpac.kmeans_workspace(clusters, dev)
    cent = init.clone()
    a = torch.zeros(n, dtype=torch.float32, device=dev)
    prev = torch.zeros(n, dtype=torch.float32, device=dev)
    regions = {T: hpac.Region(hpac.HPAC_REGION_KMEANS, xd, arg=clusters, logical_threads=T,
                              block_threads=256, stream=stream) for T in (n // 8, n)}
    for R in regions.values():
        R.set_aux(cent)
    variants = {
        "exact": (n // 8, False, lambda R: R.run_exact(xd, a)),
        "taf_h2p4": (n // 8, False, lambda R: R.run_taf(xd, a, 2, 4, 0.01, 0)),
        "taf_persistent_h2p4": (n, True, lambda R: R.run_taf(xd, a, 2, 4, 0.01, 0)),
        "taf_persistent_h3p8": (n, True, lambda R: R.run_taf(xd, a, 3, 8, 0.01, 0)),
        "taf_persistent_h8p1": (n, True, lambda R: R.run_taf(xd, a, 8, 1, 0.01, 0)),
        "iact_t8": (n // 8, False, lambda R: R.run_iact(xd, a, 8, 32, 0.02, 0, in_scale=sc)),
        "iact_persistent_t4": (n, True, lambda R: R.run_iact(xd, a, 4, 32, 0.01, 0, in_scale=sc)),
        "perfo_small2": (n // 8, False, lambda R: R.run_perfo(xd, a, hpac.HPAC_PERFO_SMALL, 2, herded=True)),
        "perfo_small4": (n // 8, False, lambda R: R.run_perfo(xd, a, hpac.HPAC_PERFO_SMALL, 4, herded=True)),
    }
    res, ref = {}, None
    for name, (T, persist, run) in variants.items():
        R = regions[T]
        for rep in range(2):                           # the first run warms up
            cent.copy_(init)
            a.zero_()
            R.set_persistent(persist)
            R.reset_state()
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            for it in range(1, max_iter + 1):
                run(R)
                ch = hpac.kmeans_update(xd, a, cent, work, prev=prev if it > 1 else None, stream=stream)
                if it > 1 and ch == 0:
                    break
                prev.copy_(a)
            torch.cuda.synchronize()
            ms = (time.perf_counter() - t0) * 1e3
        row = {"iterations": it, "ms": ms, "converged": it < max_iter}
        if name == "exact":
            ref = a.clone()
        else:
            row["mcr_vs_exact"] = hpac.quality(ref.double(), a, hpac.HPAC_METRIC_MCR, stream=stream)["value"]
            row["speedup_vs_exact"] = res["exact"]["ms"] / ms
            row["convergence_speedup"] = res["exact"]["iterations"] / it
        res[name] = row
        R.set_persistent(False)
    for R in regions.values():
        R.close()
    return {"observations": n, "features": 8, "clusters": clusters, "runs": res}


def bench_levels(hpac, torch, dev, stream, n=1 << 22, clusters=64, reps=5):
    """Decision hierarchy (Section 3.3; the paper's Fig. 7 contrast): the
    K-Means assignment region (64 centroids, ~1.5 k instructions per call) on
    observations whose logical threads each follow one cluster with 5%
    outliers from random clusters, T = N/16. TAF and iACT at thread, warp and
    block level against the exact region: time, share approximated and MCR of
    the ids. At thread level an outlier lane makes its whole warp run the
    distance loop; warp and block majorities keep the group together."""
    T = n // 16
    x, labels, cent = W.kmeans_coherent(n, clusters, T)
    xd = torch.from_numpy(x).to(dev)
    cd = torch.from_numpy(cent).to(dev)
    sc = W.iact_scale(x, n)
    out = torch.zeros(n, dtype=torch.float32, device=dev)
    exact = torch.zeros(n, dtype=torch.float32, device=dev)
    R = hpac.Region(hpac.HPAC_REGION_KMEANS, xd, arg=clusters, logical_threads=T, block_threads=256,
                    stream=stream)
    R.set_aux(cd)

    def timed(f):
        f()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(reps):
            f()
        e1.record(stream)
        torch.cuda.synchronize()
        return e0.elapsed_time(e1) / reps

    exact_ms = timed(lambda: R.run_exact(xd, exact))
    ref = exact.double()
    rows = []
    for tech in ("taf", "iact"):
        for level in (hpac.HPAC_LEVEL_THREAD, hpac.HPAC_LEVEL_WARP, hpac.HPAC_LEVEL_BLOCK):
            if tech == "taf":
                f = lambda: R.run_taf(xd, out, 2, 8, 0.01, level)
                st = R.run_taf(xd, out, 2, 8, 0.01, level, stats=True)
            else:
                f = lambda: R.run_iact(xd, out, 8, 32, 0.3, level, in_scale=sc)
                st = R.run_iact(xd, out, 8, 32, 0.3, level, in_scale=sc, stats=True)
            mcr = hpac.quality(ref, out, hpac.HPAC_METRIC_MCR, stream=stream)["value"]
            ms = timed(f)
            rows.append({"technique": tech, "level": ["thread", "warp", "block"][level], "ms": ms,
                         "speedup_vs_exact": exact_ms / ms, "approximated": st["approximated"] / n,
                         "mcr": mcr})
    R.close()
    return {"region": "K-Means assignment, 64 centroids", "observations": n, "logical_threads": T,
            "knobs": {"taf": "h2 p8 0.01", "iact": "t8 private tables, distance 0.3 (scaled)"},
            "exact_ms": exact_ms, "table": rows}


# FP64 operations of one LavaMD pair term outside the exponential: three
# differences, r^2 (a multiply and two FMAs), the exponent's scaling, q v,
# 2 q v, the potential's add and three force FMAs.
LAVAMD_PAIR_FP64_OPS = 13
# FP64 instructions the exact kernel executes per pair term: q v and the four
# sums. The differences, their squares and the exponential run in fixed point
# on the integer pipes.
LAVAMD_PAIR_FP64_INSTR = 5


def bench_lavamd(hpac, torch, dev, stream, boxes1d=16, reps=3):
    """LavaMD-style neighbour-box forces (Table 1; Section 5 approximates the
    force calculation for a neighbouring box, Figure 9): 16^3 boxes of 100
    particles, FP64. The exact run, TAF (h4 p8) and iACT (8 slots, tables shared
    by 32 or 8 lanes) at thread, warp and block level: time, share of the
    invocations approximated, potential MAPE and force NRMSE against the exact
    run. Warp- and block-level decisions keep a warp (or the box's block) on
    one path, where thread-level decisions leave the warp running the pair loop
    for any lane that computes."""
    B, NP = boxes1d, W.LAVAMD_PAR_PER_BOX
    rq = torch.from_numpy(W.lavamd_inputs(B, NP)).to(dev)
    P = rq.shape[1]
    ex = torch.empty_like(rq)
    out = torch.empty_like(rq)

    def timed(f):
        f()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(reps):
            f()
        e1.record(stream)
        torch.cuda.synchronize()
        return e0.elapsed_time(e1) / reps

    def run(**kn):
        return hpac.lavamd(rq, B, NP, W.LAVAMD_A2, fv=out, stream=stream, **kn)

    exact_ms = timed(lambda: hpac.lavamd(rq, B, NP, W.LAVAMD_A2, fv=ex, stream=stream))
    _, st = hpac.lavamd(rq, B, NP, W.LAVAMD_A2, fv=ex, stats=True, stream=stream)
    inv = st["invocations"]
    pairs = inv * NP
    f_ex = ex[1:].contiguous()
    f_rms = float(torch.sqrt(torch.mean(f_ex * f_ex)).item())
    fp64 = hpac.hpac_device_fp64_rate(stream.cuda_stream)
    rows = []
    forms = [("taf", dict(technique=hpac.LAVAMD_TAF, hsize=4, psize=8, thresh=t), f"h4 p8 {t}") for t in (0.02, 0.04)]
    forms += [("iact", dict(technique=hpac.LAVAMD_IACT, tsize=8, tperwarp=g, thresh=0.05), f"t8 g{g} 0.05")
              for g in (1, 4)]
    for tech, kn, label in forms:
        for level in (hpac.HPAC_LEVEL_THREAD, hpac.HPAC_LEVEL_WARP, hpac.HPAC_LEVEL_BLOCK):
            _, st = run(level=level, stats=True, **kn)
            mape = hpac.quality(ex[0].contiguous(), out[0].contiguous(), hpac.HPAC_METRIC_MAPE,
                                stream=stream)["value"]
            rmse = hpac.quality(f_ex, out[1:].contiguous(), hpac.HPAC_METRIC_RMSE, stream=stream)["value"]
            ms = timed(lambda: run(level=level, **kn))
            rows.append({"technique": tech, "knobs": label, "level": ["thread", "warp", "block"][level],
                         "ms": ms, "speedup_vs_exact": exact_ms / ms,
                         "approximated": st["approximated"] / inv,
                         "potential_mape": mape, "force_nrmse": rmse / f_rms})
    within = [r for r in rows if r["potential_mape"] <= QUALITY_BOUND]
    best = max(within, key=lambda r: r["speedup_vs_exact"]) if within else None
    ops = LAVAMD_PAIR_FP64_OPS * pairs / (exact_ms * 1e-3)
    instr = LAVAMD_PAIR_FP64_INSTR * pairs / (exact_ms * 1e-3)
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    peak = FP64_FMA_PER_SM_CLK * sms * 2070e6
    return {"boxes": f"{B}^3", "particles": P, "par_per_box": NP, "invocations": inv,
            "pair_terms": pairs, "exact_ms": exact_ms, "exact_pairs_per_s": pairs / (exact_ms * 1e-3),
            "exact_fp64_ops_outside_exp_per_s": ops,
            "roofline": {"bound": "alu", "unit": "T FP64-instr/s", "achieved": instr / 1e12,
                         "peak": peak / 1e12, "frac": instr / peak,
                         "peak_source": f"derived: {FP64_FMA_PER_SM_CLK} FP64 FMA/SM/clk x {sms} SMs x 2070 MHz",
                         "frac_of_measured_fma": instr / (fp64 / 2.0 * 1e12),
                         "instr_per_pair": LAVAMD_PAIR_FP64_INSTR},
            "table": rows, "fastest_within_1pct_potential_mape": best}


def bench_surrogate(hpac, torch, dev, stream, n_train=1 << 22, n_cal=1 << 20, n_inf=1 << 24,
                    epochs=24, batch=8192, lr=3e-3):
    """The learned surrogate of the Black-Scholes region: trained by the
    library's kernels on 4M exact pairs, calibrated on 1M held-out options,
    inference on 16M options with the exact fallback below the calibrated
    price, against the exact kernel and TAF on the same options."""
    def exact(x, dtype):
        out = torch.zeros(x.shape[1], dtype=dtype, device=dev)
        xx = x if dtype == torch.float32 else x.double().contiguous()
        with hpac.Region(hpac.HPAC_REGION_BLACKSCHOLES, xx, param=W.BS_RATE, stream=stream) as R:
            R.run_exact(xx, out)
        return out
    xt = torch.from_numpy(W.blackscholes_inputs(n_train, seed=31)).to(dev)
    xc = torch.from_numpy(W.blackscholes_inputs(n_cal, seed=32)).to(dev)
    xi = torch.from_numpy(W.blackscholes_inputs(n_inf, seed=33)).to(dev)
    yt = exact(xt, torch.float32)
    desc = hpac.blackscholes_desc(64)
    S = hpac.Surrogate(desc, seed=2308, stream=stream)
    S.fit_normalization(xt, yt, W.BS_RATE)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    loss = S.train(xt, yt, W.BS_RATE, batch=batch, epochs=epochs, lr=lr)
    e1.record(stream)
    torch.cuda.synchronize()
    train_ms = e0.elapsed_time(e1)
    # calibration
    pc = torch.zeros(n_cal, dtype=torch.float32, device=dev)
    S.infer(xc, pc, W.BS_RATE)
    yc = exact(xc, torch.float64)
    tau, kept = hpac.calibrate_floor(pc, yc, 0.01, 0.99, stream=stream)
    # inference with fallback vs the exact kernel
    out = torch.zeros(n_inf, dtype=torch.float32, device=dev)
    mask = torch.zeros(n_inf, dtype=torch.uint8, device=dev)
    st = S.infer(xi, out, W.BS_RATE, fallback_below=tau, mask=mask, stats=True)
    def timed(f, reps=10):
        f()
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        for _ in range(reps):
            f()
        b.record(stream)
        torch.cuda.synchronize()
        return a.elapsed_time(b) / reps
    ex32 = torch.zeros(n_inf, dtype=torch.float32, device=dev)
    with hpac.Region(hpac.HPAC_REGION_BLACKSCHOLES, xi, param=W.BS_RATE, logical_threads=n_inf // 8,
                     stream=stream) as R:
        exact_ms = timed(lambda: R.run_exact(xi, ex32))
        taf_out = torch.zeros(n_inf, dtype=torch.float32, device=dev)
        taf_stats = R.run_taf(xi, taf_out, 4, 8, 0.005, 0, stats=True)
    sur_ms = timed(lambda: S.infer(xi, out, W.BS_RATE, fallback_below=tau, mask=mask))
    nofb_ms = timed(lambda: S.infer(xi, out, W.BS_RATE))
    # input derivatives (the input half of a vector-Jacobian product) on the same options
    gin = torch.zeros(4, n_inf, dtype=torch.float32, device=dev)
    igrad_ms = timed(lambda: S.input_grad(xi, gin, W.BS_RATE))
    del gin
    S.infer(xi, out, W.BS_RATE, fallback_below=tau, mask=mask)
    ref = exact(xi, torch.float64)
    o, r, m = out.cpu().numpy().astype(np.float64), ref.cpu().numpy(), mask.cpu().numpy()
    rel = np.abs(o - r) / np.maximum(np.abs(r), 1e-30)
    rms = float(np.sqrt(np.mean(r * r)))
    tafo = taf_out.cpu().numpy().astype(np.float64)
    approx = m == 1
    # tensor work: layer 2 (H x H) per sample on the tensor cores
    flops = 2.0 * desc.hidden * desc.hidden * n_inf
    S.close()
    return {
        "train": {"pairs": n_train, "epochs": epochs, "batch": batch, "ms": train_ms,
                  "samples_per_s": n_train * epochs / (train_ms * 1e-3), "final_mse_normalized": loss},
        "calibrated_floor": tau, "calibration_served": kept / n_cal,
        "inference": {"options": n_inf, "ms": sur_ms, "ms_without_fallback": nofb_ms,
                      "exact_kernel_ms": exact_ms, "speedup_vs_exact": exact_ms / sur_ms,
                      "surrogate_fraction": st["approximated"] / n_inf,
                      "layer2_tensor_tflops": flops / (nofb_ms * 1e-3) / 1e12},
        "input_gradient": {"options": n_inf, "ms": igrad_ms,
                           "tensor_tflops": 2 * flops / (igrad_ms * 1e-3) / 1e12},
        "quality": {"nrmse": float(np.sqrt(np.mean((o - r) ** 2)) / rms),
                    "p99_rel_err_on_surrogate_outputs": float(np.quantile(rel[approx], 0.99)) if approx.any() else None,
                    "max_rel_err_on_surrogate_outputs": float(rel[approx].max()) if approx.any() else None},
        "vs_taf_same_options": {"taf_fraction_approximated": taf_stats["approximated"] / n_inf,
                                "taf_nrmse": float(np.sqrt(np.mean((tafo - r) ** 2)) / rms)},
    }


def eos_region_sweep(hpac, torch, stream, eos_h, eos_in, ref, scale_arr, n_configs=64):
    """EOS knob sweep on one state (region only): 32 TAF configurations
    (threshold 1e-4 .. 1e-1, h 2/4, p 4/16, thread/warp level) and 32 iACT
    ones (threshold 1e-4 .. 1e-1, 1/2/16/32 tables per warp, thread/warp
    level), each timed against the exact call and scored by the pressure NRMSE
    against `ref` (the exact pressures of this state); the fastest within 1%."""
    E = ref.numel()
    eos_ptr = hpac.C.c_void_p(eos_in.data_ptr())
    outp = torch.zeros(E, dtype=torch.float64, device=ref.device)
    o_ptr = hpac.C.c_void_p(outp.data_ptr())

    def timed(f, reps=5):
        f()
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        for _ in range(reps):
            f()
        b.record(stream)
        torch.cuda.synchronize()
        return a.elapsed_time(b) / reps
    t_exact = timed(lambda: hpac.hpac_run_exact(eos_h, eos_ptr, o_ptr))
    rms = torch.sqrt(torch.mean(ref * ref)).item()
    table = []
    cfgs = []
    for thr in (1e-4, 1e-3, 1e-2, 1e-1):
        for h in (2, 4):
            for pz in (4, 16):
                for lv in (0, 1):
                    cfgs.append(("taf", hpac.hpac_taf_knobs(h, pz, thr, lv, 0), dict(h=h, p=pz, thr=thr, level=lv)))
    for thr in (1e-4, 1e-3, 1e-2, 1e-1):
        for g in (32, 16, 2, 1):
            for ts in (8,):
                for lv in (0, 1):
                    cfgs.append(("iact", hpac.hpac_iact_knobs(ts, g, thr, lv, 0, hpac.C.cast(
                        scale_arr, hpac.C.POINTER(hpac.C.c_double))), dict(tsize=ts, tperwarp=g, thr=thr, level=lv)))
    for kind, k, info in cfgs[:n_configs]:
        fn = (lambda k=k: hpac.hpac_run_taf(eos_h, k, eos_ptr, o_ptr)) if kind == "taf" else \
             (lambda k=k: hpac.hpac_run_iact(eos_h, k, eos_ptr, o_ptr))
        tm = timed(fn)
        err = torch.sqrt(torch.mean((outp - ref) ** 2)).item() / rms
        table.append(dict(technique=kind, **info, speedup=t_exact / tm, p_nrmse=err))
    ok = [r for r in table if r["p_nrmse"] <= 0.01]
    best = max(ok, key=lambda r: r["speedup"]) if ok else None
    return {"configs": len(table), "exact_region_ms": t_exact, "best_within_1pct": best, "table": table}


def bench_persistent(hpac, torch, dev, stream, n=HYDRO_N, nsteps=HYDRO_STEPS, reps=3):
    """Approximation state kept across time steps (TAF windows, iACT tables in
    device memory owned by the EOS region): hydro at n^3 for nsteps with one
    logical thread per element, so a thread's window holds its own element's
    last accurate pressures and a warp's tables its 32 elements' recent
    states. Kernel-scoped state cannot approximate here (one invocation per
    thread per launch); the persistent runs are compared with the exact run."""
    E = n ** 3
    sh = stream.cuda_stream
    x, y, z, e = W.hydro_initial(n)
    Hy = hpac.Hydro(n, x, y, z, e, W.hydro_dt(n), logical_threads=E, block_threads=256, stream=stream)
    torch.cuda.synchronize()
    init = {k: v.clone() for k, v in Hy.t.items()}
    scale_arr = (hpac.C.c_double * 4)(*IACT_SCALE)
    variants = {
        "exact": (hpac.HYDRO_EXACT, None, False),
        "taf_kernel_scoped": (hpac.HYDRO_TAF, hpac.hpac_taf_knobs(4, 8, 0.005, 0, 0), False),
        "taf_persistent": (hpac.HYDRO_TAF, hpac.hpac_taf_knobs(4, 8, 0.005, 0, 0), True),
        "taf_persistent_h2p4": (hpac.HYDRO_TAF, hpac.hpac_taf_knobs(2, 4, 0.005, 0, 0), True),
        "iact_kernel_scoped": (hpac.HYDRO_IACT, hpac.hpac_iact_knobs(
            8, 32, 1e-3, 0, 0, hpac.C.cast(scale_arr, hpac.C.POINTER(hpac.C.c_double))), False),
        "iact_persistent": (hpac.HYDRO_IACT, hpac.hpac_iact_knobs(
            8, 32, 1e-3, 0, 0, hpac.C.cast(scale_arr, hpac.C.POINTER(hpac.C.c_double))), True),
    }

    def reset(persist):
        for k, v in init.items():
            Hy.t[k].copy_(v, non_blocking=True)
        Hy.eos.set_persistent(persist)
        Hy.eos.reset_state()

    res = {}
    ref_p = ref_q = None
    for name, (tech, kn, persist) in variants.items():
        times = []
        for r in range(reps + 1):
            reset(persist)
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            hpac.hpac_hydro_run(Hy.state, Hy.eos._h, nsteps, tech, kn)
            e1.record(stream)
            torch.cuda.synchronize()
            if r > 0:
                times.append(e0.elapsed_time(e1))
        p_fin, q_fin = Hy["p"].clone(), float(Hy["e"][0].item())
        # approximation count: the same run with per-step counters (untimed)
        reset(persist)
        apx = 0
        for s in range(nsteps):
            st = hpac.hpac_hydro_step(Hy.state, Hy.eos._h, tech, kn, None, tech != hpac.HYDRO_EXACT)
            apx += st.approximated if st is not None else 0
        ms = float(np.median(times))
        row = {"ms": ms, "approximated_fraction": apx / (E * nsteps)}
        if name == "exact":
            ref_p, ref_q = p_fin, q_fin
        else:
            rms = float(torch.sqrt(torch.mean(ref_p * ref_p)).item())
            row["speedup_vs_exact"] = res["exact"]["ms"] / ms
            row["qoi_rel_err"] = abs(q_fin - ref_q) / abs(ref_q)
            row["p_nrmse"] = hpac.quality(ref_p, p_fin, hpac.HPAC_METRIC_RMSE, stream=stream)["value"] / rms
        res[name] = row
    Hy.eos.set_persistent(False)
    Hy.close()
    return {"mesh": f"{n}^3", "time_steps": nsteps, "logical_threads": E,
            "knobs": {"taf": "h4 p8 0.5% (and h2 p4)", "iact": "t8 g32 1e-3 scaled"}, "runs": res}




def graph_ms(torch, R, stream, f, reps):
    """Per-call time of f() as `reps` calls captured in one CUDA graph and
    replayed (the region's stream set to the capturing stream); None if the
    capture fails."""
    side = torch.cuda.Stream()
    try:
        R.set_stream(side)
        with torch.cuda.stream(side):
            f()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            for _ in range(reps):
                f()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        with torch.cuda.stream(side):      # replay() launches on the current stream
            g.replay()
            a.record()
            g.replay()
            b.record()
        torch.cuda.synchronize()
        return a.elapsed_time(b) / reps
    except Exception:
        torch.cuda.synchronize()
        return None
    finally:
        R.set_stream(stream)


def bench_blackscholes_cfg0(hpac, torch, dev, stream, n=BS_CFG0_N, reps=200):
    """The 65,536-option Black-Scholes configuration: exact, herded
    perforation small:4 and TAF (h4 p8 0.5%) at T = N / 8, each timed over 200
    back-to-back launches and as 200 calls captured in one CUDA graph and
    replayed (the 1.3 MB working set stays in L2, so these are launch- and
    L2-bound figures), with the MAPE and NRMSE against the
    double-precision exact prices. Two readings of "sorted by strike in runs
    of 32": each aligned run of 32 consecutive options sorted (the lanes of one
    warp step see ascending strikes), and the same runs laid along one logical
    thread's sequence (T = N / 32, thread t's 32 invocations are run t), which
    gives TAF the temporal order the configuration describes."""
    xh = W.blackscholes_inputs(n)
    T32 = n // 32
    layouts = {"runs_across_lanes": (xh, n // 8),
               "runs_along_threads": (np.ascontiguousarray(xh.reshape(4, T32, 32).transpose(0, 2, 1).reshape(4, n)),
                                      T32)}
    res = {}
    for name, (xa, T) in layouts.items():
        x = torch.from_numpy(xa).to(dev)
        x64 = x.double().contiguous()
        ref = torch.zeros(n, dtype=torch.float64, device=dev)
        with hpac.Region(hpac.HPAC_REGION_BLACKSCHOLES, x64, param=W.BS_RATE, stream=stream) as R64:
            R64.run_exact(x64, ref)
        rms = float(torch.sqrt(torch.mean(ref * ref)).item())
        outs = {k: torch.zeros(n, dtype=torch.float32, device=dev) for k in ("exact", "perfo", "taf")}
        R = hpac.Region(hpac.HPAC_REGION_BLACKSCHOLES, x, param=W.BS_RATE, logical_threads=T,
                        block_threads=256, stream=stream)
        calls = {"exact": lambda: R.run_exact(x, outs["exact"]),
                 "perfo": lambda: R.run_perfo(x, outs["perfo"], BS_PERFO["kind"], BS_PERFO["m_or_percent"],
                                              herded=True),
                 "taf": lambda: R.run_taf(x, outs["taf"], **BS_TAF)}
        ms = {k: timed_ms(torch, stream, f, reps) for k, f in calls.items()}
        graph = {k: graph_ms(torch, R, stream, f, reps) for k, f in calls.items()}
        st = {"perfo": R.run_perfo(x, outs["perfo"], 0, 4, herded=True, stats=True),
              "taf": R.run_taf(x, outs["taf"], stats=True, **BS_TAF)}
        R.close()
        q = {k: {"mape": hpac.quality(ref, outs[k], hpac.HPAC_METRIC_MAPE, stream=stream)["value"],
                 "nrmse": hpac.quality(ref, outs[k], hpac.HPAC_METRIC_RMSE, stream=stream)["value"] / rms}
             for k in outs}
        res[name] = {"logical_threads": T, "launch_ms": ms, "graph_replay_ms": graph,
                     "speedup_vs_exact": {k: ms["exact"] / v for k, v in ms.items()},
                     "approximated": {k: v["approximated"] / n for k, v in st.items()},
                     "skipped": st["perfo"]["skipped"] / n, "quality": q,
                     "exact_options_per_s": n / (ms["exact"] * 1e-3)}
    hbm, _ = measured_peaks()
    ex = res["runs_across_lanes"]["graph_replay_ms"]["exact"] or res["runs_across_lanes"]["launch_ms"]["exact"]
    return {"options": n, "layouts": res,
            "kernel_row": {"bound": "hbm", "ms": ex, "bytes": 20 * n, "peak": hbm * 1e9, "unit": "B/s",
                           "achieved": 20 * n / (ex * 1e-3), "frac": 20 * n / (ex * 1e-3) / (hbm * 1e9),
                           "note": "1.3 MB working set: L2-resident and launch-bound (graph replay)"}}


# ---------------------------------------------------------------- headline

class HydroBench:
    """The hydro state at one mesh size with two EOS regions: launch-scoped
    state (T = E / 8) and state kept across time steps (T = E)."""

    def __init__(self, hpac, torch, dev, stream, n, nsteps, seed):
        self.hpac, self.torch, self.stream, self.sh = hpac, torch, stream, stream.cuda_stream
        self.n, self.nsteps, self.E = n, nsteps, n ** 3
        self.x, self.y, self.z, self.e = W.hydro_initial(n, seed=seed)
        self.dt = W.hydro_dt(n)
        self.Hy = hpac.Hydro(n, self.x, self.y, self.z, self.e, self.dt, logical_threads=self.E // HYDRO_IPT,
                             block_threads=256, stream=stream)
        self.kept = hpac.Region(hpac.HPAC_REGION_EOS, self.Hy["eos_in"], param=GAMMA, logical_threads=self.E,
                                block_threads=256, stream=stream)
        torch.cuda.synchronize()
        self.init = {k: v.clone() for k, v in self.Hy.t.items()}
        self.scale = (hpac.C.c_double * 4)(*IACT_SCALE)
        # the end-to-end run's host side, allocated once up front as a caller
        # would: pinned copies of the initial mesh and a pinned buffer for the
        # final energies
        self.pin = {k: torch.from_numpy(np.ascontiguousarray(v)).pin_memory() for k, v in
                    (("x", self.x), ("y", self.y), ("z", self.z), ("e", self.e))}
        self.e_out = torch.empty(self.E, dtype=torch.float64).pin_memory()
        self.eos_ptr = hpac.C.c_void_p(self.Hy["eos_in"].data_ptr())
        self.p_ptr = hpac.C.c_void_p(self.Hy["p"].data_ptr())

    def knobs(self, form):
        hp = self.hpac
        name, tech, kept, kn = form
        if tech == 1:
            return hp.hpac_taf_knobs(kn["hsize"], kn["psize"], kn["thresh"], kn["level"], 0)
        return hp.hpac_iact_knobs(kn["tsize"], kn["tperwarp"], kn["thresh"], kn["level"], 0,
                                  hp.C.cast(self.scale, hp.C.POINTER(hp.C.c_double)))

    def region(self, form):
        return self.kept if (form is not None and form[2]) else self.Hy.eos

    def reset(self, form):
        for k, v in self.init.items():
            self.Hy.t[k].copy_(v, non_blocking=True)
        self.Hy.eos.set_persistent(False)
        if form is not None and form[2]:
            self.kept.set_persistent(True)
            self.kept.reset_state()
        else:
            self.kept.set_persistent(False)

    def run(self, form, elem_ev=None, region_ev=None, mask=None, count=None, record=None):
        """One run from the initial state. elem_ev / region_ev: lists of event
        pairs (one per time step) around the element kernel / the region call;
        record: a list that receives, per time step, the indices of the
        elements whose EOS input carries energy; mask + count (with the exact
        run's record as count[3]): per-step counts of those elements and of
        the ones this run approximates."""
        hp, sh = self.hpac, self.sh
        self.reset(form)
        R = self.region(form)
        k = self.knobs(form) if form is not None else None
        tech = form[1] if form is not None else 0
        st = self.stream
        for s in range(self.nsteps):
            hp.hpac_hydro_nodes(self.Hy.state, sh)
            if elem_ev is not None:
                elem_ev[s][0].record(st)
            hp.hpac_hydro_elements(self.Hy.state, sh)
            if elem_ev is not None:
                elem_ev[s][1].record(st)
            if region_ev is not None:
                region_ev[s][0].record(st)
            m = hp.C.c_void_p(mask.data_ptr()) if mask is not None else None
            if tech == 0:
                hp.hpac_run_exact(R._h, self.eos_ptr, self.p_ptr)
            elif tech == 1:
                hp.hpac_run_taf(R._h, k, self.eos_ptr, self.p_ptr, m)
            else:
                hp.hpac_run_iact(R._h, k, self.eos_ptr, self.p_ptr, m)
            if region_ev is not None:
                region_ev[s][1].record(st)
            if record is not None:
                record.append(torch_nonzero(self.Hy["eos_in"][0] > 0))
            if count is not None:
                act = count[3][s]
                count[0] += act.numel()
                count[1] += (mask[act] == 1).sum()
                count[2] += (mask == 1).sum()
            hp.hpac_hydro_finalize(self.Hy.state, sh)

    def close(self):
        self.kept.close()
        self.Hy.close()


def torch_nonzero(b):
    return b.nonzero().flatten()


def events(torch, n):
    return [[torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)] for _ in range(n)]


def bench_headline(hpac, torch, dev, stream, args, world, rank, clk):
    """Selection of the headline form, then K timed steps of it (see the
    module docstring), the exact run's time for the speedup, the element
    kernel's roofline inside the timed region and the end-to-end run through
    the public API with host buffers."""
    HB = HydroBench(hpac, torch, dev, stream, args.n, args.time_steps, W.DEFAULT_SEED + rank)
    E, nsteps = HB.E, HB.nsteps
    sh = stream.cuda_stream
    # exact reference: final pressure, origin energy, the elements carrying
    # energy at each step's EOS call (the blast's reach), the exact run's time
    active = []
    HB.run(None, record=active)
    torch.cuda.synchronize()
    reg_ev = events(torch, nsteps)
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    exact_ms, exact_region_ms = [], []
    for rep in range(args.exact_reps):
        a.record(stream)
        HB.run(None, region_ev=reg_ev)
        b.record(stream)
        torch.cuda.synchronize()
        exact_ms.append(a.elapsed_time(b))
        exact_region_ms.append(sum(e0.elapsed_time(e1) for e0, e1 in reg_ev))
    p_ex = HB.Hy["p"].clone()
    qoi_ex = float(HB.Hy["e"][0].item())
    p_rms = float(torch.sqrt(torch.mean(p_ex * p_ex)).item())
    t_ex = float(np.median(exact_ms))
    t_ex_region = float(np.median(exact_region_ms))

    def quality():
        r = hpac.quality(p_ex, HB.Hy["p"], hpac.HPAC_METRIC_RMSE, stream=stream)["value"]
        q = float(HB.Hy["e"][0].item())
        nrmse = r / p_rms if p_rms > 0 else 0.0
        return {"qoi_rel_err": abs(q - qoi_ex) / abs(qoi_ex), "p_nrmse": nrmse}

    # selection: one timed run and the quality of every candidate form
    table = []
    mask = torch.zeros(E, dtype=torch.uint8, device=dev)
    for form in HEAD_FORMS:
        a.record(stream)
        HB.run(form, region_ev=reg_ev)
        b.record(stream)
        torch.cuda.synchronize()
        ms = a.elapsed_time(b)
        rms = sum(e0.elapsed_time(e1) for e0, e1 in reg_ev)
        q = quality()
        ok = all(np.isfinite(v) and v <= QUALITY_BOUND for v in q.values())
        table.append(dict(form=form[0], ms=ms, speedup=t_ex / ms, region_ms=rms,
                          region_speedup=t_ex_region / rms, **q, within_bound=bool(ok)))
    # approximated share of the active invocations (elements that carry
    # energy at that step's EOS call in the exact run), for every form within
    # the bound; the fastest approximating at least MIN_ACTIVE_APPROX of them
    # is the headline (if none does, the one approximating the largest share)
    for row in table:
        if not row["within_bound"]:
            continue
        form = next(f for f in HEAD_FORMS if f[0] == row["form"])
        cnt = [torch.zeros((), dtype=torch.int64, device=dev) for _ in range(3)] + [active]
        HB.run(form, mask=mask, count=cnt)
        act, apx_act, apx = (int(c.item()) if hasattr(c, "item") else int(c) for c in cnt[:3])
        row.update(active_invocations=act / (E * nsteps), approx_active=apx_act / max(act, 1),
                   approx_all=apx / (E * nsteps))
    ok = [r for r in table if r["within_bound"]]
    qual = [r for r in ok if r["approx_active"] >= MIN_ACTIVE_APPROX]
    best = min(qual, key=lambda r: r["ms"]) if qual else max(ok, key=lambda r: (r["approx_active"], -r["ms"]))
    best["qualifies"] = bool(qual)
    del active
    form = next(f for f in HEAD_FORMS if f[0] == best["form"])
    vacuous = min((r for r in table if r["within_bound"]), key=lambda r: r["ms"])

    # timed steps: warm-up, then K runs with their quality, the element kernel
    # timed by events inside every run
    for _ in range(args.warmup):
        HB.run(form)
        quality()
    torch.cuda.synchronize()
    if world > 1:
        import torch.distributed as dist
        dist.barrier()
    elem_ev = [events(torch, nsteps) for _ in range(args.steps)]
    q_dev = torch.zeros(args.steps, dtype=torch.float64, device=dev)
    start, stop = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    start.record(stream)
    quals = []
    for s in range(args.steps):
        HB.run(form, elem_ev=elem_ev[s])
        r = hpac.quality(p_ex, HB.Hy["p"], hpac.HPAC_METRIC_RMSE, stream=stream)
        q_dev[s] = HB.Hy["e"][0]
        quals.append(r["value"])
    stop.record(stream)
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    total_ms, _ = aggregate(start.elapsed_time(stop), 1, world, dev)
    ms_per_step = total_ms / args.steps
    value = world * E * nsteps / (ms_per_step * 1e-3)
    elem_ms = float(np.mean([e0.elapsed_time(e1) for s in range(args.steps) for e0, e1 in elem_ev[s]]))
    qoi_t = q_dev.cpu().numpy()
    timed_quality = {"qoi_rel_err": float(np.max(np.abs(qoi_t - qoi_ex)) / abs(qoi_ex)),
                     "p_nrmse": float(max(quals)) / p_rms}

    # end to end through the public API with host buffers: the initial mesh
    # from pinned host memory, hpac_hydro_init, the run under the form
    # (hpac_hydro_run), the final energy field back to the host
    pin, e_out = HB.pin, HB.e_out
    h2d = sum(int(v.numel() * 8) for v in pin.values())
    R = HB.region(form)
    k = HB.knobs(form)

    def e2e_once():
        HB.reset(form)
        for key, v in pin.items():
            HB.Hy.t[key].copy_(v, non_blocking=True)
        hpac.hpac_hydro_init(HB.Hy.state, sh)
        hpac.hpac_hydro_run(HB.Hy.state, R._h, nsteps, form[1], k)
        e_out.copy_(HB.Hy["e"], non_blocking=True)

    e2e_ms = timed_ms(torch, stream, e2e_once, args.e2e_reps)
    e2e = {"value": world * E * nsteps / (e2e_ms * 1e-3), "unit": "elements/s",
           "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": int(E * 8)}

    # the element kernel's roofline (HBM) in the timed region
    fp64_tflops = hpac.hpac_device_fp64_rate(sh)
    hbm, hbm_src = measured_peaks()
    achieved = ELEM_BYTES * E / (elem_ms * 1e-3) / 1e9
    roofline = {"bound": "hbm", "kernel": "elem_kernel", "achieved": achieved, "peak": hbm,
                "unit": "GB/s", "frac": achieved / hbm, "peak_source": hbm_src,
                "traffic": dram_traffic("elem_kernel", E), "launch_ms": elem_ms}
    n_launch = args.steps * (nsteps * 4 + 1)      # node, elem, region, finalize; quality: 1
    detail = {"mesh": f"{args.n}^3", "time_steps": nsteps, "form": form[0], "exact_ms": t_ex,
              "exact_region_ms": t_ex_region, "selection": table, "best": best,
              "fastest_within_bound": vacuous["form"], "timed_quality": timed_quality,
              "fp64_fma_tflops_measured": fp64_tflops}
    out = dict(value=value, ms_per_step=ms_per_step, form=form, best=best, t_ex=t_ex,
               t_ex_region=t_ex_region, e2e=e2e, roofline=roofline, gpu_launches=n_launch,
               detail=detail, timed_quality=timed_quality)
    return out, HB


# ---------------------------------------------------------------- kernels

def bench_kernels(hpac, torch, dev, stream, HB, clk, bs_cfg0=None):
    """Roofline of every exact hydro kernel at the headline mesh: one exact run
    with CUDA events around each phase of every time step (node, element, EOS
    region, finalize). Units and algorithmic work per unit:
      node_kernel   HBM: per node u, v, w, x, y, z read and written (96 B) and
                    1 / (12 m) (8 B); per element its 24 stored gradient
                    values (192 B) and p + q (8 B), each read once (its FP64
                    fraction, NODE_OPS per node, is reported beside it)
      elem_kernel   HBM: ELEM_BYTES per element (the issue of integer instructions
                    is what bounds it)
      EOS exact     HBM: four inputs read and the pressure written per element
                    (40 B; FP64 issue is what bounds it where there is energy)
      finalize      HBM: per element v_{n+1}, p, q read, e, v, p + q written (48 B)
    """
    E, n1 = HB.E, HB.n + 1
    Nn = n1 ** 3
    hbm, hbm_src = measured_peaks()
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    cs = clk.summary()
    mhz = cs["sm_mhz"] or cs["sm_max_mhz"] or 2070.0
    fp64_peak = FP64_FMA_PER_SM_CLK * sms * mhz * 1e6
    sh, st, hp = stream.cuda_stream, stream, hpac
    ph = [events(torch, HB.nsteps) for _ in range(4)]
    HB.reset(None)
    for s in range(HB.nsteps):
        ph[0][s][0].record(st)
        hp.hpac_hydro_nodes(HB.Hy.state, sh)
        ph[0][s][1].record(st)
        ph[1][s][0].record(st)
        hp.hpac_hydro_elements(HB.Hy.state, sh)
        ph[1][s][1].record(st)
        ph[2][s][0].record(st)
        hp.hpac_run_exact(HB.Hy.eos._h, HB.eos_ptr, HB.p_ptr)
        ph[2][s][1].record(st)
        ph[3][s][0].record(st)
        hp.hpac_hydro_finalize(HB.Hy.state, sh)
        ph[3][s][1].record(st)
    torch.cuda.synchronize()
    ms = [float(np.mean([e0.elapsed_time(e1) for e0, e1 in ph[j]])) for j in range(4)]
    rows = {
        "node_kernel": dict(bound="hbm", ms=ms[0], bytes=Nn * 104 + E * 200, peak=hbm * 1e9, unit="B/s",
                            fp64_frac=Nn * NODE_OPS / (ms[0] * 1e-3) / fp64_peak),
        "elem_kernel": dict(bound="hbm", ms=ms[1], bytes=E * ELEM_BYTES, peak=hbm * 1e9, unit="B/s"),
        "eos_exact": dict(bound="hbm", ms=ms[2], bytes=E * 40, peak=hbm * 1e9, unit="B/s"),
        "finalize_kernel": dict(bound="hbm", ms=ms[3], bytes=E * 48, peak=hbm * 1e9, unit="B/s"),
    }
    for r in rows.values():
        work = r.get("bytes", r.get("ops"))
        r["achieved"] = work / (r["ms"] * 1e-3)
        r["frac"] = r["achieved"] / r["peak"]
    if bs_cfg0 is not None:
        rows.update(bs_cfg0)
    return {"mesh": f"{HB.n}^3", "time_steps": HB.nsteps, "hbm_peak_gbs": hbm, "hbm_peak_source": hbm_src,
            "fp64_peak_source": f"derived: {FP64_FMA_PER_SM_CLK} FP64 FMA/SM/clk x {sms} SMs x {mhz:.0f} MHz",
            "kernels": rows}


def bench_hydro64(hpac, torch, dev, stream, rank, n=HYDRO_N, nsteps=HYDRO_STEPS, reps=3):
    """The 64^3 x 100-step configuration: runs with the EOS exact, under TAF
    (h4 p8 0.5%) and under iACT (t8, private tables, 1e-3), launch-scoped state
    (T = E / 8), each timed, with the quality of the final state (origin
    energy, pressure NRMSE), plus the EOS region alone on a mid-run state and
    a 64-configuration knob sweep of it."""
    HB = HydroBench(hpac, torch, dev, stream, n, nsteps, W.DEFAULT_SEED + rank)
    forms = {"exact": None,
             "taf": ("taf h4 p8 0.5%", 1, False, dict(TAF)),
             "iact": ("iact t8 g32 1e-3", 2, False, dict(IACT))}
    res = {}
    ref_p = ref_q = None
    for name, form in forms.items():
        t = timed_ms(torch, stream, lambda: HB.run(form), reps)
        row = {"ms": t, "element_updates_per_s": HB.E * nsteps / (t * 1e-3)}
        if form is None:
            ref_p, ref_q = HB.Hy["p"].clone(), float(HB.Hy["e"][0].item())
            p_rms = float(torch.sqrt(torch.mean(ref_p * ref_p)).item())
        else:
            r = hpac.quality(ref_p, HB.Hy["p"], hpac.HPAC_METRIC_RMSE, stream=stream)["value"]
            row.update(speedup_vs_exact=res["exact"]["ms"] / t, p_nrmse=r / p_rms,
                       qoi_rel_err=abs(float(HB.Hy["e"][0].item()) - ref_q) / abs(ref_q))
        res[name] = row
    # the EOS region alone on a mid-run state
    HB.reset(None)
    for _ in range(nsteps // 2):
        hpac.hpac_hydro_step(HB.Hy.state, HB.Hy.eos._h, 0, None, None, False)
    hpac.hpac_hydro_nodes(HB.Hy.state, stream.cuda_stream)
    hpac.hpac_hydro_elements(HB.Hy.state, stream.cuda_stream)
    torch.cuda.synchronize()
    region_ms = {}
    for name, form in forms.items():
        k = HB.knobs(form) if form is not None else None
        if form is None:
            f = lambda: hpac.hpac_run_exact(HB.Hy.eos._h, HB.eos_ptr, HB.p_ptr)
        elif form[1] == 1:
            f = lambda k=k: hpac.hpac_run_taf(HB.Hy.eos._h, k, HB.eos_ptr, HB.p_ptr)
        else:
            f = lambda k=k: hpac.hpac_run_iact(HB.Hy.eos._h, k, HB.eos_ptr, HB.p_ptr)
        region_ms[name] = timed_ms(torch, stream, f, 50)
    ref_mid = torch.zeros(HB.E, dtype=torch.float64, device=dev)
    hpac.hpac_run_exact(HB.Hy.eos._h, HB.eos_ptr, hpac.C.c_void_p(ref_mid.data_ptr()))
    sweep = eos_region_sweep(hpac, torch, stream, HB.Hy.eos._h, HB.Hy["eos_in"], ref_mid, HB.scale)
    HB.close()
    return {"mesh": f"{n}^3", "time_steps": nsteps, "runs": res,
            "eos_region_ms": region_ms,
            "eos_region_speedup": {k: region_ms["exact"] / v for k, v in region_ms.items()},
            "eos_sweep": sweep}


def bench_cfg4_extras(hpac, torch, dev, stream, HB, train_pairs=1 << 22, epochs=16, sweep_configs=64):
    """The rest of the large configuration on the headline mesh: the EOS
    replaced by a learned surrogate (4 -> 128 -> 128 -> 1, trained on EOS
    pairs recorded from the exact run) and a 64-configuration knob sweep of the
    EOS region on the mid-run state."""
    E, nsteps = HB.E, HB.nsteps
    sh = stream.cuda_stream
    pairs, mid = [], []
    HB.reset(None)
    for s in range(nsteps):
        hpac.hpac_hydro_nodes(HB.Hy.state, sh)
        hpac.hpac_hydro_elements(HB.Hy.state, sh)
        hpac.hpac_run_exact(HB.Hy.eos._h, HB.eos_ptr, HB.p_ptr)
        ein = HB.Hy["eos_in"]
        act = torch.nonzero((ein[0] > 0) | (ein[3] > 0) | (ein[2] != 0)).flatten()
        pairs.append((ein[:, act].clone(), HB.Hy["p"][act].clone()))
        if s + 1 == nsteps // 2:
            mid.append(ein.clone())
        hpac.hpac_hydro_finalize(HB.Hy.state, sh)
    p_ex = HB.Hy["p"].clone()
    qoi_ex = float(HB.Hy["e"][0].item())
    t_ex = timed_ms(torch, stream, lambda: HB.run(None), 1)
    # training pairs: the active elements of every step plus as many untouched
    # ones (inputs (0, 1, 0, 0) -> p = 0)
    xa = torch.cat([a for a, _ in pairs], dim=1)
    ya = torch.cat([b for _, b in pairs])
    nq = xa.shape[1]
    xq = torch.zeros(4, nq, dtype=torch.float64, device=dev)
    xq[1] = 1.0
    perm = torch.randperm(2 * nq, device=dev, generator=torch.Generator(device=dev).manual_seed(7))
    xtr = torch.cat([xa, xq], dim=1)[:, perm][:, :train_pairs].contiguous()
    ytr = torch.cat([ya, torch.zeros(nq, dtype=torch.float64, device=dev)])[perm][:train_pairs].float().contiguous()
    S = hpac.Surrogate(hpac.eos_desc(128), seed=4, stream=stream)
    S.fit_normalization(xtr, ytr, GAMMA)
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record(stream)
    loss = S.train(xtr, ytr, GAMMA, batch=8192, epochs=epochs, lr=2e-3)
    b.record(stream)
    torch.cuda.synchronize()
    train_ms = a.elapsed_time(b)

    def run_sur():
        HB.reset(None)
        for s in range(nsteps):
            hpac.hpac_hydro_nodes(HB.Hy.state, sh)
            hpac.hpac_hydro_elements(HB.Hy.state, sh)
            S.infer(HB.Hy["eos_in"], HB.Hy["p"], GAMMA)
            hpac.hpac_hydro_finalize(HB.Hy.state, sh)
    t = timed_ms(torch, stream, run_sur, 1)
    p_rms = float(torch.sqrt(torch.mean(p_ex * p_ex)).item())
    r = hpac.quality(p_ex, HB.Hy["p"], hpac.HPAC_METRIC_RMSE, stream=stream)["value"]
    sur = {"ms": t, "speedup_vs_exact": t_ex / t, "p_nrmse": r / p_rms,
           "qoi_rel_err": abs(float(HB.Hy["e"][0].item()) - qoi_ex) / abs(qoi_ex),
           "train_pairs": int(xtr.shape[1]), "train_ms": train_ms, "train_mse_normalized": loss}
    S.close()
    del xa, ya, xq, xtr, ytr, pairs
    HB.Hy["eos_in"].copy_(mid[0])
    ref = torch.zeros(E, dtype=torch.float64, device=dev)
    hpac.hpac_run_exact(HB.Hy.eos._h, HB.eos_ptr, hpac.C.c_void_p(ref.data_ptr()))
    sweep = eos_region_sweep(hpac, torch, stream, HB.Hy.eos._h, HB.Hy["eos_in"], ref, HB.scale, sweep_configs)
    return {"mesh": f"{HB.n}^3", "time_steps": nsteps, "exact_ms": t_ex, "surrogate": sur, "eos_sweep": sweep}


def emit(detail, name, obj):
    """One section: printed on its own line (before the final one) and kept
    for the detail file."""
    detail[name] = obj
    print(json.dumps({"section": name, **obj} if isinstance(obj, dict) else {"section": name, "value": obj},
                     default=float), flush=True)


def main(argv=None):
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="gb300", choices=["gb300", "reference"])
    ap.add_argument("--n", type=int, default=HEAD_N)
    ap.add_argument("--time-steps", type=int, default=HEAD_STEPS)
    ap.add_argument("--exact-reps", type=int, default=3)
    ap.add_argument("--e2e-reps", type=int, default=2)
    ap.add_argument("--reference-form", default="iact kept t4 g4 1e-3",
                    help="EOS form the reference arm (the CPU oracle) runs")
    ap.add_argument("--sections", default="all",
                    help="comma-separated sections after the headline, 'all' or 'none'")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--detail", default=os.path.join(ROOT, "_build", "bench_detail.json"))
    args = ap.parse_args(argv)
    if args.impl == "reference":
        return run_reference(args)
    args.steps = max(1, args.steps)

    import torch
    import torch.distributed as dist

    from paper_2308_16877_gb300 import hpac

    rank, world, local = env_rank()
    if world > 1:
        dist.init_process_group("nccl", init_method="env://")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    hpac.load()
    stream = torch.cuda.current_stream(dev)
    all_sections = ["kernels", "cfg4_extras", "hydro64", "blackscholes_65536", "blackscholes_16M", "sweep",
                    "search", "binomial", "kmeans", "levels", "lavamd", "surrogate", "persistent_state"]
    want = all_sections if args.sections == "all" else ([] if args.sections == "none"
                                                         else args.sections.split(","))
    detail = {}

    clk = ClockSampler(local).start()
    time.sleep(0.5)
    head, HB = bench_headline(hpac, torch, dev, stream, args, world, rank, clk)
    clk.stop()
    clocks = clk.summary()
    if rank == 0:
        emit(detail, "headline", head["detail"])

    # sections (rank 0 prints them; every rank runs them so replicas stay alike)
    def section(name, fn):
        if name in want:
            r = fn()
            if rank == 0:
                emit(detail, name, r)
            return r
        return None

    bs0 = section("blackscholes_65536", lambda: bench_blackscholes_cfg0(hpac, torch, dev, stream))
    bs = section("blackscholes_16M", lambda: bench_blackscholes(hpac, torch, dev, stream))
    extra_rows = {}
    if bs0 is not None:
        extra_rows["bs_exact_65536"] = bs0["kernel_row"]
    if bs is not None:
        extra_rows["bs_exact_16M"] = bs["kernel_row"]
    kern = section("kernels", lambda: bench_kernels(hpac, torch, dev, stream, HB, ClockSummary(clocks),
                                                    extra_rows))
    section("cfg4_extras", lambda: bench_cfg4_extras(hpac, torch, dev, stream, HB))
    HB.close()
    del HB
    torch.cuda.empty_cache()
    section("hydro64", lambda: bench_hydro64(hpac, torch, dev, stream, rank))
    section("sweep", lambda: bench_sweep(hpac, torch, dev, stream))
    section("search", lambda: bench_search(hpac, torch, dev, stream))
    section("binomial", lambda: bench_binomial(hpac, torch, dev, stream))
    section("kmeans", lambda: bench_kmeans(hpac, torch, dev, stream))
    section("levels", lambda: bench_levels(hpac, torch, dev, stream))
    section("lavamd", lambda: bench_lavamd(hpac, torch, dev, stream))
    section("surrogate", lambda: bench_surrogate(hpac, torch, dev, stream))
    section("persistent_state", lambda: bench_persistent(hpac, torch, dev, stream))

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        cpu = hydro_cpu(head["form"], n=args.n, steps=4, single_steps=1)
        cpu.pop("seconds", None)
        emit(detail, "cpu_baseline", cpu)

    if rank == 0:
        best = head["best"]
        form = head["form"]
        rl = head["roofline"]
        line = {
            "metric": METRIC, "value": sig(head["value"], 5), "unit": "elements/s", "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": sig(head["ms_per_step"], 5),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic",
            "config": {"workload": workload_name(args.n, args.time_steps, form[0]),
                       "l2": "inputs > L2 (6.5 GB state)", "parallelism": f"replicas{world}"},
            "speedup_vs_exact": {"run": sig(best["speedup"]), "eos_region": sig(best["region_speedup"])},
            "quality": {"qoi_rel_err": sig(head["timed_quality"]["qoi_rel_err"], 3),
                        "p_nrmse": sig(head["timed_quality"]["p_nrmse"], 3),
                        "approx_active": sig(best["approx_active"], 3), "bound": QUALITY_BOUND,
                        "qualifies": best["qualifies"]},
            "roofline": {"bound": rl["bound"], "kernel": rl["kernel"], "achieved": sig(rl["achieved"]),
                         "peak": sig(rl["peak"]), "unit": rl["unit"], "frac": sig(rl["frac"], 3),
                         "traffic": rl["traffic"]},
            "cpu_baseline": None if cpu is None else {k: sig(cpu[k]) for k in
                                                      ("value", "unit", "cores", "kind", "sample")},
            "e2e": sig(head["e2e"]),
            "gpu_launches": head["gpu_launches"],
            "clocks": {k: clocks.get(k) for k in ("sm_mhz", "sm_max_mhz", "reasons")},
        }
        if kern is not None:  # roofline fractions of the exact kernels (all rows in the detail file)
            short = {"node_kernel": "node", "elem_kernel": "elem", "eos_exact": "eos", "finalize_kernel": "finalize",
                     "bs_exact_16M": "bs16M"}
            line["kernels_frac"] = {short[k]: sig(v["frac"], 3) for k, v in kern["kernels"].items() if k in short}
        try:
            os.makedirs(os.path.dirname(args.detail), exist_ok=True)
            with open(args.detail, "w") as f:
                json.dump({"final": line, **detail}, f, indent=1, default=float)
        except OSError:
            pass
        print(json.dumps(line, default=float, separators=(",", ":")))
    if world > 1:
        dist.destroy_process_group()
    return 0


class ClockSummary:
    """A fixed clock summary with the sampler's interface."""

    def __init__(self, s):
        self.s = s

    def summary(self):
        return self.s


if __name__ == "__main__":
    sys.exit(main())
