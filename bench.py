#!/usr/bin/env python
"""Throughput benchmark of the lattice ES-BGK solver.

Workload: a 4096 x 4096 fully periodic Taylor-Green vortex (Ma 0.05, 1% T
perturbation, 1e-4 density noise, seed 0), D2Q16, Hermite order 3, Kn 0.05,
b = -1/2, FP32 compute and storage.  One benchmark step is one whole solve:
initial populations from device-resident fields, 1000 fused time steps, and
the nine moment fields.  value = lattice updates per second / 1e6 (MLUPS)
with the fields already in HBM; e2e = the same solves through the C ABI with
host buffers (create from pinned host fields, moments copied back to pinned
host memory), double-buffered so that each solve's copies overlap its
neighbours' steps, timed on the wall clock.  The line also carries the same
solve in compensated FP32 storage (`precision`: the storage that holds every
field within 1e-5 of the FP64 oracle at this size, with the per-storage
errors of the committed 4096^2 record), and the batched (512 channel solves)
and served (Poisson trace) forms of the metric, each with its own timed
region.

Under torchrun (N > 1) the default splits the one 4096^2 solve into y-slabs,
one per rank, with halos exchanged over NCCL (--decomp slab: scaling
"strong"); --decomp replica runs an independent replica per rank (scaling
"weak", value = all ranks' updates / the slowest rank's time).  Other
workloads: --workload batch | serve | precision | slab.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)
L2_BYTES = 129e6  # GB300 L2

HBM_FALLBACK_GBS = 6800.0
BYTES_PER_LUP = 2 * 16 * 4  # read f^n once, write f^{n+1} once, Q = 16 FP32
METRIC = "ES-BGK MLUPS"
UNIT = "MLUPS"


STORE_BYTES = {"f32": 4, "f16": 2, "bf16": 2, "f32c": 6}  # bytes per stored value (f32c: FP32 hi + FP16 lo)


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--n", type=int, default=4096, help="grid is n x n")
    ap.add_argument("--lattice-steps", type=int, default=1000)
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-batch", action="store_true",
                    help="default workload: leave out the batched-solves object")
    ap.add_argument("--no-serve", action="store_true",
                    help="default workload: leave out the serving object")
    ap.add_argument("--no-precision", action="store_true",
                    help="default workload: leave out the compensated-storage object")
    ap.add_argument("--save-moments", default=None,
                    help="precision workload: run the GPU leg only and save its sampled moments here")
    ap.add_argument("--compare-moments", default=None,
                    help="precision workload: run the oracle leg only, against moments saved by --save-moments")
    ap.add_argument("--decomp", choices=["slab", "replica"], default="slab",
                    help="with several ranks: split the one domain into y-slabs (strong scaling), or run "
                         "an independent replica per rank (weak scaling)")
    ap.add_argument("--halo-steps", type=int, default=8,
                    help="y-slabs: time steps per halo exchange (halo of 2k rows)")
    ap.add_argument("--serve-requests", type=int, default=100,
                    help="requests of the default line's serving object")
    ap.add_argument("--serve-plain-budget", type=float, default=20.0,
                    help="seconds the default line's FIFO serving baseline may run")
    ap.add_argument("--workload", choices=["tgv", "batch", "serve", "precision", "slab"], default="tgv",
                    help="tgv: 4096^2 Taylor-Green throughput (default); batch: 512-instance channel mix; "
                         "serve: Poisson arrivals run to steady state with continuous batching")
    ap.add_argument("--velocity-set", choices=["d2q16", "d2q36", "d3q64", "d3q216"], default="d2q16",
                    help="tgv workload lattice: D2Q16 (order 3), D2Q36 (order 4), D3Q64 (order 3, D = 3: the "
                         "paper's C_p = 5/2) or D3Q216 (order 4, D = 3: the paper's set); the D = 3 sets are "
                         "stored by their z-even half")
    ap.add_argument("--storage", choices=["f32", "f16", "bf16", "f32c"], default="f32",
                    help="population storage for the tgv workload (compute is FP32)")
    ap.add_argument("--requests", type=int, default=400)
    ap.add_argument("--rate", type=float, default=200.0, help="mean arrivals per second")
    ap.add_argument("--pool-mb", type=float, default=64.0, help="device-memory budget of the serving pool")
    ap.add_argument("--plain-budget", type=float, default=60.0, help="seconds the FIFO baseline may run")
    ap.add_argument("--tgv-n", type=int, default=256,
                    help="precision workload: Taylor-Green grid (4096 = the throughput workload; the FP64 "
                         "oracle then needs about half an hour on 16 cores)")
    ap.add_argument("--instances", type=int, default=512)
    ap.add_argument("--plain-sample", type=int, default=32, help="instances the one-at-a-time baseline runs")
    ap.add_argument("--no-steady", action="store_true",
                    help="batch workload: skip the run-to-steady-state mode")
    return ap.parse_args()


def tgv_workload_name(n, args):
    return f"tgv_{n}x{n}_{args.velocity_set}_{args.storage}"


LATTICES = {  # velocity set -> (nroots, dim, order, values stored per node)
    "d2q16": (4, 2, 3, 16),
    "d2q36": (6, 2, 4, 36),
    "d3q64": (4, 3, 3, 32),
    "d3q216": (6, 3, 4, 108),
}


def tgv_problem(n, args, nsteps):
    from dataclasses import replace
    from paper_1209_6548_gb300 import inputs as I
    nroots, dim, _, _ = LATTICES[args.velocity_set]
    return replace(I.tgv(n, steps=nsteps, nroots=nroots), dim=dim)


def tgv_config(n, args, nsteps):
    """The config object of the throughput workload (shared by both arms)."""
    prob = tgv_problem(n, args, nsteps)
    return {"workload": tgv_workload_name(n, args), "nx": n, "ny": n, "velocity_set": args.velocity_set.upper(),
            "storage": args.storage, "order": LATTICES[args.velocity_set][2], "kn": prob.kn, "b": prob.b,
            "lattice_steps_per_step": nsteps, "scheme": "split"}


def measured_peak():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as fh:
            return float(json.load(fh)["hbm_gbs"]), "measured"
    except Exception:
        return HBM_FALLBACK_GBS, "fallback"


def committed_traffic(source_digest: str, velocity_set: str = "d2q16", storage: str = "f32"):
    """Per-launch DRAM bytes of the step kernel on this velocity set and
    storage from the committed ncu summary, if it was taken on the current
    kernel source (else None)."""
    path = os.path.join(ROOT, "profiles", f"k_step_tgv4096_{velocity_set}.md")
    try:
        lines = open(path).read().splitlines()
    except OSError:
        return None
    vals = {}
    for ln in lines:
        if ln.startswith("- ") and ":" in ln:
            k, v = ln[2:].split(":", 1)
            vals[k.strip()] = v.strip().strip("`")
    if vals.get("kernel source sha256") != source_digest:
        return None
    try:
        return float(vals[f"dram bytes per launch (scaled to 4096^2, {storage} storage)"])
    except (KeyError, ValueError):
        return None


def committed_instructions(source_digest: str, velocity_set: str = "d2q16", storage: str = "f32"):
    """Thread-instructions per lattice update of the step kernel from the
    committed ncu summary (same digest rule as committed_traffic), or None."""
    path = os.path.join(ROOT, "profiles", f"k_step_tgv4096_{velocity_set}.md")
    try:
        lines = open(path).read().splitlines()
    except OSError:
        return None
    vals = {}
    for ln in lines:
        if ln.startswith("- ") and ":" in ln:
            k, v = ln[2:].split(":", 1)
            vals[k.strip()] = v.strip().strip("`")
    if vals.get("kernel source sha256") != source_digest:
        return None
    try:
        return float(vals[f"thread-instructions per lattice update ({storage} storage)"])
    except (KeyError, ValueError):
        return None


def issue_view(instr_per_update, cells, kernel_ms, sm_count, sm_mhz):
    """The step as instruction issue: warp-instructions issued per second
    (instructions per update from ncu, updates per second from the CUDA-event
    kernel time) against SMs x 4 schedulers x the sampled SM clock."""
    if not instr_per_update or not sm_mhz:
        return None
    achieved = instr_per_update / 32.0 * cells / (kernel_ms / 1e3)
    peak = sm_count * 4 * sm_mhz * 1e6
    return {"achieved": achieved, "peak": peak, "unit": "warp-instructions/s", "frac": achieved / peak,
            "instr_per_update": instr_per_update, "sm_mhz": sm_mhz}


def _function_text(text: str, head: str) -> str:
    """The source of the function whose definition starts with head (up to
    its matching closing brace)."""
    a = text.index(head)
    depth, k = 0, text.index("{", a)
    while True:
        if text[k] == "{":
            depth += 1
        elif text[k] == "}":
            depth -= 1
            if depth == 0:
                return text[a:k + 1]
        k += 1


def source_digest():
    """sha256 (16 hex digits) of the step kernel's source: device.cuh, the
    k_step section of lesbgk.cu, the functions that pick its launch shape and
    launch it, and its block size and ring depth; other code in the file does
    not change it."""
    import hashlib
    csrc = os.path.join(ROOT, "paper_1209_6548_gb300", "csrc")
    h = hashlib.sha256()
    with open(os.path.join(csrc, "device.cuh"), "rb") as fh:
        h.update(fh.read())
    with open(os.path.join(csrc, "lesbgk.cu")) as fh:
        text = fh.read()
    a = text.index("// The fused time step")
    h.update(text[a:text.index("// Initial populations", a)].encode())
    for head in ("int pick_launch(", "int launch_step("):
        h.update(_function_text(text, head).encode())
    h.update("".join(ln for ln in text.splitlines(True)
                     if ln.startswith(("constexpr int kBlock ", "constexpr int kRing "))).encode())
    return h.hexdigest()[:16]


class ClockSampler:
    """nvidia-smi samples of SM clock and throttle reasons during the timed region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, device_index: int):
        self.dev = device_index
        self.proc = None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.dev), f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                 "-lms", "200"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
        return self

    def __exit__(self, *exc):
        self.out = ""
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.out, _ = self.proc.communicate(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
                self.out, _ = self.proc.communicate()

    def summary(self):
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in (self.out or "").splitlines():
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                mx = float(parts[2])
            except ValueError:
                continue
            for nm, v in zip(names, parts[5:9]):
                if v.lower() == "active":
                    reasons.add(nm)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": mx, "reasons": [], "samples": 0}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": mx, "reasons": sorted(reasons),
                "samples": len(sm)}


def dist_setup():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def cpu_baseline(n: int, rows: int = 1024, steps: int = 48, velocity_set: str = "d2q16",
                 single_thread: bool = True):
    """The FP64 oracle, as it stands, on a bounded sample of the workload: the
    first `rows` rows of the n x n Taylor-Green initial state, periodic, split
    scheme, for `steps` time steps, on all host cores the process may use; and
    (single_thread) on one core, on a sixteenth of the rows for half the steps."""
    import numpy as np
    import oracle as O
    from paper_1209_6548_gb300 import inputs as I
    nroots, dim, order, _ = LATTICES[velocity_set]
    prob = I.tgv(n, nroots=nroots)
    fields = I.initial_fields(prob)[:, :rows, :].copy()
    cores = len(os.sched_getaffinity(0))
    O.set_threads(cores)
    dx = dy = 1.0 / n
    c, _ = O.gauss_hermite_1d(nroots)
    dt = 0.5 * dx / float(np.abs(c).max())
    op = O.make_params(nroots=nroots, order=order, nx=n, ny=rows, bc_y=0, kn=prob.kn, b=prob.b,
                       visc_exp=prob.visc_exp, dt=dt, dx=dx, dy=dy, scheme=prob.scheme, dim=dim)
    f = O.init(op, fields)
    t0 = time.perf_counter()
    O.run(op, f, steps)
    sec = time.perf_counter() - t0
    out = {"value": n * rows * steps / sec / 1e6, "unit": UNIT, "cores": O.get_threads(), "kind": "oracle",
           "sample": f"{n}x{rows} periodic rows of the Taylor-Green state ({velocity_set.upper()}), "
                     f"{steps} FP64 oracle steps ({sec:.1f} s)"}
    if single_thread:
        r1, s1 = max(1, rows // 16), max(1, steps // 2)
        op1 = O.make_params(nroots=nroots, order=order, nx=n, ny=r1, bc_y=0, kn=prob.kn, b=prob.b,
                            visc_exp=prob.visc_exp, dt=dt, dx=dx, dy=dy, scheme=prob.scheme, dim=dim)
        f1 = O.init(op1, fields[:, :r1, :].copy())
        O.set_threads(1)
        t0 = time.perf_counter()
        O.run(op1, f1, s1)
        sec1 = time.perf_counter() - t0
        O.set_threads(cores)
        out["single_thread"] = {"value": n * r1 * s1 / sec1 / 1e6, "unit": UNIT, "cores": 1,
                                "sample": f"{n}x{r1} rows, {s1} steps ({sec1:.1f} s)"}
    return out


def run_reference(args, world, rank):
    if rank != 0:
        return 0
    samples = []
    t_all = time.perf_counter()
    base = None
    for k in range(args.warmup + args.steps):
        base = cpu_baseline(args.n, rows=256, steps=4, velocity_set=args.velocity_set, single_thread=False)
        if k >= args.warmup:
            samples.append(base["value"])
    value = statistics.median(samples)
    base["value"] = value
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": None, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": tgv_config(args.n, args, args.lattice_steps),
        "cpu_baseline": base,
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
        "wall_s": time.perf_counter() - t_all,
    }
    print(json.dumps(line), flush=True)
    return 0


PRECISION_RECORD = os.path.join(ROOT, "profiles", "precision_tgv4096_d2q16.json")


def precision_record():
    """Largest per-field error e against the FP64 oracle, by storage, of the
    committed 4096^2 Taylor-Green record (1000 steps, every 8th node), or None."""
    try:
        with open(PRECISION_RECORD) as fh:
            errs = json.load(fh)["oracle_leg"]["errors"]["tgv4096"]
    except (OSError, KeyError, ValueError):
        return None
    return {st: max(v["e"] for v in row.values()) for st, row in errs.items()}


def measure_compensated(prob, fields, nsteps, passes, warmup, stream, local):
    """The same solve with compensated FP32 storage (FP32 + FP16 remainder, 6 B
    per stored value), the storage that holds every field within 1e-5 of the
    FP64 oracle at this size: MLUPS and the step kernel's roofline at its own
    algorithmic bytes, timed with CUDA events on the launching stream."""
    import torch
    from paper_1209_6548_gb300 import lesbgk as L

    params = L.params_from_problem(prob, dt=0.0)
    params.storage = L.F32C
    solver = L.Solver(params, h_init=fields, stream=stream)
    d_fields = torch.from_numpy(fields).cuda()
    n = prob.nx * prob.ny
    d_mom = torch.empty((9, prob.ny, prob.nx), dtype=torch.float32, device="cuda")

    def one(ev=None):
        solver.reinit(d_fields)
        if ev is not None:
            ev[0].record(stream)
        solver.step(nsteps)
        if ev is not None:
            ev[1].record(stream)
        L.moments(solver.handle, d_mom.data_ptr(), None, stream.cuda_stream)

    for _ in range(warmup):
        one()
    torch.cuda.synchronize()
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(passes)]
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with ClockSampler(local) as clk:
        t0.record(stream)
        for k in range(passes):
            one(evs[k])
        t1.record(stream)
        torch.cuda.synchronize()
    ms = t0.elapsed_time(t1)
    kernel_ms = sum(a.elapsed_time(b) for a, b in evs) / (passes * nsteps)
    solver.close()
    peak, peak_kind = measured_peak()
    bytes_per_lup = 2 * 16 * STORE_BYTES["f32c"]
    achieved = bytes_per_lup * n / (kernel_ms / 1e3) / 1e9
    c = clk.summary()
    return {"storage": "f32c", "value": n * nsteps * passes / (ms / 1e3) / 1e6, "unit": UNIT,
            "solves": passes, "kernel": "k_step_c<split>", "kernel_ms": kernel_ms,
            "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
                         "bytes_per_lup": bytes_per_lup, "peak_source": peak_kind},
            "max_field_error_vs_fp64_oracle": precision_record(),
            "error_source": "committed record profiles/precision_tgv4096_d2q16.json (this solve, 1000 steps, "
                            "every 8th node; e = max |gpu - oracle| over the field quantity's largest magnitude)",
            "bar": 1e-5,
            "clocks": {"sm_mhz": c["sm_mhz"], "sm_max_mhz": c["sm_max_mhz"], "reasons": c["reasons"]}}


def measure_batch_fixed(params, nsteps, passes, warmup, stream, local, plain_sample, barrier=None,
                        max_over_ranks=None):
    """Batched solves of fixed length: one pass = L2 flush, admit every
    instance, nsteps steps for all, the nine moment fields of every instance;
    `passes` timed passes after `warmup`.  Also times one batch step (CUDA
    events) and the plain solver on `plain_sample` of the instances one at a
    time.  Returns (dict, batch step ms, rows per item)."""
    import torch
    from paper_1209_6548_gb300 import lesbgk as L

    barrier = barrier or torch.cuda.synchronize
    max_over_ranks = max_over_ranks or (lambda x: x)
    pool = int(sum(L.batch_slot_bytes(p) for p in params) * 1.05) + (1 << 20)
    bt = L.Batch(capacity=len(params), nx=4, pool_bytes=pool, stream=stream)
    outs = [torch.empty((9, p.ny, p.nx), dtype=torch.float32, device="cuda") for p in params]

    def admit_all():
        for s in list(bt.params):
            bt.remove(s)
        return bt.add_many(params)  # one descriptor copy, one init launch

    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")  # larger than the 129 MB L2

    def one_pass():
        flush.fill_(1)  # L2 flushed between timed passes (inside a pass the steps reuse it)
        sl = admit_all()
        bt.step(nsteps)
        bt.moments_many(sl, outs)  # every instance's nine fields in one launch

    for _ in range(warmup):
        one_pass()
    torch.cuda.synchronize()
    launch = bt.launch()  # the rules' choice for these solves
    rows = launch["rows_per_item"]

    def time_steps():
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        admit_all()
        bt.step(64)  # builds the step graph of this mode
        e0.record(stream)
        bt.step(640)
        e1.record(stream)
        torch.cuda.synchronize()
        return e0.elapsed_time(e1) / 640

    # one batch step of all instances, per launch mode (the rules last)
    modes = {}
    for name, on, k, lim in (("per_step_only", False, 64, 128), ("resident_k64_ny64", True, 64, 64),
                             ("resident_k64_ny128", True, 64, 128), ("resident_k64_all", True, 64, 1 << 20)):
        bt.set_resident(on, k, lim)
        modes[name] = time_steps()
    bt.set_auto()
    step_ms = time_steps()
    with ClockSampler(local) as clk:
        barrier()
        w0 = time.perf_counter()
        for _ in range(passes):
            one_pass()
        barrier()
        wsec = max_over_ranks(time.perf_counter() - w0)
    bt.close()
    n = len(params)
    idx = list(range(0, n, max(1, n // plain_sample)))[:plain_sample]
    lups = [p.nx * p.ny * nsteps for p in params]
    torch.cuda.synchronize()
    p0 = time.perf_counter()
    for i in idx:
        s = L.Solver(params[i], stream=stream)
        s.step(nsteps)
        L.moments(s.handle, outs[i].data_ptr(), None, stream.cuda_stream)
        s.close()
    torch.cuda.synchronize()
    psec = time.perf_counter() - p0
    plain_sec_per_lup = psec / sum(lups[i] for i in idx)
    clocks = clk.summary()
    out = {"solves_per_s_this_rank": n * passes / wsec, "wall_s": wsec, "passes": passes,
           "instance_mlups_this_rank": sum(lups) * passes / wsec / 1e6,
           "step_ms": step_ms, "rows_per_item": rows, "launch": launch, "step_ms_by_mode": modes,
           "plain": {"solves_per_s": len(idx) / psec, "sample": f"{len(idx)} of the {n} instances, one at a time",
                     "mlups": 1.0 / plain_sec_per_lup / 1e6,
                     "est_solves_per_s_full_mix": 1.0 / (plain_sec_per_lup * sum(lups) / n)},
           "clocks": {"sm_mhz": clocks["sm_mhz"], "sm_max_mhz": clocks["sm_max_mhz"], "reasons": clocks["reasons"]}}
    return out, step_ms, rows, pool


def measure_serve(requests, rate, pool_mb, plain_budget, stream, local, seed=0, cavity_share=0.1):
    """Serving: a seeded Poisson stream of `requests` solves at `rate` per
    second (the serving mix, run to steady state), the continuous-batching loop
    against the plain solver serving the same trace one request at a time
    (FIFO, within plain_budget seconds).  Returns a dict."""
    from paper_1209_6548_gb300 import serve as S

    probs = S.serving_mix(requests, seed=seed, cavity_share=cavity_share)
    conv = S.Convergence()
    warm = S.ServingLoop(capacity=8, pool_bytes=int(pool_mb * 2**20), stream=stream, conv=conv)
    warm.run(S.poisson_trace(8, rate, probs[:8], seed=99))  # kernel loading, graph build
    warm.batch.close()
    loop = S.ServingLoop(capacity=1024, pool_bytes=int(pool_mb * 2**20), stream=stream, conv=conv)
    reqs = S.poisson_trace(requests, rate, probs, seed=seed)
    with ClockSampler(local) as clk:
        t0 = time.perf_counter()
        done = loop.run(reqs)
        wall = time.perf_counter() - t0
    loop.batch.close()
    served = S.latency_summary(done)
    plain_reqs = S.poisson_trace(requests, rate, probs, seed=seed)
    p0 = time.perf_counter()
    plain_done = S.run_plain_fifo(plain_reqs, conv=conv, stream=stream, time_budget=plain_budget)
    plain_wall = time.perf_counter() - p0
    plain = S.latency_summary(plain_done)
    clocks = clk.summary()
    return {"requests": requests, "rate_per_s": rate, "pool_mb": pool_mb, "check_every": loop.check_every,
            "solves_per_s": served.get("solves_per_s"), "completed": served.get("completed"),
            "latency": {"p50_s": served.get("p50_s"), "p99_s": served.get("p99_s"), "mean_s": served.get("mean_s")},
            "status": served.get("status"), "wall_s": wall,
            "convergence": "r < 1e-8, or steady_drift: Aitken transient of r < 1e-8 with the total mass drifting "
                           "linearly (the wall rule's mass exchange); cap 400k steps",
            "plain_fifo": {**plain, "wall_s": plain_wall, "budget_s": plain_budget,
                           "note": "the same trace, one request at a time, within the budget"},
            "clocks": {"sm_mhz": clocks["sm_mhz"], "sm_max_mhz": clocks["sm_max_mhz"], "reasons": clocks["reasons"]}}


def run_batch(args, world, rank, local):
    """Batched solves: the seeded mix of independent channel flows (nx = 4, ny
    log-uniform 16-1024, Couette / Fourier / Poiseuille, Kn log-uniform
    0.01-0.5, b in {-1/2, 0, 1/2}, D2Q16), each run for 2000 steps.  One bench
    step = admit every instance into the batch, 2000 steps for all, the nine
    moment fields of every instance.  value = solves/s.  The plain solver runs a
    sample of the same instances one at a time (lesbgk_create, lesbgk_step,
    lesbgk_moments) for the baseline.  Second mode (unless --no-steady): the
    same instances run to steady state (r < 1e-8, or settled on the wall-mass
    drift, as in the serving loop) in one batch, all admitted at once, against
    the plain solver running them to steady state one at a time within
    --plain-budget; solves/s counts solved instances only."""
    import collections
    import numpy as np
    import torch
    from paper_1209_6548_gb300 import build as B
    from paper_1209_6548_gb300 import inputs as I
    from paper_1209_6548_gb300 import lesbgk as L
    from paper_1209_6548_gb300 import serve as S

    from paper_1209_6548_gb300 import shard as SH

    torch.cuda.set_device(local)
    pg = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
        pg = dist
    B.build()
    nsteps = args.lattice_steps if args.lattice_steps != 1000 else 2000
    # one mix of instances x world solves, split across ranks by cost (LPT)
    all_probs = I.batch_mix(n=args.instances * world, seed=0, steps=nsteps)
    _, probs = SH.shard(all_probs, rank, world, steps=nsteps)
    params = [L.params_from_problem(p) for p in probs]

    def barrier():
        torch.cuda.synchronize()
        if pg is not None:
            pg.barrier()

    def max_over_ranks(x):
        if pg is None:
            return x
        t = torch.tensor([x], dtype=torch.float64, device="cuda")
        pg.all_reduce(t, op=pg.ReduceOp.MAX)
        return float(t.item())
    stream = torch.cuda.current_stream()
    fixed, step_ms, rows, pool = measure_batch_fixed(params, nsteps, args.steps, args.warmup, stream, local,
                                                     args.plain_sample, barrier, max_over_ranks)
    n = len(params)
    wsec = fixed["wall_s"]
    value = len(all_probs) * args.steps / wsec
    idx = list(range(0, n, max(1, n // args.plain_sample)))[: args.plain_sample]
    cells = sum(4 * p.ny for p in params)
    peak, peak_kind = measured_peak()
    eff = 2 * 16 * 4 * cells / (step_ms / 1e3) / 1e9
    clocks = fixed["clocks"]
    steady = None
    if not args.no_steady:
        reqs = [S.Request(rid=k, arrival=0.0, problem=p) for k, p in enumerate(probs)]
        loop = S.ServingLoop(capacity=n, pool_bytes=pool, stream=stream)
        barrier()
        t0 = time.perf_counter()
        done = loop.run(reqs)
        barrier()
        ssec = max_over_ranks(time.perf_counter() - t0)
        loop.batch.close()
        steps = np.array([r.steps for r in done])
        plain_reqs = [S.Request(rid=k, arrival=0.0, problem=probs[i]) for k, i in enumerate(idx)]
        pdone = S.run_plain_fifo(plain_reqs, stream=stream, time_budget=args.plain_budget)
        pwall = sum(r.completed - r.admitted for r in pdone)
        solved = [r for r in done if r.status in S.SOLVED]
        psolved = [r for r in pdone if r.status in S.SOLVED]
        steady = {"solves_per_s": len(solved) * world / ssec, "wall_s": ssec, "solved": len(solved),
                  "status": dict(collections.Counter(r.status for r in done)),
                  "steps_median": float(np.median(steps)), "steps_max": int(steps.max()),
                  "criterion": "r < 1e-8, or steady_drift: Aitken transient of r < 1e-8 with the total mass "
                               "drifting linearly (the wall rule's mass exchange); cap 400k steps",
                  "plain": {"solved": len(psolved), "solves_per_s": len(psolved) / max(pwall, 1e-9),
                            "status": dict(collections.Counter(r.status for r in pdone)),
                            "sample": f"the first {len(pdone)} of {len(idx)} sampled instances within "
                                      f"{args.plain_budget:g} s, one at a time"}}
    line = {
        "metric": "batched solves/s", "value": value, "unit": "solves/s", "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": wsec / args.steps * 1e3, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": f"batch_mix_{args.instances}_per_gpu_nx4_d2q16", "instances": len(all_probs),
                   "instances_this_rank": n, "sharding": "LPT by nodes x steps", "lattice_steps_per_solve": nsteps,
                   "total_nodes": cells, "rows_per_item": rows, "graph_steps": 64,
                   "l2": "L2 flushed between timed passes (256 MB write); within a pass the %.0f MB working "
                         "set is partly L2-resident" % (2 * 64 * cells / 1e6)},
        "instance_mlups": sum(4 * p.ny * nsteps for p in all_probs) * args.steps / wsec / 1e6,
        "launch": fixed["launch"], "step_ms_by_mode": fixed["step_ms_by_mode"],
        "plain": fixed["plain"],
        "roofline": {"bound": "hbm", "achieved": eff, "peak": peak, "unit": "GB/s", "frac": eff / peak,
                     "traffic": None, "peak_source": peak_kind, "kernel": "k_batch_step<4,3,4>",
                     "kernel_ms": step_ms,
                     "note": "algorithmic bytes of one batch step over its time; the working set is served "
                             "partly from L2 (about 40% of the reads in the ncu capture)"},
        # per pass at least: one init launch or more (the staged fields), one step kernel per step
        # (one per chain of the class), one moment launch
        "gpu_launches": (1 + nsteps + 1) * args.steps,
        "clocks": {"sm_mhz": clocks["sm_mhz"], "sm_max_mhz": clocks["sm_max_mhz"], "reasons": clocks["reasons"]},
        "steady": steady,
    }
    if rank == 0:
        print(json.dumps(line), flush=True)
    if pg is not None:
        pg.destroy_process_group()
    return 0


def run_serve(args, world, rank, local):
    """Serving: a seeded Poisson stream (args.rate per second) of channel solves
    (the batched mix with ny 16-512 and 20% on D2Q36) and 10% lid-driven
    256^2 cavities (served beside the batch by the wide lane), each run to steady state
    (residual below 1e-8, or a residual that has stopped changing); admission
    by a fixed device-memory pool.  Reports p50/p99 latency (completion minus
    arrival), solves/s and offered vs achieved load, against the plain solver
    serving the same trace one request at a time (FIFO)."""
    import numpy as np
    import torch
    from paper_1209_6548_gb300 import build as B
    from paper_1209_6548_gb300 import serve as S

    torch.cuda.set_device(local)
    B.build()
    stream = torch.cuda.current_stream()
    sv = measure_serve(args.requests, args.rate, args.pool_mb, args.plain_budget, stream, local, seed=rank)
    line = {
        "metric": "served solves/s (p50/p99 latency)", "value": sv["solves_per_s"], "unit": "solves/s",
        "n_gpus": world, "steps": 1, "warmup": 1, "ms_per_step": sv["wall_s"] * 1e3, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": f"serve_{args.requests}_poisson{args.rate:g}", "requests": args.requests,
                   "rate_per_s": args.rate, "pool_mb": args.pool_mb, "check_every": sv["check_every"],
                   "mix": "nx 4, ny 16-512, Couette/Fourier/Poiseuille, Kn 0.01-0.5, 20% D2Q36; "
                          "10% lid-driven cavities 256^2 (lid 0.05, Kn 0.05-0.5) in the wide lane",
                   "convergence": sv["convergence"]},
        "latency": sv["latency"], "offered_per_s": args.rate, "achieved_per_s": sv["solves_per_s"],
        "status": sv["status"], "wall_s": sv["wall_s"], "plain_fifo": sv["plain_fifo"],
        "gpu_launches": None, "clocks": sv["clocks"],
    }
    if rank == 0:
        print(json.dumps(line), flush=True)
    return 0


def run_slab(args, world, rank, local):
    """One 4096^2 solve split over the ranks in y-slabs (slab.py): each rank's
    solver holds its slab plus a halo of 2k rows, exchanged with its
    neighbours over NCCL every k steps (k = --halo-steps); the conservation
    totals are one FP64 allreduce.  value = the whole domain's lattice
    updates per second (strong scaling: the work is fixed as N grows)."""
    import numpy as np
    import torch
    import torch.distributed as dist
    from paper_1209_6548_gb300 import build as B
    from paper_1209_6548_gb300 import inputs as I
    from paper_1209_6548_gb300 import lesbgk as L
    from paper_1209_6548_gb300 import slab as SL

    torch.cuda.set_device(local)
    if "MASTER_ADDR" in os.environ:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    else:  # one process without torchrun: a group of one
        import socket
        with socket.socket() as sk:
            sk.bind(("127.0.0.1", 0))
            port = sk.getsockname()[1]
        dist.init_process_group("nccl", init_method=f"tcp://127.0.0.1:{port}", rank=0, world_size=1,
                                device_id=torch.device("cuda", local))
    B.build()
    n, nsteps, k = args.n, args.lattice_steps, args.halo_steps
    nroots, dim, order, q = LATTICES[args.velocity_set]
    prob = tgv_problem(n, args, nsteps)
    fields = I.initial_fields(prob)
    storage = {"f32": L.F32, "f16": L.F16, "bf16": L.BF16, "f32c": L.F32C}[args.storage]
    stream = torch.cuda.current_stream()
    # the whole domain's time step (tau_ref depends on its fields) and spacing, as the library sets them
    whole = L.Solver(L.params_from_problem(prob), h_init=fields, stream=stream)
    dt, dx, dy = whole.info.dt, whole.info.dx, whole.info.dy
    whole.close()
    del whole
    torch.cuda.empty_cache()
    slab = SL.partition(n, world, 2 * k, True)[rank]
    st = SL.GpuSlab(prob, slab, fields, dt, dx, dy, storage, stream=stream)
    d_fields = torch.from_numpy(SL.slab_fields(fields, slab)).cuda()
    mom = torch.empty((9, slab.rows, n), dtype=torch.float32, device="cuda")

    def one_solve(ev=None):
        st.solver.reinit(d_fields)
        SL.exchange_dist(st, slab, dist)
        if ev is not None:
            ev[0].record(stream)
        done = 0
        while done < nsteps:
            m = min(k, nsteps - done)
            st.step(m)
            done += m
            if m == k and done < nsteps:
                SL.exchange_dist(st, slab, dist)
        if ev is not None:
            ev[1].record(stream)
        hs = np.zeros(4)
        L._check(L.lib().lesbgk_moments_rows(L.C.c_void_p(st.solver.handle), slab.lo, slab.rows,
                                            L.C.c_void_p(mom.data_ptr()), L.C.c_void_p(hs.ctypes.data),
                                            L.C.c_void_p(stream.cuda_stream)))
        tot = torch.tensor(hs, dtype=torch.float64, device="cuda")
        dist.all_reduce(tot)  # the decomposition's one FP64 reduction
        return tot

    for _ in range(args.warmup):
        one_solve()
    torch.cuda.synchronize()
    dist.barrier()
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    with ClockSampler(local) as clk:
        torch.cuda.synchronize()
        dist.barrier()
        w0 = time.perf_counter()
        for i in range(args.steps):
            tot = one_solve(evs[i])
        torch.cuda.synchronize()
        dist.barrier()
        wall = time.perf_counter() - w0
    t = torch.tensor([wall], dtype=torch.float64, device="cuda")
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    wall = float(t.item())
    step_ms = sum(a.elapsed_time(b) for a, b in evs) / (args.steps * nsteps)
    clocks = clk.summary()
    lups = n * n * nsteps * args.steps

    # end to end through the C ABI with host buffers: each rank creates its
    # slab's solver from pinned host fields (lesbgk_create) and reads its own
    # rows' moments back to pinned host memory
    e2e = None
    if not args.no_e2e:
        h_fields = torch.from_numpy(SL.slab_fields(fields, slab)).pin_memory()
        h_out = torch.empty((9, slab.rows, n), dtype=torch.float32).pin_memory()
        params = st.solver.params
        ws, nbytes = st.solver.workspace, st.solver.nbytes
        st.solver.close()

        class _Handle:  # the store the exchange drives, around a raw handle
            def __init__(self, h):
                self.solver = type("S", (), {"handle": h, "stream": stream})()

        def e2e_solve():
            h = L.create(params, ws.data_ptr(), nbytes, h_fields.numpy(), stream.cuda_stream)
            hs = _Handle(h)
            store = SL.GpuSlab.__new__(SL.GpuSlab)
            store._torch, store._L, store.slab, store.solver = torch, L, slab, hs.solver
            SL.exchange_dist(store, slab, dist)
            done = 0
            while done < nsteps:
                m = min(k, nsteps - done)
                L.step(h, m, stream.cuda_stream)
                done += m
                if m == k and done < nsteps:
                    SL.exchange_dist(store, slab, dist)
            hsum = np.zeros(4)
            L._check(L.lib().lesbgk_moments_rows(L.C.c_void_p(h), slab.lo, slab.rows, L.C.c_void_p(mom.data_ptr()),
                                                L.C.c_void_p(hsum.ctypes.data), L.C.c_void_p(stream.cuda_stream)))
            h_out.copy_(mom, non_blocking=True)
            tot = torch.tensor(hsum, dtype=torch.float64, device="cuda")
            dist.all_reduce(tot)
            torch.cuda.synchronize()
            L.destroy(h)

        for _ in range(2):
            e2e_solve()
        torch.cuda.synchronize()
        dist.barrier()
        w0 = time.perf_counter()
        for _ in range(args.steps):
            e2e_solve()
        torch.cuda.synchronize()
        dist.barrier()
        t = torch.tensor([time.perf_counter() - w0], dtype=torch.float64, device="cuda")
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        e2e = {"value": lups / float(t.item()) / 1e6, "unit": UNIT,
               "h2d_bytes_per_step": int(h_fields.numel() * 8) * world,
               "d2h_bytes_per_step": int(h_out.numel() * 4 + 4 * 8) * world}
    if rank == 0:
        line = {
            "metric": METRIC, "value": lups / wall / 1e6, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": wall / args.steps * 1e3, "higher_is_better": True,
            "scaling": "strong", "vs_baseline": None, "dtype": args.storage, "data": "synthetic",
            "config": {"workload": tgv_workload_name(n, args), "nx": n, "ny": n,
                       "velocity_set": args.velocity_set.upper(), "storage": args.storage, "order": order,
                       "lattice_steps_per_step": nsteps, "scheme": "split",
                       "parallelism": (f"y-slabs x{world}: {slab.rows} or so rows per rank, halo {2 * k} rows "
                                       f"exchanged over NCCL every {k} steps") if world > 1 else
                                      "one slab: the whole domain, no exchange",
                       "l2": "inputs larger than L2"},
            "slab_ms_per_lattice_step_rank0": step_ms,
            "totals": tot.cpu().numpy().tolist(),
            "e2e": e2e,
            "gpu_launches": (1 + nsteps + 2) * args.steps,
            "clocks": {"sm_mhz": clocks["sm_mhz"], "sm_max_mhz": clocks["sm_max_mhz"], "reasons": clocks["reasons"]},
        }
        print(json.dumps(line), flush=True)
    if args.no_e2e:
        st.close()
    dist.destroy_process_group()
    return 0


def run_precision(args, world, rank, local):
    """Per-field error of FP32, FP16, BF16 and compensated FP32 population
    storage (FP32 compute) against the FP64 oracle: an n^2 Taylor-Green vortex
    (split scheme; n = --tgv-n, 256 by default, 4096 for the throughput
    workload itself, compared at every 8th node in x and y there) and the
    force-driven Poiseuille channel (g = 1e-4, Kn 0.2, b = 0, ny = 1024; the
    flow does not vary in x, so a 4-node-wide periodic slice computes the same
    solution as the 512-wide channel), 1000 steps each.  Errors per field as
    in the parity tests: e = max|gpu - ref| / (largest magnitude of the
    field's quantity), e_own = ... / max|ref field|, e_pert = ... /
    max|ref - rest value|.
    --save-moments DIR: the GPU leg only, writing its sampled moments to DIR;
    --compare-moments DIR: the oracle leg only, against moments so saved (the
    4096^2 oracle run takes hours: it may run on other host cores than the GPU
    box's)."""
    import numpy as np
    import oracle as O
    from dataclasses import replace
    from paper_1209_6548_gb300 import inputs as I

    steps = 1000
    cases = [(f"tgv{args.tgv_n}", I.tgv(args.tgv_n, steps=steps)),
             ("poiseuille_1024", I.poiseuille(nx=4, ny=1024, steps=steps))]
    stores = ("f32", "f16", "bf16", "f32c")
    groups = {"rho": ["rho"], "T": ["T"], "u": ["ux", "uy"], "sigma": ["sxx", "sxy", "syy"], "q": ["qx", "qy"]}
    names = list(O.MOMENT_NAMES)
    rest = np.zeros(9)
    rest[0] = rest[3] = 1.0

    def stride(prob):
        return 8 if prob.nx >= 2048 else 1

    def time_step_of(prob, fields):
        # the time step the library takes (its rule, restated on the test side)
        from tests.common import time_step
        return time_step(prob, fields)

    gpu = {}
    thr = {}
    if not args.compare_moments:
        import torch
        from paper_1209_6548_gb300 import build as B
        from paper_1209_6548_gb300 import lesbgk as L
        torch.cuda.set_device(local)
        B.build()
        code = {"f32": L.F32, "f16": L.F16, "bf16": L.BF16, "f32c": L.F32C}
        for cname, prob in cases:
            fields = I.initial_fields(prob) if prob.init == "tgv" else None
            dt = time_step_of(prob, fields)
            k = stride(prob)
            for st in stores:
                p = L.params_from_problem(prob, dt=dt)
                p.storage = code[st]
                sv = L.Solver(p, h_init=fields)
                sv.step(steps)
                gpu[(cname, st)] = sv.moments()[:, ::k, ::k].cpu().numpy().astype(np.float64)
                sv.close()
        if args.save_moments:
            os.makedirs(args.save_moments, exist_ok=True)
            np.savez(os.path.join(args.save_moments, f"gpu_moments_tgv{args.tgv_n}.npz"),
                     **{f"{c}|{st}": v.astype(np.float32) for (c, st), v in gpu.items()})  # the GPU's own FP32
        # throughput of each storage on the 4096^2 case
        n = 4096
        prob = I.tgv(n)
        fields = I.initial_fields(prob)
        stream = torch.cuda.current_stream()
        for st in stores:
            p = L.params_from_problem(prob)
            p.storage = code[st]
            sv = L.Solver(p, h_init=fields, stream=stream)
            sv.step(20)
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            sv.step(200)
            e1.record(stream)
            torch.cuda.synchronize()
            ms = e0.elapsed_time(e1) / 200
            bpl = 2 * 16 * STORE_BYTES[st]
            thr[st] = {"mlups": n * n / (ms / 1e3) / 1e6, "kernel_ms": ms,
                       "gbs": bpl * n * n / (ms / 1e3) / 1e9, "bytes_per_lup": bpl}
            sv.close()
        if args.save_moments:
            line = {"metric": "GPU moments saved for the precision comparison", "dir": args.save_moments,
                    "throughput_4096": thr, "source_sha256": source_digest()}
            if rank == 0:
                print(json.dumps(line), flush=True)
            return 0
    else:
        z = np.load(os.path.join(args.compare_moments, f"gpu_moments_tgv{args.tgv_n}.npz"))
        gpu = {tuple(key.split("|")): z[key].astype(np.float64) for key in z.files}

    O.set_threads(len(os.sched_getaffinity(0)))
    out = {}
    t_or = 0.0
    from tests.common import oracle_params
    for cname, prob in cases:
        fields = I.initial_fields(prob) if prob.init == "tgv" else None
        dt = time_step_of(prob, fields)
        op = oracle_params(prob, dt)
        t0 = time.perf_counter()
        ref, _ = O.moments(op, O.run(op, O.init(op, fields), steps))
        t_or += time.perf_counter() - t0
        k = stride(prob)
        ref = ref[:, ::k, ::k]
        for st in stores:
            g = gpu[(cname, st)]
            row = {}
            for grp, mem in groups.items():
                scale = max(float(np.max(np.abs(ref[names.index(m)]))) for m in mem)
                for m in mem:
                    i = names.index(m)
                    d = float(np.max(np.abs(g[i] - ref[i])))
                    own = float(np.max(np.abs(ref[i])))
                    pert = float(np.max(np.abs(ref[i] - rest[i])))
                    row[m] = {"e": d / scale, "e_own": d / own if own > 0 else None,
                              "e_pert": (d / pert) if pert > 1e-6 else None, "abs": d}
            out.setdefault(cname, {})[st] = row
    worst = {st: max(max(v["e"] for v in out[c][st].values()) for c in out) for st in stores}
    line = {"metric": "per-field error vs FP64 oracle by population storage", "value": worst["f32"],
            "unit": "max relative error (FP32 storage)", "n_gpus": world, "steps": steps, "warmup": 0,
            "higher_is_better": False, "dtype": "f32 compute", "data": "synthetic",
            "config": {"workload": f"precision_tgv{args.tgv_n}_poiseuille1024", "lattice_steps": steps,
                       "cases": [c for c, _ in cases], "sampled_every": {c: stride(p) for c, p in cases}},
            "worst_e": worst, "errors": out, "throughput_4096": thr or None,
            "oracle_seconds": t_or, "cpu_cores": O.get_threads()}
    if rank == 0:
        print(json.dumps(line), flush=True)
    return 0


def main():
    args = parse()
    world, rank, local = dist_setup()
    if args.impl == "reference":
        return run_reference(args, world, rank)
    if args.workload == "batch":
        return run_batch(args, world, rank, local)
    if args.workload == "serve":
        return run_serve(args, world, rank, local)
    if args.workload == "precision":
        return run_precision(args, world, rank, local)
    if args.workload == "slab" or (world > 1 and args.decomp == "slab"):
        return run_slab(args, world, rank, local)

    import numpy as np
    import torch
    from paper_1209_6548_gb300 import build as B
    from paper_1209_6548_gb300 import inputs as I
    from paper_1209_6548_gb300 import lesbgk as L

    torch.cuda.set_device(local)
    pg = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
        pg = dist

    def barrier():
        torch.cuda.synchronize()
        if pg is not None:
            pg.barrier()
        torch.cuda.synchronize()

    def max_over_ranks(x: float) -> float:
        if pg is None:
            return x
        t = torch.tensor([x], dtype=torch.float64, device="cuda")
        pg.all_reduce(t, op=pg.ReduceOp.MAX)
        return float(t.item())

    B.build()
    n, nsteps = args.n, args.lattice_steps
    nroots, dim, order, q = LATTICES[args.velocity_set]
    prob = tgv_problem(n, args, nsteps)
    fields = I.initial_fields(prob)
    params = L.params_from_problem(prob, dt=0.0)
    params.storage = {"f32": L.F32, "f16": L.F16, "bf16": L.BF16, "f32c": L.F32C}[args.storage]
    stream = torch.cuda.current_stream()
    d_fields = torch.from_numpy(fields).cuda()
    solver = L.Solver(params, h_init=fields, stream=stream)
    d_mom = torch.empty((9, n, n), dtype=torch.float32, device="cuda")
    cells = n * n
    launches_per_step = 1 + nsteps + 1  # init, steps, moments (no totals asked for)
    info = solver.info
    shape = (info.cells_per_thread, info.rows_per_segment)

    def one_solve(ev=None):
        solver.reinit(d_fields)
        if ev is not None:
            ev[0].record(stream)
        solver.step(nsteps)
        if ev is not None:
            ev[1].record(stream)
        L.moments(solver.handle, d_mom.data_ptr(), None, stream.cuda_stream)

    for _ in range(args.warmup):
        one_solve()
    barrier()
    step_events = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
                   for _ in range(args.steps)]
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with ClockSampler(local) as clk:
        t0.record(stream)
        for k in range(args.steps):
            one_solve(step_events[k])
        t1.record(stream)
        torch.cuda.synchronize()
    barrier()
    ms = max_over_ranks(t0.elapsed_time(t1))
    kernel_ms = sum(a.elapsed_time(b) for a, b in step_events) / (args.steps * nsteps)
    kernel_ms = max_over_ranks(kernel_ms)
    lups = cells * nsteps * args.steps * world
    value = lups / (ms / 1e3) / 1e6

    # end to end through the C ABI with host buffers
    e2e = None
    if not args.no_e2e:
        h_fields = torch.from_numpy(fields).pin_memory()
        h_out = torch.empty((9, n, n), dtype=torch.float32).pin_memory()
        h_sums = np.zeros(4)
        ws = solver.workspace
        nbytes = solver.nbytes
        solver.close()
        h2d = fields.nbytes
        d2h = h_out.numel() * 4 + h_sums.nbytes

        # double-buffered through the public calls: two workspaces, two
        # streams; solve k's upload and checks (lesbgk_create, which waits for
        # its own stream only) run while solve k-1 steps, and solve k-1's
        # moments come back to the host (lesbgk_moments_host) while solve k
        # steps; the solves' steps themselves run one solve after another
        # (each waits for the previous solve's last step), and every solve's
        # copies are inside the timed region
        ws2 = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        lanes = [(ws, stream), (ws2, torch.cuda.Stream())]

        def e2e_run(count, marks=None):
            prev = None
            stepped = None  # event after the previous solve's last step
            for k in range(count):
                w, s = lanes[k % 2]
                h = L.create(params, w.data_ptr(), nbytes, h_fields.numpy(), s.cuda_stream)
                if stepped is not None:
                    s.wait_event(stepped)
                L.step(h, nsteps, s.cuda_stream)
                stepped = torch.cuda.Event()
                stepped.record(s)
                if prev is not None:
                    L.moments_host(prev[0], h_out.numpy(), h_sums, prev[1].cuda_stream)
                    L.destroy(prev[0])
                    if marks is not None:
                        marks.append(time.perf_counter())
                prev = (h, s)
            L.moments_host(prev[0], h_out.numpy(), h_sums, prev[1].cuda_stream)
            L.destroy(prev[0])
            if marks is not None:
                marks.append(time.perf_counter())

        e2e_run(max(2, args.warmup // 2))
        barrier()
        marks = []
        with ClockSampler(local) as eclk:
            w0 = time.perf_counter()
            e2e_run(args.steps, marks)
            barrier()
            wsec = max_over_ranks(time.perf_counter() - w0)
        ec = eclk.summary()
        done_ms = [(t - w0) * 1e3 for t in marks]  # when each solve's moments were on the host
        e2e = {"value": cells * nsteps * args.steps * world / wsec / 1e6, "unit": UNIT,
               "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h, "solve_done_ms": done_ms,
               "pipeline": "two workspaces and streams: solve k's upload overlaps solve k-1's steps, "
                           "solve k-1's download overlaps solve k's steps; the steps of the solves run in turn",
               "clocks": {"sm_mhz": ec["sm_mhz"], "reasons": ec["reasons"]}}
        del ws2, lanes

    # the same solve in the storage that meets the 1e-5 bar at this size
    prec_obj = None
    if (world == 1 and not args.no_precision and args.velocity_set == "d2q16" and args.storage == "f32"
            and n == 4096 and nsteps == 1000):
        prec_obj = measure_compensated(prob, fields, nsteps, 2, 1, stream, local)

    # the batched and served forms of the metric, each with its own timed
    # region, on one GPU (the config-4 and config-5 workloads at bench size)
    batch_obj = serve_obj = None
    if world == 1 and not args.no_batch:
        bprobs = I.batch_mix(n=args.instances, seed=0, steps=2000)
        bfixed, bstep_ms, brows, _ = measure_batch_fixed([L.params_from_problem(p) for p in bprobs], 2000,
                                                         args.steps, args.warmup, stream, local, args.plain_sample)
        batch_obj = {"workload": f"batch_mix_{args.instances}_nx4_d2q16", "instances": args.instances,
                     "lattice_steps_per_solve": 2000, "solves_per_s": bfixed["solves_per_s_this_rank"],
                     "vs_plain": bfixed["solves_per_s_this_rank"] / bfixed["plain"]["est_solves_per_s_full_mix"],
                     **{k: v for k, v in bfixed.items() if k != "solves_per_s_this_rank"},
                     "l2": "L2 flushed between timed passes"}
    if world == 1 and not args.no_serve:
        serve_obj = measure_serve(args.serve_requests, args.rate, args.pool_mb, args.serve_plain_budget, stream,
                                  local, seed=0)
        serve_obj["vs_plain_solves_per_s"] = ((serve_obj["solves_per_s"] or 0.0) /
                                              max(serve_obj["plain_fifo"].get("solves_per_s") or 1e-9, 1e-9))

    peak, peak_kind = measured_peak()
    bytes_per_lup = 2 * q * STORE_BYTES[args.storage]  # q: values stored per node
    achieved = bytes_per_lup * cells / (kernel_ms / 1e3) / 1e9
    digest = source_digest()
    traffic = committed_traffic(digest, args.velocity_set, args.storage)
    base = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        rows, steps = {"d2q16": (1024, 48), "d2q36": (256, 48), "d3q64": (256, 48),
                       "d3q216": (8, 8)}[args.velocity_set]  # about 10-30 s of oracle work
        base = cpu_baseline(n, rows=rows, steps=steps, velocity_set=args.velocity_set)
    if rank == 0:
        clocks = clk.summary()
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": tgv_workload_name(n, args), "nx": n, "ny": n,
                       "velocity_set": args.velocity_set.upper(), "storage": args.storage,
                       "order": order, "kn": prob.kn, "b": prob.b,
                       "lattice_steps_per_step": nsteps, "scheme": "split",
                       "l2": ("inputs larger than L2 (two population buffers of %.2f GB)"
                              if q * n * n * STORE_BYTES[args.storage] > L2_BYTES else
                              "a small case: the two population buffers of %.2f GB fit in L2")
                             % (q * n * n * STORE_BYTES[args.storage] / 1e9),
                       "parallelism": f"replica x{world}"},
            "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
                         "frac": achieved / peak, "traffic": traffic, "peak_source": peak_kind,
                         "kernel": (f"k_step<{nroots},{order},split,{args.storage},nz={q // (nroots * nroots)}> "
                                    if q // (nroots * nroots) < 3 else "k_step_z<split> (one warp per z-level) ")
                                   + f"rows={shape[1]}",
                         "kernel_ms": kernel_ms,
                         "bytes_per_lup": bytes_per_lup, "source_sha256": digest,
                         "of_nominal_hbm": achieved / 7900.0,
                         "issue": issue_view(committed_instructions(digest, args.velocity_set, args.storage), cells,
                                             kernel_ms, torch.cuda.get_device_properties(local).multi_processor_count,
                                             clocks["sm_mhz"])},
            "cpu_baseline": base,
            "e2e": e2e,
            "precision": prec_obj,
            "batch": batch_obj,
            "serve": serve_obj,
            "gpu_launches": launches_per_step * args.steps,
            "clocks": {"sm_mhz": clocks["sm_mhz"], "sm_max_mhz": clocks["sm_max_mhz"],
                       "reasons": clocks["reasons"]},
        }
        print(json.dumps(line), flush=True)
    if pg is not None:
        pg.destroy_process_group()
    return 0


if __name__ == "__main__":
    sys.exit(main())
