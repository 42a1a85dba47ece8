#!/usr/bin/env python
"""Benchmark: FP64 RK3 time steps of the reacting Navier-Stokes right-hand side on one GB300.

Workload: the oblique-shock / boundary-layer interaction on 2048 x 256 cells (five-species air,
17 reactions, artificial diffusivity on; paper_2210_05547_gb300.inputs.sbli_case). One step is a
full two-register RK3 step: three right-hand sides and three stage updates, every kernel of the
hot path. Metric: Mpts*RHS/s = cells x right-hand sides per second over all GPUs.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

With N > 1 the script is launched by torch.distributed.run, one process per GPU; each rank runs
an independent replica (seed = rank), no collective on the data path ("weak" scaling). Inputs
are resident in HBM for `value`; `e2e` repeats the measurement through the public API with the
state copied from pinned host memory and back every step. The L2 cache is flushed between timed
steps by writing a 256 MiB buffer outside the timed events.
"""
from __future__ import annotations

import argparse
import json
import os
import resource
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "Mpts*RHS/s FP64"
UNIT = "Mpts*RHS/s"
STAGES = 3
L2_FLUSH_BYTES = 256 << 20
# Most of the path runs on 64-bit integers, so rooflines are in warp instructions: executed (ncu's
# smsp__inst_executed, as thread instructions per cell: 32 per warp instruction) against four per
# clock and SM; the binary64 unit's instructions (sm__inst_executed_pipe_fp64) against its two lanes
# per clock and SM beside them (profiles/instructions_per_case.md).
ISSUE_PEAK_TINSTR = 152 * 4 * 32 * 2.07e9 / 1e12      # thread instructions
FP64_PEAK_TINSTR = 152 * 2 * 2.07e9 / 1e12
PEAK_SOURCE = "derived: 152 SMs x 4 warp instructions/clk x 32 x 2.07 GHz"
# instructions per cell (state): (all, binary64 unit)
CLOSURE_INSTR = (15496, 284.7)
CLOSURE3_INSTR = (14698, 438.5)
THERMO_INSTR = (19944, 417.1)
RHS_INSTR = (52789, 714.7)              # of the RK3 step of the shock case at 1024 x 256
# DRAM bytes (read + write) of one k_closure launch per point, from ncu at 1024 x 256
CLOSURE_DRAM_BYTES_PER_POINT = 564.4


def issue_roofline(instr, units_per_s):
    """Roofline of a kernel that executes `instr` (all, binary64) per unit of work."""
    ach = instr[0] * units_per_s / 1e12
    return {"bound": "alu", "achieved": ach, "peak": ISSUE_PEAK_TINSTR,
            "unit": "T thread instructions/s", "frac": ach / ISSUE_PEAK_TINSTR,
            "instr_per_point": instr[0], "fp64_instr_per_point": instr[1],
            "fp64_pipe_frac": instr[1] * units_per_s / 1e12 / FP64_PEAK_TINSTR,
            "peak_source": PEAK_SOURCE}


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--nx", type=int, default=2048, help="cells in x (profiling of small cases)")
    ap.add_argument("--ny", type=int, default=256, help="cells in y (profiling of small cases)")
    ap.add_argument("--no-mixed", action="store_true", help="skip the mixed-precision measurement")
    ap.add_argument("--no-sm", action="store_true", help="skip the Stefan-Maxwell measurement")
    ap.add_argument("--no-lte", action="store_true", help="skip the LTE measurement")
    ap.add_argument("--no-3d", action="store_true",
                    help="skip the three-dimensional jet-in-crossflow measurement")
    ap.add_argument("--no-air11", action="store_true",
                    help="skip the eleven-species measurements")
    ap.add_argument("--serve-requests", type=int, default=24,
                    help="requests of the serving measurement, the first ones of the 500-request "
                         "serving stream (0 skips it)")
    ap.add_argument("--serve-fp64", action="store_true",
                    help="also serve the stream in FP64 through the server")
    ap.add_argument("--thermo-states", type=float, default=1e8,
                    help="states of the pointwise thermochemistry sweep (0 skips it)")
    ap.add_argument("--jet3d-size", default="512x256x128",
                    help="cells of the three-dimensional jet measurement, NXxNYxNZ (profiling of "
                         "small cases)")
    return ap.parse_args()


def workload_config(cfg, world):
    return {"workload": f"sbli_{cfg['nx']}x{cfg['ny']}_cneq5_fp64_rk3", "nx": cfg["nx"],
            "ny": cfg["ny"], "points": cfg["nx"] * cfg["ny"], "species": 5, "reactions": 17,
            "gas": cfg["kind"], "artificial_diffusivity": bool(cfg["artificial_diffusivity"]),
            "mach": round(cfg["mach"], 4), "shock_deflection_deg": round(cfg["shock_deflection_deg"], 4),
            "rhs_per_step": STAGES, "l2": "flushed between timed steps (256 MiB write)",
            "replicas": world, "parallelism": "replicas" if world > 1 else "single"}


# ------------------------------------------------------------------------------------------------
# clocks sampled with nvidia-smi during the timed region
# ------------------------------------------------------------------------------------------------

class ClockSampler:
    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, device_index):
        self.proc = None
        self.lines = []
        try:
            import torch
            p = torch.cuda.get_device_properties(device_index)
            target = f"{p.pci_domain_id:08X}:{p.pci_bus_id:02X}:{p.pci_device_id:02X}.0"
        except Exception:
            target = str(device_index)
        self.target = target

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", self.target, f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except Exception:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.thread.join(timeout=2)
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [x.strip() for x in ln.split(",")]
            if len(parts) < 8:
                continue
            try:
                sm.append(float(parts[0]))
                smax.append(float(parts[1]))
            except ValueError:
                continue
            for nm, val in zip(names, parts[4:8]):
                if val.lower() == "active":
                    reasons.add(nm)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(smax),
                "reasons": sorted(reasons), "samples": len(sm)}


# ------------------------------------------------------------------------------------------------
# CPU baseline: the oracle as it stands, on a bounded sample of the same case
# ------------------------------------------------------------------------------------------------

def _oracle_case(nx, ny):
    from oracle import flow as F
    from oracle import gas as G
    from paper_2210_05547_gb300 import inputs as I
    from paper_2210_05547_gb300.abi import TABLE_AIR5
    cfg = I.sbli_case(nx, ny)
    tab = G.load_table(TABLE_AIR5)
    n = sum(a * b for _, (a, b) in F.state_layout(5, nx, ny))
    return cfg, F.make_case(cfg, tab, I.state_noise(n, cfg["seed"]))


def _oracle_steps(cfg, case, steps):
    from oracle import flow as F
    U, dQ = case.U0.copy(), case.U0 * 0.0
    for _ in range(steps):
        for k in range(STAGES):
            U, dQ, _ = F.rk_stage(case, U, dQ, k, cfg["dt"])


# One sample size for both CPU legs (the cpu_baseline of the GPU arm and the reference arm): a
# 320 x 128 cut of the same shock/boundary-layer case; one oracle RK3 step takes a few seconds on
# one core once the operator matrices exist.
CPU_NX, CPU_NY = 320, 128


def oracle_step_rate(nx, ny, steps=1, warm=1):
    """Run `warm` untimed oracle RK3 steps (the oracle builds its operator matrices on first
    use), then `steps` timed ones, on the SBLI case at nx x ny; return (Mpts*RHS/s, cores, s)."""
    cfg, case = _oracle_case(nx, ny)
    _oracle_steps(cfg, case, warm)
    r0 = resource.getrusage(resource.RUSAGE_SELF)
    t0 = time.perf_counter()
    _oracle_steps(cfg, case, steps)
    wall = time.perf_counter() - t0
    r1 = resource.getrusage(resource.RUSAGE_SELF)
    cpu = (r1.ru_utime - r0.ru_utime) + (r1.ru_stime - r0.ru_stime)
    cores = max(1, round(cpu / wall))
    return nx * ny * STAGES * steps / wall / 1e6, cores, wall


def _oracle_proc(nx, ny, barrier, out):
    # one thread per process: numerical libraries must not start their own thread pools
    for var in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS"):
        os.environ[var] = "1"
    try:
        cfg, case = _oracle_case(nx, ny)
        _oracle_steps(cfg, case, 1)                 # untimed: operator matrices built
        barrier.wait(timeout=300)
        t0 = time.perf_counter()
        _oracle_steps(cfg, case, 1)
        out.put(("ok", time.perf_counter() - t0))
    except BaseException as exc:                    # reported to the parent, not lost
        out.put(("error", f"{type(exc).__name__}: {exc}"))


def oracle_all_cores(nx, ny, deadline_s=600.0):
    """One warmed oracle RK3 step of the nx x ny sample in each of as many processes as the host
    has cores (spawned, no GPU), all started together. Returns a dict: value (Mpts*RHS/s of the
    whole host), cores, slowest step in s; or {"unavailable": reason} when a process fails or the
    deadline passes."""
    import multiprocessing
    import queue
    nproc = max(1, min(64, len(os.sched_getaffinity(0))))
    try:
        ctx = multiprocessing.get_context("spawn")
        barrier, out = ctx.Barrier(nproc), ctx.Queue()
        procs = [ctx.Process(target=_oracle_proc, args=(nx, ny, barrier, out))
                 for _ in range(nproc)]
        for p in procs:
            p.start()
    except Exception as exc:
        return {"unavailable": f"could not start {nproc} processes: {type(exc).__name__}: {exc}"}
    walls, errors, t_end = [], [], time.monotonic() + deadline_s
    while len(walls) + len(errors) < nproc and time.monotonic() < t_end:
        try:
            kind, val = out.get(timeout=2.0)
            (walls if kind == "ok" else errors).append(val)
        except queue.Empty:
            dead = [p.exitcode for p in procs if p.exitcode not in (None, 0)]
            if dead and len(walls) + len(errors) < nproc:
                errors.append(f"process exit codes {sorted(set(dead))}")
                break
    for p in procs:
        p.join(timeout=10 if len(walls) == nproc else 0.1)
        if p.is_alive():
            p.terminate()
            p.join(timeout=10)
    if len(walls) < nproc:
        why = errors[0] if errors else f"deadline of {deadline_s:.0f} s passed"
        return {"unavailable": f"{len(walls)} of {nproc} processes finished: {why}"}
    return {"value": nproc * nx * ny * STAGES / max(walls) / 1e6, "cores": nproc,
            "slowest_s": max(walls)}


# ------------------------------------------------------------------------------------------------
# arms
# ------------------------------------------------------------------------------------------------

def reference_arm(args, rank, world):
    if rank != 0:
        return 0
    from paper_2210_05547_gb300 import inputs as I
    cfg = I.sbli_case()
    nx, ny = CPU_NX, CPU_NY   # the same bounded sample as the cpu_baseline leg
    for _ in range(args.warmup):
        oracle_step_rate(nx, ny, warm=0)
    rates, walls, cores = [], [], 1
    for _ in range(args.steps):
        r, cores, w = oracle_step_rate(nx, ny, warm=0)
        rates.append(r)
        walls.append(w)
    total = sum(walls)
    value = nx * ny * STAGES * args.steps / total / 1e6
    sample = (f"oracle RK3 steps on the same shock/boundary-layer case at {nx}x{ny} cells "
              f"(full workload 2048x256), one step per timed iteration")
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * total / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": workload_config(cfg, 1),
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle",
                             "sample": sample},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


def max_over_ranks(ms, world, device=None):
    """Time of the slowest rank, which is the whole job's time (MAX all-reduce when world > 1)."""
    import torch
    t = torch.tensor([float(ms)], dtype=torch.float64, device=device)
    if world > 1:
        import torch.distributed as dist
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_rate(world, points, steps, ms):
    """Whole-job Mpts*RHS/s: every rank advances its own replica of `points` cells."""
    return world * points * STAGES * steps / (ms / 1e3) / 1e6


def field_ranges(cfg, ns=5):
    """Offsets of each conserved field in the state vector (layout of include/hyp.h)."""
    nx, ny = cfg["nx"], cfg["ny"]
    nc = nx * ny
    names = ["rho"] + [f"rs{s}" for s in range(1, ns)] + ["rhoE"]
    out, o = {}, 0
    for name in names:
        out[name] = (o, o + nc)
        o += nc
    out["rhou"] = (o, o + (nx + 1) * ny)
    o += (nx + 1) * ny
    out["rhov"] = (o, o + nx * (ny + 1))
    return out


def table_columns(path):
    """Molar masses and charges of a gas table's species (SPECIES lines: M is the first value,
    the optional charge the fifteenth)."""
    M, q = [], []
    with open(path) as fh:
        for line in fh:
            tok = line.split("#", 1)[0].split()
            if tok[:1] == ["SPECIES"]:
                M.append(float(tok[2]))
                q.append(int(tok[15]) if len(tok) > 15 else 0)
    return M, q


def thermo_sweep(A, gas, dev, n, seed, reps=2, precision=0):
    """Throughput of hyp_thermo_eval on n independent states resident in HBM: T log-uniform in
    [300, 15000] K, rho log-uniform in [1e-4, 1] kg/m^3, mass fractions Dirichlet(1) (for a table
    with charged species: Dirichlet(1) over the heavy species and the electrons that make the
    state neutral), e = e(T, Y) from hyp_thermo_energy. All outputs requested (T, p, wdot, mu, k,
    D, status)."""
    import math
    import torch
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    ns = gas.ns
    u = torch.rand(n, generator=g, device=dev, dtype=torch.float64)
    T0 = torch.exp(math.log(300.0) + u * math.log(15000.0 / 300.0))
    u.uniform_(generator=g)
    rho = torch.exp(math.log(1e-4) + u * math.log(1e4))
    del u
    Y = torch.empty((ns, n), device=dev, dtype=torch.float64).exponential_(generator=g)
    M, q = table_columns(gas.path)
    if any(c < 0 for c in q):
        ie = q.index(-1)
        Y[ie] = 0.0
        Y /= Y.sum(dim=0, keepdim=True)
        Y[ie] = M[ie] * sum(Y[s] / M[s] for s in range(ns) if q[s] > 0)
    Y /= Y.sum(dim=0, keepdim=True)
    e = torch.empty(n, device=dev, dtype=torch.float64)
    A.thermo_energy(gas, T0, Y, e)
    T, p, mu, k = (torch.empty(n, device=dev, dtype=torch.float64) for _ in range(4))
    wdot, D = (torch.empty((ns, n), device=dev, dtype=torch.float64) for _ in range(2))
    status = torch.empty(n, device=dev, dtype=torch.uint8)
    A.thermo_eval(gas, rho, e, Y, T, p, wdot, mu, k, D, status, precision=precision)   # warm-up
    torch.cuda.synchronize()
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    ev[0].record()
    for _ in range(reps):
        A.thermo_eval(gas, rho, e, Y, T, p, wdot, mu, k, D, status, precision=precision)
    ev[1].record()
    torch.cuda.synchronize()
    ms = ev[0].elapsed_time(ev[1]) / reps
    err = float(((T - T0).abs() / T0).max())
    bad = int((status != 0).sum())
    roof = None
    if precision == 0 and ns == 5:
        roof = {"kernel": "k_thermo_eval", **issue_roofline(THERMO_INSTR, n / (ms / 1e3))}
    return {"value": n / (ms / 1e3) / 1e6, "unit": "Mstates/s", "states": n, "ms_per_sweep": ms,
            "roofline": roof,
            "bytes_per_state": 8 * (2 + ns) + 8 * (4 + 2 * ns) + 1,
            "max_rel_T_roundtrip": err, "status_nonzero": bad,
            "species": ns,
            "inputs": "T log-uniform 300-15000 K, rho log-uniform 1e-4-1 kg/m^3, Y Dirichlet(1)"
                      + (" over the heavy species, neutral" if any(c < 0 for c in q) else "")}


def serving_bench(A, I, nreq, seed, precision, air11=0.25, inflight=4, steps=(500, 2000)):
    """Continuous batching of a stream of independent solves (serving workload): a closed loop
    with `inflight` requests on the GPU measures capacity (on a short stream of 20-80 steps per
    request), then the first nreq requests of the serving stream (grids 128x32 to 1024x256, Mach
    5-20, `steps` RK3 steps each) arrive as a Poisson process at 0.8 x capacity.
    A share `air11` of the requests runs on eleven-species air, served by a second server (the
    eleven-species library) beside the five-species one on the same GPU. Reports time-to-solution
    percentiles and the throughput over the serving window."""
    import numpy as np

    def work(r):
        c, n, _ = r
        return c["nx"] * c["ny"] * 3 * n

    def servers():
        return {"air5": A.Server(precision=precision, max_members=64),
                "air11": A.Server(precision=precision, max_members=64, path=A.TABLE_AIR11)}

    # capacity: a closed loop that keeps `inflight` requests on the GPU (the concurrency the
    # arrival process sustains), not a burst, whose batches would be larger than any the arrivals
    # ever form
    calib = I.serving_requests(24, seed=seed + 1, steps=(20, 80), air11=air11)
    sv = servers()
    t0 = time.perf_counter()
    todo, pending = list(calib), []
    while todo or pending:
        while todo and len(pending) < inflight:
            c, n, _ = todo.pop(0)
            pending.append((sv[c["table"]], sv[c["table"]].submit(c, n)))
        time.sleep(0.002)
        pending = [(x, i) for x, i in pending if not x.stats(i)["done"]]
        if time.perf_counter() - t0 > 900:
            raise RuntimeError("serving calibration did not finish in 900 s")
    cap = sum(work(r) for r in calib) / (time.perf_counter() - t0)      # points*RHS per second
    for x in sv.values():
        x.close()
    reqs = I.serving_requests(nreq, seed=seed, steps=steps, air11=air11)
    mean_work = sum(work(r) for r in reqs) / len(reqs)
    lam = 0.8 * cap / mean_work                                            # requests per second
    sv = servers()
    ids = []
    t_start = time.perf_counter()
    t_next = t_start
    for c, n, gap in reqs:
        t_next += gap / lam
        delay = t_next - time.perf_counter()
        if delay > 0:
            time.sleep(delay)
        ids.append((c["table"], sv[c["table"]].submit(c, n)))
    for x in sv.values():
        x.wait(timeout=1800)
    st = [sv[t].stats(i) for t, i in ids]
    per = {}
    for t, x in sv.items():
        cnt = x.counters()
        mine = [r for r in reqs if r[0]["table"] == t]
        per[t] = {"requests": len(mine),
                  "busy_throughput_mpts_rhs_s": sum(work(r) for r in mine) / max(cnt["busy_s"], 1e-30) / 1e6,
                  "mean_batch": cnt["member_steps"] / max(cnt["batch_steps"], 1),
                  "max_batch": cnt["max_members"]}
        x.close()
    tts = np.array([s["t_finish"] - s["t_submit"] for s in st])
    wait = np.array([s["t_admit"] - s["t_submit"] for s in st])
    span = max(s["t_finish"] for s in st) - min(s["t_submit"] for s in st)
    total = sum(work(r) for r in reqs)
    return {"requests": nreq, "precision": "mixed" if precision else "fp64",
            "arrivals": f"Poisson at 0.8 x capacity (closed loop, {inflight} requests in flight)",
            "capacity_mpts_rhs_s": cap / 1e6, "rate_req_s": lam,
            "tts_p50_s": float(np.percentile(tts, 50)), "tts_p99_s": float(np.percentile(tts, 99)),
            "queue_wait_p50_s": float(np.percentile(wait, 50)),
            "throughput_mpts_rhs_s": total / span / 1e6,
            "servers": per,
            "errors": int(sum(1 for s in st if s["error"])),
            "status_nonzero": int(sum(1 for s in st if s["status"])),
            "status_requests": [{"name": c["name"], "nx": c["nx"], "ny": c["ny"],
                                 "mach": round(c["mach"], 3), "T_wall": round(c.get("T_wall", 0.0), 1),
                                 "steps": n, "status": s["status"]}
                                for (c, n, _), s in zip(reqs, st) if s["status"]],
            "workload": f"the first {nreq} requests of the serving stream: grids 128x32 to "
                        f"1024x256, boundary layers Mach 5-20 (wall 300-1500 K) and shock "
                        f"interactions, {steps[0]}-{steps[1]} RK3 steps each, {air11:.0%} on "
                        f"eleven-species air"}


def serving_plain_fp64(A, I, nreq, seed, air11=0.25, steps=(500, 2000)):
    """The same requests as serving_bench, stepped one at a time through the plain FP64 path
    (hyp_state_init, then hyp_rk_stage per stage on the request's own grid), back to back: the
    throughput the serving path is compared against."""
    import torch
    reqs = I.serving_requests(nreq, seed=seed, steps=steps, air11=air11)
    work = 0
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for c, n, _ in reqs:
        gas = A.gas_model_load(c)
        m = A.state_size(gas, c)
        U = torch.empty(m, dtype=torch.float64, device="cuda")
        dQ = torch.empty_like(U)
        st = A.state_init(gas, c, U, dQ, I.state_noise(m, c["seed"]))
        for _ in range(n):
            for k in range(STAGES):
                A.rk_stage(st, k, c["dt"])
        work += c["nx"] * c["ny"] * STAGES * n
        del st, U, dQ
    torch.cuda.synchronize()
    wall = time.perf_counter() - t0
    return {"requests": nreq, "precision": "fp64", "value": work / wall / 1e6,
            "unit": UNIT, "wall_s": wall,
            "note": "the serving requests stepped one at a time through hyp_rk_stage (FP64), "
                    "set-up included, no batching"}


def jet3d_bench(A, I, dev, rank, world, barrier, flush, steps=2, warmup=1, size=(512, 256, 128)):
    """Sonic jet through a circular orifice into the Mach 8 crossflow, 512 x 256 x 128 cells,
    spanwise periodic: RK3 steps timed with CUDA events (L2 flushed between steps), FP64, with
    binary32 transport, and FP64 replayed from one step captured into a CUDA graph."""
    import torch
    nx, ny, nz = size
    cfg = I.jet_case(nx, ny, nz, seed=7 + rank)
    gas = A.gas_model_load(cfg)
    n = A.state_size(gas, cfg)
    out = {"workload": f"jet_{nx}x{ny}x{nz}_cneq5_rk3", "cells": nx * ny * nz,
           "jet_J": cfg["jet_J"], "unit": UNIT}
    for prec, key in ((A.FP64, "fp64"), (A.MIXED, "mixed"), (A.FP64, "fp64_graph")):
        U = torch.empty(n, dtype=torch.float64, device=dev)
        dQ = torch.empty_like(U)
        st = A.state_init(gas, cfg, U, dQ, I.state_noise(n, cfg["seed"]))
        for _ in range(warmup):
            for k in range(STAGES):
                A.rk_stage(st, k, cfg["dt"], precision=prec)

        def step():
            for k in range(STAGES):
                A.rk_stage(st, k, cfg["dt"], precision=prec)

        graph = None
        if key == "fp64":
            A.grid_profile(st.grid, True)
        if key == "fp64_graph":
            torch.cuda.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                step()
            step = graph.replay
        ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
              for _ in range(steps)]
        barrier()
        for i in range(steps):
            ev[i][0].record()
            step()
            ev[i][1].record()
            flush.fill_(float(i))
        barrier()
        ms = max_over_ranks(sum(a.elapsed_time(b) for a, b in ev), world, dev)
        out[key] = {"value": job_rate(world, out["cells"], steps, ms), "ms_per_step": ms / steps,
                    "status_flags": A.grid_status(st.grid),
                    "finite": bool(torch.isfinite(st.U).all().item())}
        if key == "fp64":
            A.grid_profile(st.grid, False)
            cms, ccount = A.grid_profile_read(st.grid).get("k_closure", (0.0, 0))
            if ccount:
                avg_s = cms / ccount / 1e3
                roof = {"kernel": "k_closure3", "launches": ccount, "avg_launch_ms": avg_s * 1e3,
                        "share_of_step": cms / max(sum(a.elapsed_time(b) for a, b in ev), 1e-30),
                        **issue_roofline(CLOSURE3_INSTR, out["cells"] / avg_s)}
                out["roofline"] = roof
        del step, graph, st, U, dQ
        torch.cuda.empty_cache()
    return out


def ours_arm(args, rank, world, local_rank):
    import torch
    import torch.distributed as dist
    from paper_2210_05547_gb300 import abi as A
    from paper_2210_05547_gb300 import inputs as I

    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    if world > 1:
        dist.init_process_group("nccl", device_id=dev)

    def barrier():
        if world > 1:
            dist.barrier()
        torch.cuda.synchronize()

    cfg = I.sbli_case(args.nx, args.ny, seed=rank)
    gas = A.gas_model_load(cfg)
    n = A.state_size(gas, cfg)
    U = torch.empty(n, dtype=torch.float64, device=dev)
    dQ = torch.empty_like(U)
    st = A.state_init(gas, cfg, U, dQ, I.state_noise(n, cfg["seed"]))
    flush = torch.empty(L2_FLUSH_BYTES // 4, dtype=torch.float32, device=dev)
    dt = cfg["dt"]
    points = cfg["nx"] * cfg["ny"]

    def step():
        for k in range(STAGES):
            A.rk_stage(st, k, dt)

    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize()

    # ---------------- device-timed region ----------------
    clocks = ClockSampler(local_rank)
    clocks.start()
    time.sleep(0.3)
    A.grid_profile(st.grid, True)
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
          for _ in range(args.steps)]
    barrier()
    t_wall = time.perf_counter()
    for i in range(args.steps):
        ev[i][0].record()
        step()
        ev[i][1].record()
        flush.fill_(float(i))
    barrier()
    t_wall = time.perf_counter() - t_wall
    A.grid_profile(st.grid, False)
    prof = A.grid_profile_read(st.grid)
    clk = clocks.stop()
    dev_ms = sum(a.elapsed_time(b) for a, b in ev)
    max_ms = max_over_ranks(dev_ms, world, dev)
    value = job_rate(world, points, args.steps, max_ms)
    launches = sum(c for _, c in prof.values())
    status = A.grid_status(st.grid)

    # ---------------- the mixed-precision path on the same state ----------------
    mixed = None
    if not args.no_mixed:
        def step_mixed():
            for k in range(STAGES):
                A.rk_stage(st, k, dt, precision=A.MIXED)
        for _ in range(args.warmup):
            step_mixed()
        A.grid_profile(st.grid, True)
        em = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
              for _ in range(args.steps)]
        barrier()
        for i in range(args.steps):
            em[i][0].record()
            step_mixed()
            em[i][1].record()
            flush.fill_(float(i))
        barrier()
        A.grid_profile(st.grid, False)
        mprof = A.grid_profile_read(st.grid)
        m_ms = max_over_ranks(sum(a.elapsed_time(b) for a, b in em), world, dev)
        # error of one mixed right-hand side against the FP64 path at the current state
        R64 = torch.empty_like(U)
        R32 = torch.empty_like(U)
        A.rhs(gas, st.grid, U, R64)
        A.rhs(gas, st.grid, U, R32, precision=A.MIXED)
        torch.cuda.synchronize()
        errs = {}
        for name, (a0, a1) in field_ranges(cfg).items():
            ref = R64[a0:a1]
            errs[name] = float((R32[a0:a1] - ref).abs().max() / ref.abs().max().clamp_min(1e-300))
        del R64, R32
        mixed = {"value": job_rate(world, points, args.steps, m_ms),
                 "unit": UNIT, "ms_per_step": m_ms / args.steps,
                 "dtype": "f64 with f32 transport, diffusion and forward-rate exponentials",
                 "rhs_err_vs_fp64_path": errs, "max_rhs_err": max(errs.values()),
                 "err_bound": "1e-6 of max|R| per field against the FP64 oracle "
                              "(tests/test_gpu_mixed.py); wall heat flux and skin friction "
                              "within 1e-4 after 1000 steps",
                 "kernels": {k: {"ms": v[0], "launches": v[1]} for k, v in mprof.items() if v[1]}}

    # ---------------- end to end through the public API, host buffers ----------------
    e2e = None
    if not args.no_e2e:
        Uh = torch.empty(n, dtype=torch.float64, pin_memory=True)
        Uh.copy_(U)
        torch.cuda.synchronize()
        ee = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
              for _ in range(args.steps)]
        barrier()
        for i in range(args.steps):
            ee[i][0].record()
            U.copy_(Uh, non_blocking=True)
            step()
            Uh.copy_(U, non_blocking=True)
            ee[i][1].record()
            flush.fill_(float(i))
        barrier()
        e_ms = max_over_ranks(sum(a.elapsed_time(b) for a, b in ee), world, dev)
        e2e = {"value": job_rate(world, points, args.steps, e_ms),
               "unit": UNIT, "h2d_bytes_per_step": n * 8, "d2h_bytes_per_step": n * 8}

    # ---------------- roofline of the dominant kernel ----------------
    # k_closure is the largest launch of the serialised launch list (the nine line phases together
    # take a little more). The event time of a second-stream line phase that runs beside it includes
    # the time it waits for issue slots, so the ranking is not taken from the live totals.
    name = "k_closure" if "k_closure" in prof else max(prof.items(), key=lambda kv: kv[1][0])[0]
    kms, kcount = prof[name]
    avg_s = kms / max(kcount, 1) / 1e3
    roof = {"kernel": name, "launches": kcount, "avg_launch_ms": avg_s * 1e3,
            "share_of_step": kms / max(dev_ms, 1e-30)}
    if name == "k_closure":
        roof.update(issue_roofline(CLOSURE_INSTR, points / avg_s),
                    traffic=CLOSURE_DRAM_BYTES_PER_POINT * points)
    else:
        roof.update(bound="alu", achieved=None, peak=ISSUE_PEAK_TINSTR,
                    unit="T thread instructions/s", frac=None, traffic=None,
                    note="per-point instruction count not measured for this kernel")

    # ---------------- model variants on the same workload (FP64, same steps) ----------------
    def variant(cfg_v):
        gas_v = A.gas_model_load(cfg_v)
        n_v = A.state_size(gas_v, cfg_v)
        Uv = torch.empty(n_v, dtype=torch.float64, device=dev)
        dQv = torch.empty_like(Uv)
        stv = A.state_init(gas_v, cfg_v, Uv, dQv, I.state_noise(n_v, cfg["seed"]))
        for _ in range(args.warmup):
            for k in range(STAGES):
                A.rk_stage(stv, k, dt)
        es = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
              for _ in range(args.steps)]
        barrier()
        for i in range(args.steps):
            es[i][0].record()
            for k in range(STAGES):
                A.rk_stage(stv, k, dt)
            es[i][1].record()
            flush.fill_(float(i))
        barrier()
        v_ms = max_over_ranks(sum(a.elapsed_time(b) for a, b in es), world, dev)
        out = {"value": job_rate(world, points, args.steps, v_ms), "unit": UNIT,
               "ms_per_step": v_ms / args.steps, "status_flags": A.grid_status(stv.grid)}
        del stv, Uv, dQv
        return out, v_ms

    smd = None
    if not args.no_sm:
        smd, s_ms = variant(dict(cfg, diffusion_model="stefan_maxwell"))
        smd.update(cost_vs_algebraic=s_ms / max_ms,
                   note="Stefan-Maxwell system (Eq. 17) solved at every face instead of the "
                        "algebraic model (Eq. 18); same case, FP64")
    jet3d = None
    if not args.no_3d:
        jet3d = jet3d_bench(A, I, dev, rank, world, barrier, flush,
                            size=tuple(int(v) for v in args.jet3d_size.split("x")))
    air11 = None
    if not args.no_air11:
        air11, a_ms = variant(I.with_species(cfg))
        air11.update(cost_vs_air5=a_ms / max_ms,
                     note="eleven-species air (N2, O2, NO, N, O, N2+, O2+, NO+, N+, O+, e-; 49 "
                          "reactions; ambipolar ions, zero-current electrons) on the same case "
                          "from the same neutral initial state, FP64")
    lte = None
    if not args.no_lte:
        lte, l_ms = variant(dict(cfg, kind="lte"))
        lte.update(cost_vs_cneq=l_ms / max_ms,
                   note="local thermodynamic equilibrium (Sec. 2.2.2): Gibbs-minimum composition "
                        "and equilibrium conductivity per point, no species equations; same "
                        "case, FP64")

    serving = serving_fp64 = serving_plain = None
    if args.serve_requests > 0:
        serving = serving_bench(A, I, args.serve_requests, 100 + rank, A.MIXED)
        serving_plain = serving_plain_fp64(A, I, args.serve_requests, 100 + rank)
        serving["vs_plain_fp64_one_at_a_time"] = (serving["throughput_mpts_rhs_s"]
                                                  / serving_plain["value"])
        if args.serve_fp64:
            serving_fp64 = serving_bench(A, I, args.serve_requests, 100 + rank, A.FP64)

    sweep = None
    if args.thermo_states > 0:
        del flush
        torch.cuda.empty_cache()
        sweep = thermo_sweep(A, gas, dev, int(args.thermo_states), 1000 + rank)
        sweep["mixed"] = thermo_sweep(A, gas, dev, int(args.thermo_states), 1000 + rank,
                                      precision=A.MIXED)
        if not args.no_air11:
            gas11 = A.gas_model_load(I.with_species(cfg))
            sweep["air11"] = thermo_sweep(A, gas11, dev, int(args.thermo_states), 2000 + rank)
            sweep["air11"]["mixed"] = thermo_sweep(A, gas11, dev, int(args.thermo_states),
                                                   2000 + rank, precision=A.MIXED)

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu:
        r, cores, w = oracle_step_rate(CPU_NX, CPU_NY, steps=4, warm=1)
        cpu = {"value": r, "unit": UNIT, "cores": cores, "kind": "oracle",
               "sample": f"four oracle RK3 steps (12 RHS) of the same case at {CPU_NX}x{CPU_NY} "
                         f"cells after one untimed step, {w:.1f} s"}
        every = oracle_all_cores(CPU_NX, CPU_NY)
        if "value" in every:
            cpu["all_cores"] = {"value": every["value"], "unit": UNIT, "cores": every["cores"],
                                "kind": "oracle",
                                "sample": f"one warmed step of the same sample in each of "
                                          f"{every['cores']} single-threaded processes at once "
                                          f"(slowest {every['slowest_s']:.1f} s)"}
        else:
            cpu["all_cores"] = every

    if rank == 0:
        line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
                "steps": args.steps, "warmup": args.warmup, "ms_per_step": max_ms / args.steps,
                "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
                "data": "synthetic", "config": workload_config(cfg, world), "e2e": e2e,
                "gpu_launches": launches, "roofline": roof, "cpu_baseline": cpu, "clocks": clk,
                "whole_rhs": issue_roofline(RHS_INSTR, value / world * 1e6),
                "wall_s_timed": t_wall, "status_flags": status, "mixed": mixed,
                "serving": serving, "serving_fp64": serving_fp64,
                "serving_plain_fp64": serving_plain, "stefan_maxwell": smd,
                "lte": lte, "air11": air11, "jet3d": jet3d, "thermo_sweep": sweep,
                "kernels": {k: {"ms": v[0], "launches": v[1]} for k, v in prof.items() if v[1]},
                "kernels_note": "live CUDA-event time of each kernel summed over the timed steps; "
                                "the phases on the second stream overlap the closure, so the sum "
                                "exceeds the step time and is not a serial breakdown (the "
                                "serialised shares are in the ncu launch list)"}
        print(json.dumps(line), flush=True)
    if world > 1:
        dist.destroy_process_group()
    return 0


def main():
    args = parse()
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))
    if world != args.gpus and "RANK" in os.environ:
        world = int(os.environ["WORLD_SIZE"])
    if args.impl == "reference":
        return reference_arm(args, rank, world)
    return ours_arm(args, rank, world, local_rank)


if __name__ == "__main__":
    sys.exit(main())
