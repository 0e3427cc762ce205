"""Benchmark: batched N-1 contingency power flows (DPF, Alg. 1) on one GB300.

Workload (default line): the N-1 contingency batch -- a 2,000-bus synthetic
grid (2,700 branches), one case per single-branch outage that does not island
the grid (2,379 cases), all sharing one Y_bus with a per-case branch-removal
correction.

A step is one whole batched solve, inputs resident on the GPU: the base case
(no outage) by the library's Newton-Raphson, then every N-1 case by Alg. 1
started from the base case's solution (the warm start of Sec. 5.4.2) shifted
by the DC angle change of its outage (`--n1-start dc`, the default; `base`:
no shift), refined FP32 iterations (DPF_FP32R) with the FP64 convergence
test every 100 iterations on the cases whose FP32 mismatch is within 5e-6
p.u. and every 500 on every case (presets.N1_DC_TEST; unshifted: 50 and 100)
and per-case early stopping at 1e-6 p.u., up to `--n1-budget` iterations
(3,500 with the shift, settings presets.N1_DC; 4,000 without,
presets.N1_WARM).  `value` counts only the
cases the FP64 test declares converged (max |f| <= 1e-6 p.u.), per second;
the others are reported, not counted.  A solve takes ~0.5 s and moves ~0.5 GB
per iteration, far beyond the 129 MB L2 (no flush needed).

Sub-records on the same line: the flat-start FP32 iteration rate of the same
batch (Table 2, the kernels' own roofline; no case reaches 1e-6 from the flat
start within Table 2's budget), the 30-bus batch where every case converges
(`c1batch`), the 10,000-bus time series over a year of hourly snapshots
(`timeseries`), and the 64-grid uneven batch with parameter identification
(`uneven`).

--impl reference times the CPU FP64 oracle on the same warm-started N-1 solves
(a bounded sample of the cases per step, the same start) on the host cores.
"""
from __future__ import annotations

import argparse
import dataclasses
import hashlib
import json
import math
import os
import statistics
import subprocess
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
ITERS_PER_SOLVE = 1000  # Table 2: maximum iterations of one DPF solve from the flat start
from paper_2603_28203_gb300.presets import N1_BUDGET, N1_DC_BUDGET  # iterations of one N-1 solve  # noqa: E402
CHECK_EVERY = 25
TOL = 1e-6
LR = 1e-3               # flat-start FP32 iterations of the N-1 batch (Table 2 otherwise)
METRIC = "power-flow solves/s to 1e-6 p.u. mismatch; fwd+adjoint HBM GB/s vs peak"


def _workload():
    import gridgen
    g = gridgen.config_grid("c3_n1_2kbus")
    outages = gridgen.n1_outages(g)
    return g, outages


# ---------------------------------------------------------------------------
# CPU oracle legs (cpu_baseline and the reference arm)
# ---------------------------------------------------------------------------
_ORACLE_CACHE = {}


def _oracle_base():
    """The base case's solution by the oracle's Newton-Raphson (cached per process)."""
    import gridgen
    import oracle
    from oracle.ybus import grid_ybus
    if "base" not in _ORACLE_CACHE:
        g = gridgen.config_grid("c3_n1_2kbus")
        _ORACLE_CACHE["grid"] = g
        _ORACLE_CACHE["base"] = oracle.nr_solve(grid_ybus(g), g.p_spec, g.q_spec, g.bus_type, g.vm_set)
    return _ORACLE_CACHE["grid"], _ORACLE_CACHE["base"]


def n1_settings(start):
    """(optimiser settings, start and test options, default budget) of the
    N-1 solve: start "dc" = the base case's solution shifted by each outage's
    DC angle change, "base" = the base case's solution.  The test options
    hold the FP64 test interval (check_every) and the FP32 gate."""
    from paper_2603_28203_gb300 import presets
    if start == "dc":
        return presets.N1_DC, dict(presets.N1_DC_START, **presets.N1_DC_TEST), N1_DC_BUDGET
    if start == "base":
        return presets.N1_WARM, dict(presets.N1_TEST), N1_BUDGET
    raise ValueError(f"unknown N-1 start {start!r}")


def _oracle_dpf_options(budget, start):
    import oracle
    from paper_2603_28203_gb300 import _abi
    s, t, _ = n1_settings(start)
    sched = {_abi.SCHED_PLATEAU: "plateau", _abi.SCHED_STEP: "step", _abi.SCHED_CONST: "const"}[s["sched"]]
    return oracle.DPFOptions(lr=s["lr"], beta1=s["beta1"], beta2=s["beta2"], eps=s["eps"],
                             sched=sched, factor=s["factor"], patience=s["patience"],
                             threshold=s["threshold"], cooldown=s["cooldown"], max_iter=budget, tol=TOL,
                             check_every=t["check_every"])


def _oracle_case(args):
    """One warm-started N-1 case through the oracle: the DC outage shift of
    the base case's angles (start "dc"; a sparse direct solve), then the
    Alg. 1 loop: (iterations, seconds, status)."""
    import oracle
    from oracle.ybus import grid_ybus
    ell, budget, start = args
    g, base = _oracle_base()
    Y = grid_ybus(g.without_branch(int(ell)))
    t0 = time.perf_counter()
    va0 = base["va"]
    if start == "dc":
        va0 = va0 + oracle.dc_outage_shift(g.n_bus, g.f_bus, g.t_bus, g.x, g.tap, g.bus_type, va0, int(ell))
    r = oracle.dpf_solve(Y, g.p_spec, g.q_spec, g.bus_type, g.vm_set, _oracle_dpf_options(budget, start),
                         va0=va0, vm0=base["vm"], va_slack=g.va_slack)
    return r["iters"], time.perf_counter() - t0, r["status"]


def _oracle_cases(args):
    """Several cases in one process: (case-iterations, seconds, converged)."""
    cases, budget, start = args
    n, t, c = 0, 0.0, 0
    for ell in cases:
        it, dt, st = _oracle_case((ell, budget, start))
        n, t, c = n + it, t + dt, c + int(st == 0)
    return n, t, c


def _oracle_pool_run(chunks, budget, start):
    """Run `chunks` (one list of cases per host core) through a spawn pool;
    the time is the slowest core's."""
    import multiprocessing as mp
    cores = len(chunks)
    with mp.get_context("spawn").Pool(cores) as pool:
        pool.map(_oracle_base_init, range(cores))  # start-up and the base case, untimed
        res = pool.map(_oracle_cases, [(c, budget, start) for c in chunks])
    return sum(r[0] for r in res), max(r[1] for r in res), sum(r[2] for r in res)


def _oracle_base_init(_):
    _oracle_base()
    return 0


def cpu_oracle_sample(outages, budget, rounds, start):
    """The oracle on `rounds` warm-started N-1 cases per host core (seeded
    sample without replacement); solves/s counts the converged ones."""
    cores = len(os.sched_getaffinity(0))
    rng = np.random.default_rng(7)
    pick = [int(c) for c in rng.choice(outages, size=min(outages.size, cores * rounds), replace=False)]
    chunks = [pick[i::cores] for i in range(cores)]
    n_it, t, conv = _oracle_pool_run(chunks, budget, start)
    shift = "the DC outage shift of the base case, then " if start == "dc" else ""
    return dict(value=conv / t, unit="solves/s", cores=cores, kind="oracle",
                sample=f"{len(pick)} warm-started N-1 cases ({rounds} per core), each through the FP64 "
                       f"numpy/scipy oracle ({shift}Alg. 1 loop to 1e-6 p.u. or {budget} iterations); "
                       f"{conv} converged; {n_it} case-iterations in {t:.1f} s (slowest core)",
                converged=conv, cases=len(pick), case_iterations_per_s=n_it / t)


# ---------------------------------------------------------------------------
# clocks
# ---------------------------------------------------------------------------
class ClockSampler:
    QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_id, path):
        self.path = path
        self.proc = None
        try:
            self.f = open(path, "w")
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(gpu_id), f"--query-gpu={self.QUERY}", "--format=csv,noheader,nounits",
                 "-lms", "200"], stdout=self.f, stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None

    @staticmethod
    def gpu_id(local):
        """nvidia-smi id of torch device `local` (UUID when torch exposes it)."""
        import torch
        try:
            u = str(torch.cuda.get_device_properties(local).uuid)
            return u if u.startswith("GPU-") else "GPU-" + u
        except Exception:
            vis = os.environ.get("CUDA_VISIBLE_DEVICES")
            return vis.split(",")[local] if vis else str(local)

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(5)
        except Exception:
            self.proc.kill()
        self.f.close()
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                mx.append(float(parts[2]))
            except ValueError:
                continue
            for n, v in zip(names, parts[5:9]):
                if v.lower() == "active":
                    reasons.add(n)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
                "samples": len(sm)}


# ---------------------------------------------------------------------------
# roofline helpers
# ---------------------------------------------------------------------------
def algorithmic_bytes(n_bus, n_pv, n_pq, nnz, n_case, spec_per_case=False, refined=False):
    """Bytes each kernel must move per launch (every array element once).

    k_fwd, per case: read V (8 B/bus), write w (8 B/bus), write Q_calc at pv
      buses (4 B); refined FP32 (DPF_FP32R): the gathered operand is dV (8),
      and the epilogue reads V_ref (8) and (I_ref, f_ref) (16) instead of the
      specified injections;
    k_adj, per case: read w (8 B/bus); at pv buses read Q_calc (4); at every
      pv/pq bus read+write theta (16, double-float), read |V| (8), read+write
      V (16), read+write the two Adam moments of theta (16); at pq buses also
      write |V| (8) and read+write its moments (16); refined: the same (dV
      takes V's place; V is rebuilt from the master).
    Shared per launch: Y in CSR (16 B per nonzero + 4 B row pointers + bus
    types) and the shared specified P, Q (8 B/bus) -- or, with a specification
    per case, P and Q per element (8 B, FP32) read by both passes.
    """
    shared = 16 * nnz + 4 * (n_bus + 1) + n_bus
    spec_f = n_case * 8 * n_bus if spec_per_case else 8 * n_bus
    spec_a = n_case * 8 * (n_pv + n_pq) if spec_per_case else 8 * n_bus
    if refined:
        fwd = n_case * (40 * n_bus + 4 * n_pv) + shared
        adj = n_case * (8 * n_bus + 60 * n_pv + 80 * n_pq) + shared + spec_a
    else:
        fwd = n_case * (16 * n_bus + 4 * n_pv) + shared + spec_f
        adj = n_case * (8 * n_bus + 60 * n_pv + 80 * n_pq) + shared + spec_a
    return fwd, adj


def iteration_flops(n_bus, nnz, n_case):
    """FP32 operations of one iteration: the two complex products with Y (8 per
    nonzero each), 30 per bus for S, the mismatch, c and w, 60 for the gradient,
    the optimiser step and the new V."""
    return n_case * (16 * nnz + 90 * n_bus)


def timed_kernel(n_bus, nnz, n_case, us, sms, sm_max_mhz):
    """The on-chip iterations as the timed step runs them (its FP64 tests and
    starts counted in), against the nominal FP32 rate."""
    peak = sms * 128 * 2 * sm_max_mhz * 1e6 / 1e12
    tf = iteration_flops(n_bus, nnz, n_case) / (us * 1e-6) / 1e12
    return {"kernel": "k_resident_cta<float, refined, Adam>", "bound": "instruction issue", "us_per_iteration": us,
            "achieved": tf, "peak": peak, "unit": "TFLOP/s", "frac": tf / peak,
            "peak_source": f"nominal: {sms} SMs x 128 FMA x {sm_max_mhz:.0f} MHz"}


def _peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        d = json.load(open(p))
        return float(d["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


def _kernel_hash():
    """Hash of the source of the iteration kernels (forward and adjoint
    passes); a committed ncu traffic figure counts only while it matches."""
    h = hashlib.sha256()
    h.update(open(os.path.join(ROOT, "paper_2603_28203_gb300", "csrc", "dpf_kernels.cuh"), "rb").read())
    return h.hexdigest()[:16]


def _ncu_traffic(name):
    """DRAM bytes per launch from a committed ncu summary, if it is current
    (its recorded source hash equals the kernels')."""
    p = os.path.join(ROOT, "profiles", f"{name}.md")
    if not os.path.exists(p):
        return None
    h, b = None, None
    for line in open(p).read().splitlines():
        if line.startswith("source_hash:"):
            h = line.split(":", 1)[1].strip()
        if line.startswith("dram_bytes_per_launch:"):
            b = float(line.split(":", 1)[1].strip())
    return b if (h == _kernel_hash() and b is not None) else None


def _l2_read_peak(dpf, torch, stream):
    """Read bandwidth of the library's plain probe kernel (dpf_read_bandwidth):
    a 32 MB buffer (far below the 129 MB L2, so L2-resident after the probe's
    untimed launches) and a 4 GB one (HBM), best of 10 measurements of 20
    launches each, CUDA events on `stream`."""
    dev = torch.device("cuda", torch.cuda.current_device())
    out = {}
    for name, nbytes in (("l2", 32 << 20), ("hbm", 4 << 30)):
        x = torch.ones(nbytes // 4, dtype=torch.float32, device=dev)
        out[name] = max(dpf.dpf_read_bandwidth(x, reps=20, stream=stream) for _ in range(10))
        del x
    return {"gbs": out["l2"], "hbm_read_gbs": out["hbm"],
            "how": "dpf_read_bandwidth: 16-byte ld.global.cg reads, SMs x 8 CTAs, best of 10 x 20 launches; "
                   "32 MB buffer (L2-resident) and 4 GB buffer (HBM read)"}


# ---------------------------------------------------------------------------
# GPU arm
# ---------------------------------------------------------------------------
def _outputs(torch, K, N, dev, pinned=False):
    def mk(shape, dt):
        t = torch.empty(shape, dtype=dt, device="cpu" if pinned else dev)
        return t.pin_memory() if pinned else t
    return dict(va=mk((K, N), torch.float64), vm=mk((K, N), torch.float64), iters=mk(K, torch.int32),
                status=mk(K, torch.int32), max_mismatch=mk(K, torch.float64), loss=mk(K, torch.float64))


class N1Job:
    """One step of the benchmark: the base case by Newton-Raphson, then every
    N-1 case warm-started from it (shifted by its outage's DC angle change
    for start "dc"; refined FP32 DPF iterations)."""

    def __init__(self, dpf, torch, g, outages, stream, budget, args):
        settings, start_opts, _ = n1_settings(args.n1_start)
        self.dpf, self.torch, self.g, self.stream = dpf, torch, g, stream
        dev = torch.device("cuda", torch.cuda.current_device())
        self.K, self.N = outages.size, g.n_bus
        self.y = dpf.dpf_build_ybus(g, stream=stream)
        self.nr = dpf.dpf_nr_create(self.y, 1)
        self.ws = dpf.dpf_workspace_create(self.y, self.K)
        self.outage = torch.tensor(outages, dtype=torch.int32, device=dev)
        self.base = dict(va=torch.zeros((1, self.N), dtype=torch.float64, device=dev),
                         vm=torch.zeros((1, self.N), dtype=torch.float64, device=dev),
                         status=torch.zeros(1, dtype=torch.int32, device=dev))
        self.res = _outputs(torch, self.K, self.N, dev)
        self.opts = dpf.SolveOpts(precision=dpf.FP32R, tol=TOL, max_iter=budget, flat_start=0,
                                  lanes=args.lanes or None, warps=args.warps or None,
                                  row_blocks=args.row_blocks or None, pdl=0 if args.no_pdl else None, **settings,
                                  **start_opts)
        self.shape_by = "command line" if (args.lanes or args.warps or args.row_blocks) else \
            "library default" if args.no_autotune else "dpf_autotune"

    def base_case(self):
        d = self.dpf
        d.dpf_nr_solve(self.nr, precision=d.FP64, tol=1e-10, max_iter=20, n_case=1, va=self.base["va"],
                       vm=self.base["vm"], status=self.base["status"], stream=self.stream)

    def autotune(self):
        d = self.dpf
        self.base_case()
        with self.torch.cuda.stream(self.stream):
            self.opts = d.dpf_autotune(self.y, self.ws, self.opts, iters=50, stream=self.stream, n_case=self.K,
                                       outage=self.outage, va_start=self.base["va"][0], vm_start=self.base["vm"][0])

    def step(self):
        d = self.dpf
        self.base_case()
        d.dpf_solve_batch(self.y, self.ws, self.opts, stream=self.stream, n_case=self.K, outage=self.outage,
                          va_start=self.base["va"][0], vm_start=self.base["vm"][0], **self.res)

    def launches(self):
        return self.dpf.dpf_kernel_launches(self.ws) + self.nr.stats()["launches"]

    def kernel_times(self, n_iter):
        """Event-bracketed forward / adjoint launches of n_iter iterations of the
        same warm-started solve (all cases active), on the same stream."""
        d = self.dpf
        with self.torch.cuda.stream(self.stream):
            d.dpf_solve_begin(self.y, self.ws, self.opts, stream=self.stream, n_case=self.K, outage=self.outage,
                              va_start=self.base["va"][0], vm_start=self.base["vm"][0])
            d.dpf_solve_iterate(self.ws, self.opts.check_every, stream=self.stream)
            d.dpf_profile_enable(self.ws, True)
            d.dpf_solve_iterate(self.ws, n_iter, stream=self.stream)
            t = d.dpf_kernel_times(self.ws, stream=self.stream)
            d.dpf_profile_enable(self.ws, False)
            d.dpf_solve_end(self.ws, stream=self.stream, n_case=self.K)
            self.stream.synchronize()
        return t


def run_ours(args):
    import torch
    import torch.distributed as dist

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    # host-core baseline before the first CUDA call (spawned pool)
    g, outages = _workload()
    cpu = None
    if rank == 0 and not args.no_cpu_baseline:
        cpu = cpu_oracle_sample(outages, args.n1_budget, args.cpu_rounds, args.n1_start)

    torch.cuda.set_device(local)
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    from paper_2603_28203_gb300.build import LIB, build
    if not os.path.exists(LIB):
        build()
    import paper_2603_28203_gb300 as dpf
    from paper_2603_28203_gb300.shard import reduce_max, reduce_sum

    dev = torch.device("cuda", local)
    stream = torch.cuda.Stream(dev)
    job = N1Job(dpf, torch, g, outages, stream, args.n1_budget, args)
    K, N = job.K, job.N
    if job.shape_by == "dpf_autotune":
        job.autotune()
    with torch.cuda.stream(stream):
        for _ in range(args.warmup):
            job.step()
        stream.synchronize()
        clocks_dir = os.environ.get("DPF_CLOCKS_DIR") or tempfile.gettempdir()
        clocks = ClockSampler(ClockSampler.gpu_id(local), os.path.join(clocks_dir, f"clocks_rank{rank}.csv"))
        time.sleep(0.3)
        if world > 1:
            dist.barrier()
        torch.cuda.synchronize()
        launches0 = job.launches()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(args.steps):
            job.step()
        e1.record(stream)
        torch.cuda.synchronize()
        if world > 1:
            dist.barrier()
        t_ms = e0.elapsed_time(e1)
        launches = job.launches() - launches0
        clk = clocks.stop()
        t_done = dpf.dpf_iterations_done(job.ws)
    st = job.res["status"].cpu().numpy()
    it = job.res["iters"].cpu().numpy()
    mm = job.res["max_mismatch"].cpu().numpy()
    conv = int((st == dpf.CASE_CONVERGED).sum())
    t_max = reduce_max(t_ms, dist if world > 1 else None)
    conv_all = reduce_sum(float(conv * args.steps), dist if world > 1 else None)
    case_iters = reduce_sum(float(it.sum()) * args.steps, dist if world > 1 else None)
    value = conv_all / (t_max / 1e3)

    # per-kernel durations (same workload, same stream, event-bracketed launches)
    fwd_ms, adj_ms, n_fwd, n_adj = job.kernel_times(args.profile_steps)
    n_pv = int((g.bus_type == 1).sum())
    n_pq = int((g.bus_type == 0).sum())
    fwd_b, adj_b = algorithmic_bytes(N, n_pv, n_pq, job.y.nnz, K, refined=True)
    peak, peak_kind = _peaks()
    adj_avg, fwd_avg = adj_ms / max(n_adj, 1), fwd_ms / max(n_fwd, 1)
    achieved = adj_b / (adj_avg / 1e3) / 1e9
    fwd_gbs = fwd_b / (fwd_avg / 1e3) / 1e9
    l2 = _l2_read_peak(dpf, torch, stream)
    fwd_name = "k_fwd2<true>" if (job.opts.pair_cases or 0) & 1 else "k_fwd<float,true>"
    adj_name = "k_adj2<true>" if (job.opts.pair_cases or 0) & 2 else "k_adj<float,false,true>"

    e2e = None if args.no_e2e else run_e2e(dpf, torch, job, args)
    plain = None if args.no_plain else run_plain(dpf, torch, job, st, it, args)
    subs = {}
    if not args.no_subrecords:
        subs["n1_flat_fp32"] = run_flat_fp32(dpf, torch, job, args, peak, l2)
        subs["c1batch"] = c1batch_record(dpf, torch, args.c1_cases, plain_cases=args.plain_cases)
        subs["timeseries"] = timeseries_record(dpf, torch, args.ts_hours, newton=True)
        subs["uneven"] = uneven_record(dpf, torch, args)

    if rank == 0:
        ce = job.opts.check_every
        line = {
            "metric": METRIC,
            "value": value,
            "unit": "solves/s",
            "n_gpus": world,
            "steps": args.steps,
            "warmup": args.warmup,
            "ms_per_step": t_max / args.steps,
            "higher_is_better": True,
            "scaling": "weak",
            "vs_baseline": None,
            "dtype": "f32 (refined: FP32 iterations on the FP64 residual of each test; FP64 convergence test)",
            "data": "synthetic (seeded generator; stands in for the paper's grids)",
            "config": {
                "workload": "N-1 contingency batch: 2,000-bus synthetic grid, 2,700 branches, "
                            f"{K} non-islanding single-branch outages per GPU, shared CSR Y_bus (nnz {job.y.nnz}) "
                            "+ per-case branch-removal correction; each case warm-started from the base case "
                            "(solved by Newton-Raphson in the same step)"
                            + (", shifted by the DC angle change of its outage (CG in the same step)"
                               if args.n1_start == "dc" else ""),
                "n1_start": args.n1_start,
                "n_bus": N, "n_branch": g.n_branch, "cases_per_gpu": int(K), "nnz": job.y.nnz,
                "iteration_precision": "fp32r", "check_every": ce, "gate_pu": job.opts.gate,
                "refresh_every": job.opts.refresh_every or 100, "tol_pu": TOL,
                "budget_iterations": args.n1_budget,
                "optimizer": "Adam + ReduceLROnPlateau, presets."
                             + ("N1_DC" if args.n1_start == "dc" else "N1_WARM")
                             + " (searched, Sec. 5.3's procedure)",
                "dc_shift": ({k: getattr(job.opts, k) for k in ("dc_tol", "dc_max_iter")}
                             if args.n1_start == "dc" else None),
                "solve_definition": f"Alg. 1 from the (shifted) base case's solution until FP64 max mismatch <= "
                                    f"{TOL} p.u. (counted) or {args.n1_budget} iterations (not counted)",
                "step": "one whole batched solve: base case (Newton-Raphson, FP64)"
                        + (" + the DC outage shift of every case (CG)" if args.n1_start == "dc" else "")
                        + " + all N-1 cases (DPF)",
                "l2": "per-iteration traffic ~0.6 GB >> 129 MB L2 (no flush needed)",
                "parallelism": f"replicas x{world} (independent cases, no data-path collective)",
                "launch_shape": {"lanes": job.opts.lanes, "warps": job.opts.warps, "row_blocks": job.opts.row_blocks,
                                 "pair_cases": job.opts.pair_cases, "stage_v": job.opts.stage_v,
                                 "chosen_by": job.shape_by},
            },
            "converged": conv,
            "converged_frac": conv / K,
            "not_converged": int(K - conv),
            "iterations_converged_p50": float(np.median(it[st == 0])) if conv else None,
            "mismatch_p50": float(np.median(mm)),
            "mismatch_max": float(np.max(mm)),
            "case_iterations_per_s": case_iters / (t_max / 1e3),
            "iterations_per_solve": int(t_done),
            "fp64_checks_in_timed_region": args.steps * (math.ceil(t_done / ce) + 1),
            "graph_replays_in_timed_region": args.steps * (t_done // ce),
            "roofline": {
                "kernel": f"{adj_name} (adjoint SpMV + gradient + Adam, refined FP32)",
                "bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
                "frac": achieved / peak, "peak_source": peak_kind,
                "traffic": _ncu_traffic("k_adj_fp32r_n1_2kbus"),
                "algorithmic_bytes_per_launch": adj_b, "avg_launch_ms": adj_avg,
                "fwd": {"kernel": fwd_name, "achieved": fwd_gbs, "frac": fwd_gbs / peak,
                        "algorithmic_bytes_per_launch": fwd_b, "avg_launch_ms": fwd_avg,
                        "traffic": _ncu_traffic("k_fwd_fp32r_n1_2kbus"),
                        "l2_peak_gbs": l2["gbs"], "frac_of_l2_peak": fwd_gbs / l2["gbs"]},
                "fwd_adj_combined_gbs": (fwd_b + adj_b) / ((fwd_avg + adj_avg) / 1e3) / 1e9,
                "fwd_adj_combined_frac": (fwd_b + adj_b) / ((fwd_avg + adj_avg) / 1e3) / 1e9 / peak,
                "timed_launches": n_adj,
                "l2_peak": l2,
                "note": "the two passes larger grids iterate with, timed apart; the timed solve keeps a case "
                        "of this size on chip (k_resident_cta) and is bound by instruction issue",
                "step_us_per_iteration": 1e3 * t_max / args.steps / t_done if t_done else None,
                "timed_kernel": timed_kernel(N, job.y.nnz, K, 1e3 * t_max / args.steps / t_done,
                                             torch.cuda.get_device_properties(dev).multi_processor_count,
                                             float(clk.get("sm_max_mhz") or 2070.0)) if t_done else None,
            },
            "gpu_launches": int(launches),
            "clocks": clk,
            "e2e": e2e,
            "plain_form": plain,
            "speedup_vs_plain_form": (value / plain["value"]) if plain and plain["value"] else None,
            "cpu_baseline": cpu,
            **subs,
        }
        print(json.dumps(line))
    if world > 1:
        dist.barrier()
        dist.destroy_process_group()


def run_e2e(dpf, torch, job, args):
    """The same step through the public API with host buffers: the base case
    by Newton-Raphson (device), its state read to pinned host memory, then
    dpf_solve_batch with host_io (the outage list and the shared start go in,
    every case's solution, iterations, status and mismatch come out)."""
    K, N = job.K, job.N
    h_out = torch.tensor(job.outage.cpu().numpy(), dtype=torch.int32).pin_memory()
    h = _outputs(torch, K, N, None, pinned=True)
    hb = {k: torch.empty(N, dtype=torch.float64).pin_memory() for k in ("va", "vm")}
    times, conv = [], 0
    for rep in range(1 + args.e2e_steps):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        job.base_case()
        hb["va"].copy_(job.base["va"][0])
        hb["vm"].copy_(job.base["vm"][0])
        dpf.dpf_solve_batch(job.y, job.ws, job.opts, stream=job.stream, n_case=K, host_io=True, outage=h_out,
                            va_start=hb["va"], vm_start=hb["vm"], **h)
        torch.cuda.synchronize()
        if rep > 0:
            times.append(time.perf_counter() - t0)
            conv = int((h["status"].numpy() == dpf.CASE_CONVERGED).sum())
    t = sum(times) / len(times)
    h2d = K * 4 + 2 * N * 8
    d2h = 2 * N * 8 + 2 * K * N * 8 + 2 * K * 4 + 2 * K * 8
    return {"value": conv / t, "unit": "solves/s", "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h,
            "converged": conv, "step": "Newton-Raphson base case + one dpf_solve_batch call (host_io) over all "
            "cases, wall clock", "steps": len(times), "ms_per_step": 1e3 * t}


def run_plain(dpf, torch, job, st, it, args):
    """The plain form on the same GPU: Alg. 1 one case at a time in FP64,
    separate launches per iteration and a host stop test after each, from the
    same base-case start, same settings and budget.  A sample of cases (half
    of them ones the batch converged) gives the per-iteration time and checks
    the outcomes; its solves/s for the whole batch is the batch's converged
    count over the time the plain form needs for the batch's iterations."""
    dev = torch.device("cuda", torch.cuda.current_device())
    conv_idx = np.nonzero(st == 0)[0]
    other = np.nonzero(st != 0)[0]
    n = args.plain_cases
    pick = np.concatenate([conv_idx[: n // 2], other[: n - min(n // 2, conv_idx.size)]]).astype(np.int64)
    ws1 = dpf.dpf_workspace_create(job.y, 1)
    out = job.outage[torch.tensor(pick, device=dev)].contiguous()
    r = _outputs(torch, pick.size, job.N, dev)
    opts = dataclasses.replace(job.opts, precision=dpf.FP64, plain=1, lanes=None, warps=None, row_blocks=None,
                               pair_cases=None, stage_v=None)
    kw = dict(va_start=job.base["va"][0], vm_start=job.base["vm"][0])
    with torch.cuda.stream(job.stream):
        dpf.dpf_solve_batch(job.y, ws1, dataclasses.replace(opts, max_iter=50), stream=job.stream, n_case=1,
                            outage=out[:1], **kw, **{k: v[:1] for k, v in r.items()})  # warm-up
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        dpf.dpf_solve_batch(job.y, ws1, opts, stream=job.stream, n_case=pick.size, outage=out, **kw, **r)
        torch.cuda.synchronize()
        t = time.perf_counter() - t0
    ws1.free()
    pst, pit = r["status"].cpu().numpy(), r["iters"].cpu().numpy()
    t_it = t / max(int(pit.sum()), 1)
    batch_conv = int((st == 0).sum())
    return {"value": batch_conv / (float(it.sum()) * t_it), "unit": "solves/s", "precision": "fp64",
            "sample_cases": int(pick.size), "sample_converged": int((pst == 0).sum()),
            "sample_converged_in_batch": int(min(n // 2, conv_idx.size)), "sample_seconds": t,
            "ms_per_iteration": 1e3 * t_it,
            "form": "one case at a time, separate launches per iteration, host stop test every iteration; "
                    "batch time = the batch's case-iterations x the sample's time per iteration"}


def run_flat_fp32(dpf, torch, job, args, peak, l2):
    """The product loop's iteration rate: FP32 iterations of the same N-1 batch
    from the flat start (Table 2 settings, lr 1e-3), timed over whole check
    intervals (each a graph replay holding the FP64 test), kernel rooflines
    from event-bracketed launches; then the converged count after Table 2's
    budget of 1,000 iterations."""
    s = job.stream
    K, N, g = job.K, job.N, job.g
    opts = dpf.SolveOpts(lr=LR, tol=TOL, check_every=CHECK_EVERY, precision=dpf.FP32, max_iter=10 ** 7,
                         lanes=args.lanes or None, warps=args.warps or None, row_blocks=args.row_blocks or None,
                         pdl=0 if args.no_pdl else None)
    with torch.cuda.stream(s):
        if job.shape_by == "dpf_autotune":
            opts = dpf.dpf_autotune(job.y, job.ws, opts, iters=50, stream=s, n_case=K, outage=job.outage)
        ce = CHECK_EVERY
        n_it = max(ce, (args.flat_iters + ce - 1) // ce * ce)
        dpf.dpf_solve_begin(job.y, job.ws, opts, stream=s, n_case=K, outage=job.outage)
        dpf.dpf_solve_iterate(job.ws, 4 * ce, stream=s)
        s.synchronize()
        l0 = dpf.dpf_kernel_launches(job.ws)
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(s)
        dpf.dpf_solve_iterate(job.ws, n_it, stream=s)
        e1.record(s)
        s.synchronize()
        ms = e0.elapsed_time(e1)
        launches = dpf.dpf_kernel_launches(job.ws) - l0
        dpf.dpf_profile_enable(job.ws, True)
        dpf.dpf_solve_iterate(job.ws, args.profile_steps, stream=s)
        fwd_ms, adj_ms, nf, na = dpf.dpf_kernel_times(job.ws, stream=s)
        dpf.dpf_profile_enable(job.ws, False)
        dpf.dpf_solve_end(job.ws, stream=s, n_case=K)
        r = _outputs(torch, K, N, torch.device("cuda", torch.cuda.current_device()))
        dpf.dpf_solve_batch(job.y, job.ws, dataclasses.replace(opts, max_iter=ITERS_PER_SOLVE), stream=s, n_case=K,
                            outage=job.outage, **r)
        s.synchronize()
    barrier_us = dpf.dpf_grid_barrier_cost(4, 2000, stream=s)
    n_pv = int((g.bus_type == 1).sum())
    n_pq = int((g.bus_type == 0).sum())
    fwd_b, adj_b = algorithmic_bytes(N, n_pv, n_pq, job.y.nnz, K)
    fa, aa = fwd_ms / max(nf, 1), adj_ms / max(na, 1)
    fg, ag = fwd_b / (fa / 1e3) / 1e9, adj_b / (aa / 1e3) / 1e9
    st = r["status"].cpu().numpy()
    mm = r["max_mismatch"].cpu().numpy()
    return {
        "settings": f"flat start, FP32 iterations, Adam lr {LR} with Table 2's betas and plateau",
        "ms_per_iteration": ms / n_it,
        "case_iterations_per_s": K * n_it / (ms / 1e3),
        "timed_iterations": n_it, "fp64_checks_in_timed_region": n_it // ce,
        "graph_replays_in_timed_region": n_it // ce, "kernel_launches_in_timed_region": int(launches),
        "roofline": {"kernel": "k_adj (adjoint SpMV + gradient + Adam)", "bound": "hbm", "unit": "GB/s",
                     "achieved": ag, "peak": peak, "frac": ag / peak, "avg_launch_ms": aa,
                     "algorithmic_bytes_per_launch": adj_b, "traffic": _ncu_traffic("k_adj_n1_2kbus"),
                     "fwd": {"kernel": "k_fwd2" if (opts.pair_cases or 0) & 1 else "k_fwd", "achieved": fg,
                             "frac": fg / peak, "avg_launch_ms": fa, "algorithmic_bytes_per_launch": fwd_b,
                             "frac_of_l2_peak": fg / l2["gbs"], "traffic": _ncu_traffic("k_fwd_n1_2kbus")},
                     "fwd_adj_combined_gbs": (fwd_b + adj_b) / ((fa + aa) / 1e3) / 1e9,
                     "fwd_adj_combined_frac": (fwd_b + adj_b) / ((fa + aa) / 1e3) / 1e9 / peak,
                     "note": "the two passes, timed apart; the timed iterations run on chip"},
        "launch_shape": {"lanes": opts.lanes, "warps": opts.warps, "row_blocks": opts.row_blocks,
                         "pair_cases": opts.pair_cases, "stage_v": opts.stage_v},
        "after_table2_budget": {"iterations": ITERS_PER_SOLVE, "converged": int((st == 0).sum()),
                                "mismatch_p50": float(np.median(mm)), "mismatch_max": float(mm.max())},
        "persistent_launch": {
            "grid_barrier_us": barrier_us, "ctas_per_sm": 4,
            "pipelined_iteration_us": 1e3 * ms / n_it, "bracketed_fwd_plus_adj_us": 1e3 * (fa + aa),
            "note": "one persistent kernel per iteration would replace the two programmatic-dependent launches by "
                    "two grid-wide barriers (forward -> adjoint -> next forward); the pipelined pair already runs "
                    "below the sum of the separately bracketed kernels"},
    }


def c1batch_record(dpf, torch, K, plain_cases=4, precisions=None):
    """Solves/s to 1e-6 p.u. where Alg. 1 reaches it from the flat start: K
    load variants (x U(0.95, 1.05), seeded) of the 30-bus grid in one batch,
    Table 2 settings with lr 1e-2, up to 20,000 iterations, FP64 test every 25.
    Counts only the cases the FP64 test declares converged; the oracle
    recomputes the mismatch of sampled returned states; the plain FP64 form
    solves `plain_cases` of the same cases one at a time."""
    import gridgen
    import oracle
    from oracle.ybus import grid_ybus
    g = gridgen.config_grid("c1_30bus_fp64")
    dev = torch.device("cuda", torch.cuda.current_device())
    rng = np.random.default_rng(0)
    sc = 1 + 0.05 * rng.uniform(-1, 1, (K, 1))
    P, Q = g.p_spec[None] * sc, g.q_spec[None] * sc
    Pt = torch.tensor(P, device=dev)
    Qt = torch.tensor(Q, device=dev)
    y = dpf.dpf_build_ybus(g)
    ws = dpf.dpf_workspace_create(y, K)
    Y = grid_ybus(g)
    out = {}
    precisions = precisions or ((dpf.FP32R, "fp32r"),)
    for prec, name in precisions:
        r = _outputs(torch, K, g.n_bus, dev)
        o = dpf.SolveOpts(precision=prec, lr=1e-2, max_iter=20000, check_every=CHECK_EVERY)
        dpf.dpf_solve_batch(y, ws, o, n_case=K, p_spec=Pt, q_spec=Qt, **r)  # warm-up
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        dpf.dpf_solve_batch(y, ws, o, n_case=K, p_spec=Pt, q_spec=Qt, **r)
        torch.cuda.synchronize()
        wall = time.perf_counter() - t0
        st, it, mm = (r[k].cpu().numpy() for k in ("status", "iters", "max_mismatch"))
        va, vm = r["va"].cpu().numpy(), r["vm"].cpu().numpy()
        err = 0.0
        for k in [0, K // 2, K - 1]:
            f, _ = oracle.mismatch(Y, va[k], vm[k], P[k], Q[k], g.bus_type)
            err = max(err, abs(float(np.abs(f).max()) - float(mm[k])))
        conv = int((st == 0).sum())
        out[name] = {"wall_s": wall, "converged": conv, "solves_to_1e-6_per_s": conv / wall,
                     "iterations_p50": float(np.median(it)), "iterations_max": int(it.max()),
                     "max_mismatch_max": float(mm.max()), "reported_vs_oracle_mismatch_max_abs_diff": err}
    if plain_cases:
        ws1 = dpf.dpf_workspace_create(y, 1)
        r = _outputs(torch, plain_cases, g.n_bus, dev)
        o = dpf.SolveOpts(precision=dpf.FP64, lr=1e-2, max_iter=20000, plain=1)
        dpf.dpf_solve_batch(y, ws1, dataclasses.replace(o, max_iter=50), n_case=1, p_spec=Pt[:1], q_spec=Qt[:1],
                            **{k: v[:1] for k, v in r.items()})
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        dpf.dpf_solve_batch(y, ws1, o, n_case=plain_cases, p_spec=Pt[:plain_cases].contiguous(),
                            q_spec=Qt[:plain_cases].contiguous(), **r)
        torch.cuda.synchronize()
        wall = time.perf_counter() - t0
        conv = int((r["status"].cpu().numpy() == 0).sum())
        out["plain_form_fp64"] = {"cases": plain_cases, "converged": conv, "wall_s": wall,
                                  "solves_to_1e-6_per_s": conv / wall,
                                  "form": "one case at a time, separate launches, host stop test every iteration"}
        best = max(v["solves_to_1e-6_per_s"] for k, v in out.items() if k != "plain_form_fp64")
        out["speedup_vs_plain_form"] = best / (conv / wall) if conv else None
        ws1.free()
    ws.free()
    y.free()
    return {"grid": "c1_30bus_fp64", "cases": K, "tol_pu": TOL, "loads": "x U(0.95, 1.05) per case (seed 0)",
            "settings": "flat start, Table 2 with lr 1e-2, <= 20,000 iterations, FP64 test every 25", **out}


def timeseries_record(dpf, torch, T, newton=False, precision=None):
    """The 10,000-bus grid over T hourly snapshots of the load model, solved
    in windows of 96 by the library's warm-start driver with Table 3's
    settings (first window flat, later windows from the previous window's
    solutions), refined FP32 iterations with the FP64 test; injections in and
    solutions out every window.  The oracle recomputes the mismatch of sampled
    snapshots from the returned voltages.  `newton`: the series again with the
    first window solved by Newton-Raphson from the flat start, the later
    windows by Alg. 1 from it, with the oracle's mismatch of sampled later
    snapshots at their start and at their end.  Then the series with the other
    warm-start reading (every snapshot of a window from the previous window's
    last solution)."""
    import gridgen
    import oracle
    from oracle.ybus import grid_ybus
    from paper_2603_28203_gb300.timeseries import solve_time_series
    precision = dpf.FP32R if precision is None else precision
    g = gridgen.config_grid("c4_timeseries_10kbus")
    t0 = time.perf_counter()
    P, Q = gridgen.time_series(g, T, seed=4)
    t_gen = time.perf_counter() - t0
    y = dpf.dpf_build_ybus(g)
    ws = dpf.dpf_workspace_create(y, 96)
    solve_time_series(y, ws, P[:96], Q[:96], window=96, precision=precision)  # warm-up (first window)
    torch.cuda.synchronize()
    clocks = ClockSampler(ClockSampler.gpu_id(torch.cuda.current_device()),
                          os.path.join(os.environ.get("DPF_CLOCKS_DIR") or tempfile.gettempdir(), "clocks_ts.csv"))
    time.sleep(0.2)
    t0 = time.perf_counter()
    out = solve_time_series(y, ws, P, Q, window=96, precision=precision)
    torch.cuda.synchronize()
    wall = time.perf_counter() - t0
    clk = clocks.stop()
    Y = grid_ybus(g)
    rng = np.random.default_rng(0)
    sample = sorted(set([0, 95, 96, T - 1] + [int(t) for t in rng.choice(T, 4, replace=False)]))
    err = 0.0
    for t in sample:
        f, _ = oracle.mismatch(Y, out["va"][t], out["vm"][t], P[t], Q[t], g.bus_type)
        err = max(err, abs(float(np.max(np.abs(f))) - float(out["max_mismatch"][t])))
    st, it = out["status"], out["iters"]
    # which snapshots have a power-flow solution at all: Newton-Raphson (Alg. 2,
    # the library's, FP64) from the flat start, window by window
    nrh = dpf.dpf_nr_create(y, 96)
    dev = torch.device("cuda", torch.cuda.current_device())
    feas = 0
    for w0 in range(0, T, 96):
        Kw = min(96, T - w0)
        nst = torch.zeros(Kw, dtype=torch.int32, device=dev)
        buf = {k: torch.zeros((Kw, g.n_bus), dtype=torch.float64, device=dev) for k in ("va", "vm")}
        dpf.dpf_nr_solve(nrh, precision=dpf.FP64, tol=1e-8, max_iter=30, n_case=Kw,
                         p_spec=torch.tensor(P[w0:w0 + Kw], device=dev), q_spec=torch.tensor(Q[w0:w0 + Kw], device=dev),
                         status=nst, **buf)
        feas += int((nst == dpf.CASE_CONVERGED).sum())
    nrh.free()
    n_pv = int((g.bus_type == 1).sum())
    n_pq = int((g.bus_type == 0).sum())
    fwd_b, adj_b = algorithmic_bytes(g.n_bus, n_pv, n_pq, y.nnz, 1, spec_per_case=True,
                                     refined=precision == dpf.FP32R)
    bytes_total = float(it.sum()) * (fwd_b + adj_b - 2 * (16 * y.nnz + 5 * g.n_bus))  # per-case streams
    peak, src = _peaks()
    rec = {
        "grid": "c4_timeseries_10kbus", "n_bus": int(g.n_bus), "n_branch": int(g.n_branch), "snapshots": int(T),
        "window": 96, "settings": "Table 3 (first window flat, later windows warm from the previous window)",
        "precision": "fp32r" if precision == dpf.FP32R else "fp32", "tol_pu": TOL,
        "generation_s": t_gen, "wall_s": wall, "snapshots_per_s": T / wall,
        "converged": int((st == 0).sum()), "solves_to_1e-6_per_s": int((st == 0).sum()) / wall,
        "snapshots_with_a_newton_solution": feas,
        "iterations_total": int(it.sum()), "iterations_p50": float(np.median(it)),
        "iterations_first_window_p50": float(np.median(it[:96])),
        "status_counts": {str(k): int((st == k).sum()) for k in (0, 1, 2)},
        "max_mismatch_p50": float(np.median(out["max_mismatch"])),
        "max_mismatch_p99": float(np.percentile(out["max_mismatch"], 99)),
        "algorithmic_gbs": bytes_total / wall / 1e9, "frac_of_hbm_peak": bytes_total / wall / 1e9 / peak,
        "sampled_snapshots": sample, "reported_vs_fp64_oracle_mismatch_max_abs_diff": err, "clocks": clk,
        "note": "wall clock of the whole series incl. per-window injection uploads and solution downloads; "
                "the per-iteration working set (~96 x 10k elements) is L2-resident, so the HBM fraction is "
                "effective, not a DRAM measurement",
    }
    if newton:
        # the first window by Newton-Raphson from the flat start (the caption
        # of Fig. 4), later windows Alg. 1 warm-started from it
        nr = dpf.dpf_nr_create(y, 96)
        kw = dict(window=96, precision=precision, first_newton=nr, newton_from="flat")
        solve_time_series(y, ws, P[:96], Q[:96], **kw)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        out_n = solve_time_series(y, ws, P, Q, **kw)
        torch.cuda.synchronize()
        wall_n = time.perf_counter() - t0
        nr.free()
        later = [t for t in sample if t >= 96]
        start_mm, end_mm = [], []
        for t in later:  # snapshot t starts from the solution of t - 96
            f0, _ = oracle.mismatch(Y, out_n["va"][t - 96], out_n["vm"][t - 96], P[t], Q[t], g.bus_type)
            f1, _ = oracle.mismatch(Y, out_n["va"][t], out_n["vm"][t], P[t], Q[t], g.bus_type)
            start_mm.append(float(np.max(np.abs(f0))))
            end_mm.append(float(np.max(np.abs(f1))))
        st_n = out_n["status"]
        rec["first_window_newton"] = {
            "wall_s": wall_n, "snapshots_per_s": T / wall_n,
            "first_window_newton_converged_1e-10": int((st_n[:96] == 0).sum()),
            "first_window_newton_steps_p50": float(np.median(out_n["iters"][:96])),
            "later_windows_dpf_converged": int((st_n[96:] == 0).sum()), "later_windows": int(max(0, T - 96)),
            "max_mismatch_p50_later_windows": float(np.median(out_n["max_mismatch"][96:])) if T > 96 else None,
            "sampled_later_snapshots": later,
            "sampled_start_max_mismatch_oracle": start_mm, "sampled_end_max_mismatch_oracle": end_mm}
    # the other warm-start reading: a window's every snapshot from the previous
    # window's last solution
    solve_time_series(y, ws, P[:96], Q[:96], window=96, precision=precision, warm_from="last")
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    out_l = solve_time_series(y, ws, P, Q, window=96, precision=precision, warm_from="last")
    torch.cuda.synchronize()
    wall_l = time.perf_counter() - t0
    rec["warm_from_last_snapshot"] = {
        "wall_s": wall_l, "snapshots_per_s": T / wall_l, "converged": int((out_l["status"] == 0).sum()),
        "max_mismatch_p50_later_windows": float(np.median(out_l["max_mismatch"][96:])) if T > 96 else None}
    ws.free()
    y.free()
    return rec


def uneven_record(dpf, torch, args):
    """The uneven batch of the parameter-identification workload: 64 synthetic
    grids of log-uniform sizes (300 to 80,000 buses; seeded) in one
    block-diagonal system with one slack per island, and 16 hourly operating
    points (the time-series load model) as the cases.  Times (a) FP32 DPF
    iterations over the whole batch and (b) one parameter-identification step
    (the loss and its branch adjoint w.r.t. the series g, b of every branch,
    then the two Adam updates) at the iterate the solve reached.  FP64 oracle
    check of S_calc on one operating point."""
    import gridgen
    import oracle
    from oracle.ybus import grid_ybus
    from paper_2603_28203_gb300.paramid import identify_branches
    dev = torch.device("cuda", torch.cuda.current_device())
    stream = torch.cuda.Stream(dev)
    t0 = time.time()
    sizes = gridgen.uneven_sizes(64, 100)
    grids = [gridgen.make_grid(int(n), 1000 + i, load_scale=0.1) for i, n in enumerate(sizes)]
    cat = gridgen.concat_grids(grids)
    K = 16
    P, Q = gridgen.time_series(cat, K, seed=5)
    t_gen = time.time() - t0
    n_pv = int((cat.bus_type == 1).sum())
    n_pq = int((cat.bus_type == 0).sum())
    y = dpf.dpf_build_ybus(cat, stream=stream)
    ws = dpf.dpf_workspace_create(y, K)
    p_t = torch.tensor(P, dtype=torch.float64, device=dev)
    q_t = torch.tensor(Q, dtype=torch.float64, device=dev)
    opts = dpf.SolveOpts(lr=1e-3, precision=dpf.FP32, check_every=25, max_iter=10 ** 6,
                         lanes=args.lanes or None, warps=args.warps or None, row_blocks=args.row_blocks or None)
    fixed_shape = bool(args.lanes or args.warps or args.row_blocks)
    n_it = max(25, (args.uneven_iters + 24) // 25 * 25)
    with torch.cuda.stream(stream):
        if not (args.no_autotune or fixed_shape):
            opts = dpf.dpf_autotune(y, ws, opts, iters=20, stream=stream, n_case=K, p_spec=p_t, q_spec=q_t)
        dpf.dpf_solve_begin(y, ws, opts, stream=stream, n_case=K, p_spec=p_t, q_spec=q_t)
        dpf.dpf_solve_iterate(ws, 50, stream=stream)
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        stream.synchronize()
        e0.record(stream)
        dpf.dpf_solve_iterate(ws, n_it, stream=stream)
        e1.record(stream)
        stream.synchronize()
        ms_it = e0.elapsed_time(e1) / n_it
        dpf.dpf_profile_enable(ws, True)
        dpf.dpf_solve_iterate(ws, 50, stream=stream)
        f_ms, a_ms, nf, na = dpf.dpf_kernel_times(ws, stream=stream)
        dpf.dpf_profile_enable(ws, False)
        out = {k: torch.empty((K, cat.n_bus), dtype=torch.float64, device=dev) for k in ("va", "vm")}
        st = torch.empty(K, dtype=torch.int32, device=dev)
        mm = torch.empty(K, dtype=torch.float64, device=dev)
        dpf.dpf_solve_end(ws, stream=stream, n_case=K, va=out["va"], vm=out["vm"], status=st, max_mismatch=mm)
        stream.synchronize()
        pert = gridgen.perturb_branches(cat, 5)
        y0 = 1.0 / (pert.r + 1j * pert.x)
        g0 = torch.tensor(y0.real, dtype=torch.float64, device=dev)
        b0 = torch.tensor(y0.imag, dtype=torch.float64, device=dev)
        identify_branches(y, ws, out["va"], out["vm"], p_t, q_t, g0, b0, iters=2, stream=stream)
        stream.synchronize()
        n_pid = args.uneven_pid_steps
        e0.record(stream)
        identify_branches(y, ws, out["va"], out["vm"], p_t, q_t, g0, b0, iters=n_pid, stream=stream)
        e1.record(stream)
        stream.synchronize()
        ms_pid = e0.elapsed_time(e1) / n_pid
        pc, qc = dpf.dpf_power(y, ws, out["va"][:1].contiguous(), out["vm"][:1].contiguous(), precision=dpf.FP32,
                               stream=stream)
        stream.synchronize()
    S = oracle.s_calc(grid_ybus(cat), out["vm"][0].cpu().numpy() * np.exp(1j * out["va"][0].cpu().numpy()))
    err = max(np.abs(pc[0].cpu().numpy() - S.real).max(), np.abs(qc[0].cpu().numpy() - S.imag).max())
    fwd_b, adj_b = algorithmic_bytes(cat.n_bus, n_pv, n_pq, y.nnz, K, spec_per_case=True)
    peak, src = _peaks()
    stc = st.cpu().numpy()
    ws.free()
    y.free()
    return {
        "config": {"grids": int(len(sizes)), "bus_sizes": "log-uniform 300-80,000 (seed 100)",
                   "n_bus": int(cat.n_bus), "n_branch": int(cat.n_branch), "operating_points": K,
                   "largest_grid": int(sizes.max()), "smallest_grid": int(sizes.min()),
                   "precision": "fp32 iterations, FP64 master and test", "generation_s": round(t_gen, 1),
                   "launch_shape": {"lanes": opts.lanes, "warps": opts.warps, "row_blocks": opts.row_blocks,
                                    "chosen_by": "command line" if fixed_shape else
                                    "library default" if args.no_autotune else "dpf_autotune"}},
        "ms_per_iteration": ms_it, "timed_iterations": n_it,
        "case_iterations_per_s": K / (ms_it / 1e3),
        "bus_iterations_per_s": K * cat.n_bus / (ms_it / 1e3),
        "roofline": {"bound": "hbm", "unit": "GB/s", "peak": peak, "peak_source": src,
                     "achieved": (fwd_b + adj_b) / (ms_it / 1e3) / 1e9,
                     "frac": (fwd_b + adj_b) / (ms_it / 1e3) / 1e9 / peak,
                     "algorithmic_bytes_per_iteration": fwd_b + adj_b,
                     "fwd_us": 1e3 * f_ms / max(nf, 1), "adj_us": 1e3 * a_ms / max(na, 1),
                     "adj_frac": adj_b / (a_ms / max(na, 1) / 1e3) / 1e9 / peak},
        "paramid_step_ms": ms_pid,
        "paramid_step": "Y values from (g, b) + forward pass + branch adjoint (g, b of every branch) over all "
                        "operating points + 2 Adam updates (dpf_paramid_step, operating points staged once)",
        "status_counts": {str(k): int((stc == k).sum()) for k in (0, 1, 2)},
        "max_mismatch_p50": float(np.median(mm.cpu().numpy())),
        "fp32_S_max_abs_error_vs_fp64_oracle": float(err),
    }


# ---------------------------------------------------------------------------
# scaling sweep (--workload scaling): single grids, node and edge scaling
# ---------------------------------------------------------------------------
def run_scaling(args):
    """Time FP32 DPF iterations of single grids (K = 1) as the bus and branch
    counts grow: the linear-cost claim of Sec. 5.2 / 5.4.3.  One JSON line per
    grid; each carries the FP64 oracle check of S_calc on sampled buses."""
    import torch
    import gridgen
    import oracle
    from oracle.ybus import grid_ybus
    from paper_2603_28203_gb300.build import LIB, build
    if not os.path.exists(LIB):
        build()
    import paper_2603_28203_gb300 as dpf
    dev = torch.device("cuda", 0)
    stream = torch.cuda.Stream(dev)
    sizes = [int(x) for x in args.scaling_sizes.split(",") if x]
    extra = [int(x) for x in args.scaling_edges.split(",") if x]
    grids = [("nodes", gridgen.make_grid(n, 1, load_scale=0.1)) for n in sizes]
    if extra:
        base = gridgen.make_grid(10_000, 1, load_scale=0.1)
        grids += [("edges", gridgen.add_random_branches(base, m, 7)) for m in extra]
    for kind, g in grids:
        y = dpf.dpf_build_ybus(g, stream=stream)
        ws = dpf.dpf_workspace_create(y, 1)
        opts = dpf.SolveOpts(lr=1e-3, precision=dpf.FP32, check_every=25, max_iter=10 ** 6,
                             lanes=args.lanes or None, warps=args.warps or None, row_blocks=args.row_blocks or None)
        with torch.cuda.stream(stream):
            if not (args.no_autotune or args.lanes or args.warps or args.row_blocks):
                opts = dpf.dpf_autotune(y, ws, opts, iters=50, stream=stream, n_case=1)
            dpf.dpf_solve_begin(y, ws, opts, stream=stream, n_case=1)
            dpf.dpf_solve_iterate(ws, 50, stream=stream)
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            n_it = 500
            e0.record(stream)
            dpf.dpf_solve_iterate(ws, n_it, stream=stream)
            e1.record(stream)
            stream.synchronize()
            ms = e0.elapsed_time(e1) / n_it
            dpf.dpf_profile_enable(ws, True)
            dpf.dpf_solve_iterate(ws, 50, stream=stream)
            f_ms, a_ms, nf, na = dpf.dpf_kernel_times(ws, stream=stream)
            dpf.dpf_profile_enable(ws, False)
            # sampled parity of the forward evaluation against the oracle
            rng = np.random.default_rng(0)
            va = torch.tensor(0.05 * rng.standard_normal((1, g.n_bus)), dtype=torch.float64, device=dev)
            vm = torch.tensor(1 + 0.02 * rng.standard_normal((1, g.n_bus)), dtype=torch.float64, device=dev)
            p, q = dpf.dpf_power(y, ws, va, vm, precision=dpf.FP32, stream=stream)
            stream.synchronize()
        Y = grid_ybus(g)
        S = oracle.s_calc(Y, vm[0].cpu().numpy() * np.exp(1j * va[0].cpu().numpy()))
        err = max(np.abs(p[0].cpu().numpy() - S.real).max(), np.abs(q[0].cpu().numpy() - S.imag).max())
        n_pv = int((g.bus_type == 1).sum())
        n_pq = int((g.bus_type == 0).sum())
        fwd_b, adj_b = algorithmic_bytes(g.n_bus, n_pv, n_pq, y.nnz, 1)
        print(json.dumps({"workload": "scaling", "kind": kind, "n_bus": g.n_bus, "n_branch": g.n_branch,
                          "nnz": y.nnz, "ms_per_iteration": ms, "us_per_iteration_per_1k_nnz": 1e3 * ms / (y.nnz / 1e3),
                          "fwd_us": 1e3 * f_ms / max(nf, 1), "adj_us": 1e3 * a_ms / max(na, 1),
                          "launch_shape": {"lanes": opts.lanes, "warps": opts.warps, "row_blocks": opts.row_blocks,
                                           "stage_y": opts.stage_y},
                          "algorithmic_gbs": (fwd_b + adj_b) / (ms / 1e3) / 1e9,
                          "fp32_S_max_abs_error_vs_fp64_oracle": float(err)}), flush=True)
        ws.free()
        y.free()

def _lib_for_workload():
    import torch
    from paper_2603_28203_gb300.build import LIB, build
    if not os.path.exists(LIB):
        build()
    import paper_2603_28203_gb300 as dpf
    torch.cuda.set_device(0)
    return dpf, torch


def run_uneven(args):
    """--workload uneven: the uneven 64-grid batch (one JSON line)."""
    dpf, torch = _lib_for_workload()
    print(json.dumps({"workload": "uneven", **uneven_record(dpf, torch, args)}), flush=True)


def run_timeseries(args):
    """--workload timeseries: the 10,000-bus time series (one JSON line), plus
    the variant whose first window goes through Newton-Raphson."""
    dpf, torch = _lib_for_workload()
    prec = dict(fp32r=dpf.FP32R, fp32=dpf.FP32)[args.ts_precision]
    print(json.dumps({"workload": "timeseries", **timeseries_record(dpf, torch, args.ts_hours, newton=True,
                                                                      precision=prec)}), flush=True)


def run_flat(args):
    """--workload flat: the flat-start FP32 iteration rate of the N-1 batch
    alone (the n1_flat_fp32 sub-record; one JSON line)."""
    dpf, torch = _lib_for_workload()
    g, outages = _workload()
    stream = torch.cuda.Stream(torch.device("cuda", 0))
    job = N1Job(dpf, torch, g, outages, stream, args.n1_budget, args)
    peak, _ = _peaks()
    l2 = _l2_read_peak(dpf, torch, stream)
    print(json.dumps({"workload": "flat", **run_flat_fp32(dpf, torch, job, args, peak, l2)}), flush=True)


def run_c1batch(args):
    """--workload c1batch: the 30-bus batch in every precision (one JSON line)."""
    dpf, torch = _lib_for_workload()
    rec = c1batch_record(dpf, torch, args.c1_cases, plain_cases=args.plain_cases,
                         precisions=((dpf.FP64, "fp64"), (dpf.MIXED, "mixed"), (dpf.FP32, "fp32"),
                                     (dpf.FP32R, "fp32r")))
    print(json.dumps({"workload": "c1batch", **rec}), flush=True)


def _nr_point_worker(item):
    """FP64 oracle Newton-Raphson of one grid at one operating point."""
    import oracle
    from oracle.ybus import grid_ybus
    g, p, q = item
    r = oracle.nr_solve(grid_ybus(g), p, q, g.bus_type, g.vm_set)
    return r["va"], r["vm"], bool(r["converged"])


def run_paramid(args):
    """Parameter identification against the ground truth (the uneven-batch
    experiment at a size the FP64 oracle can measure): `--pid-grids` synthetic
    grids of log-uniform 300-3,000 buses in one block-diagonal batch,
    `--pid-points` (16) hourly operating points measured by the oracle's
    Newton-Raphson at the true branch parameters -- the first hours of the
    load model at which every grid has a solution (`--pid-hours first`), or
    hours spread over the year (`spread`: 64 candidates evenly spaced) --
    branch r and x perturbed by U(-10%, +10%), then Adam on the series g, b
    of every branch from the branch adjoint (dpf_paramid_step).  Reports the
    relative errors of r and x before and after, the loss, and the time per
    step.  One JSON line."""
    import multiprocessing as mp
    import gridgen
    sizes = gridgen.uneven_sizes(args.pid_grids, 200, lo=300, hi=3000)
    grids = [gridgen.make_grid(int(n), 2000 + i, load_scale=0.1) for i, n in enumerate(sizes)]
    cat = gridgen.concat_grids(grids)
    K = args.pid_points  # operating points: the first candidate hours at which every grid has a solution
    hours = np.arange(48) if args.pid_hours == "first" else np.linspace(0, 8759, 64).round().astype(int)
    H = hours.size
    PQ = [gridgen.time_series(cat, 1, seed=5, t0=int(h)) for h in hours]
    P = np.concatenate([a for a, _ in PQ])
    Q = np.concatenate([b for _, b in PQ])
    off = np.cumsum([0] + [g.n_bus for g in grids])
    items = []
    for gi, g in enumerate(grids):
        sl = slice(off[gi], off[gi + 1])
        for k in range(H):
            items.append((g, P[k, sl], Q[k, sl]))
    t0 = time.perf_counter()
    with mp.get_context("spawn").Pool(len(os.sched_getaffinity(0))) as pool:  # before any CUDA call
        res = pool.map(_nr_point_worker, items)
    t_nr = time.perf_counter() - t0
    va = np.zeros((H, cat.n_bus))
    vm = np.zeros((H, cat.n_bus))
    ok = np.ones(H, bool)
    for j, (a, m, conv) in enumerate(res):
        gi, k = divmod(j, H)
        va[k, off[gi]:off[gi + 1]] = a
        vm[k, off[gi]:off[gi + 1]] = m
        ok[k] &= conv
    import torch
    from paper_2603_28203_gb300.build import LIB, build
    if not os.path.exists(LIB):
        build()
    import paper_2603_28203_gb300 as dpf
    from paper_2603_28203_gb300.paramid import identify_branches
    dev = torch.device("cuda", 0)
    stream = torch.cuda.Stream(dev)
    kk = np.where(ok)[0][:K]
    t = lambda a: torch.tensor(np.ascontiguousarray(a[kk]), dtype=torch.float64, device=dev)
    y = dpf.dpf_build_ybus(cat, stream=stream)
    ws = dpf.dpf_workspace_create(y, len(kk))
    z_true = cat.r + 1j * cat.x
    pert = gridgen.perturb_branches(cat, 5)
    ys0 = 1.0 / (pert.r + 1j * pert.x)
    g0 = torch.tensor(ys0.real, dtype=torch.float64, device=dev)
    b0 = torch.tensor(ys0.imag, dtype=torch.float64, device=dev)
    n = args.pid_steps
    with torch.cuda.stream(stream):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        pid_prec = dict(fp32=dpf.FP32, fp64=dpf.FP64)[args.pid_precision]
        g, b, hist = identify_branches(y, ws, t(va), t(vm), t(P), t(Q), g0, b0, n, lr=args.pid_lr,
                                       precision=pid_prec, record_every=max(1, n // 4), stream=stream)
        torch.cuda.synchronize()
        wall = time.perf_counter() - t0
        out0 = dpf.dpf_loss_backward(y, ws, t(va), t(vm), t(P), t(Q), g_series=g0, b_series=b0,
                                     precision=dpf.FP64, want=("loss",), stream=stream)
        out1 = dpf.dpf_loss_backward(y, ws, t(va), t(vm), t(P), t(Q), g_series=g, b_series=b,
                                     precision=dpf.FP64, want=("loss",), stream=stream)
        stream.synchronize()
    z1 = 1.0 / (g.cpu().numpy() + 1j * b.cpu().numpy())
    z0 = pert.r + 1j * pert.x
    rel = lambda a, b_: np.abs(a - b_) / np.abs(b_)
    def stats(z):
        er, ex = rel(z.real, z_true.real), rel(z.imag, z_true.imag)
        return {"r_median": float(np.median(er)), "r_max": float(er.max()),
                "x_median": float(np.median(ex)), "x_max": float(ex.max())}
    print(json.dumps({
        "workload": "paramid",
        "config": {"grids": int(len(sizes)), "bus_sizes": "log-uniform 300-3,000 (seed 200)",
                   "n_bus": int(cat.n_bus), "n_branch": int(cat.n_branch), "operating_points": int(len(kk)),
                   "hours_with_a_solution": f"{int(ok.sum())} of {H} candidates ({args.pid_hours})",
                   "hours_used": [int(h) for h in hours[kk]],
                   "measurements": "FP64 oracle Newton-Raphson at the true parameters",
                   "perturbation": "r, x x U(0.9, 1.1) per branch (seed 5)",
                   "steps": n, "lr": args.pid_lr, "precision": f"{args.pid_precision} forward and adjoint, FP64 loss"},
        "oracle_nr_s": t_nr,
        "error_before": stats(z0), "error_after": stats(z1),
        "loss_fp64_before": float(out0["loss"].sum()), "loss_fp64_after": float(out1["loss"].sum()),
        "ms_per_step": 1e3 * wall / n,
    }), flush=True)
    ws.free()
    y.free()


def dc_bytes_per_iteration(n_bus, nnz, n_case):
    """Bytes one CG iteration of dpf_dc_solve must move (FP64): per element,
    k_dc_spmv_dir reads z (gathered, each value once from DRAM), p and q and
    writes p' and q' (40), k_dc_update_case reads p', q', x, r and writes x,
    r, z (56); B in CSR (8 B value + 4 B column per nonzero, row pointers),
    the inverse diagonal and the bus types once per launch."""
    shared = 12 * nnz + 4 * (n_bus + 1) + 8 * n_bus + n_bus
    return n_case * n_bus * (40 + 56) + 2 * shared


# Nominal FP64 rate of the part (no measured FP64 peak exists for this machine):
# 1.25 TFLOP/s, about 2 FP64 FMA per clock per SM at 152 SMs and 2.07 GHz.
FP64_NOMINAL_TFLOPS = 1.25


def dc_flops_per_iteration(n_bus, nnz, n_case, n_slack=1):
    """Flops of one CG iteration (FMA = 2; carried out in double-float
    arithmetic, each about 2^-48 accurate): per unknown row of a case,
    the row of B' z (one FMA per nonzero), p' = z + beta p, q' = (B'z) +
    beta q and the p'.q' term (3 FMA); then x, r, r.z and r.r (4 FMA) and
    z = r * (1 / B_ii) (1 multiply).  Slack rows do none of it; a slack
    row's nonzeros are left in (an upper bound by a few entries)."""
    rows = n_bus - n_slack
    return n_case * (2 * nnz + rows * (2 * 7 + 1))


def run_dc(args):
    """The DC approximation (Sec. 2's comparison model, Alg. 2's optional
    initialisation) on the N-1 batch: dpf_dc_solve's batched CG for all
    2,379 cases (relative residual 1e-10), sampled cases against the oracle,
    and Alg. 1 from the DC angles vs from the flat start after the same
    number of iterations.  One JSON line."""
    import torch
    import oracle
    from paper_2603_28203_gb300.build import LIB, build
    if not os.path.exists(LIB):
        build()
    import paper_2603_28203_gb300 as dpf
    g, outages = _workload()
    K = outages.size
    dev = torch.device("cuda", 0)
    stream = torch.cuda.Stream(dev)
    y = dpf.dpf_build_ybus(g, stream=stream)
    ws = dpf.dpf_workspace_create(y, K)
    od = torch.tensor(outages, dtype=torch.int32, device=dev)
    with torch.cuda.stream(stream):
        dpf.dpf_dc_solve(y, ws, K, outage=od, tol=1e-10, stream=stream)  # warm-up
        stream.synchronize()
        t0 = time.perf_counter()
        out = dpf.dpf_dc_solve(y, ws, K, outage=od, tol=1e-10, stream=stream)
        stream.synchronize()
        wall = time.perf_counter() - t0
    it = out["iters"].cpu().numpy()
    th = out["va"].cpu().numpy()
    rng = np.random.default_rng(0)
    err = 0.0
    for k in sorted(set([0, K - 1] + [int(v) for v in rng.choice(K, 4, replace=False)])):
        ref = oracle.dc_solve(g.n_bus, g.f_bus, g.t_bus, g.x, g.tap, g.bus_type, g.p_spec, va_slack=g.va_slack,
                              outage=int(outages[k]))
        err = max(err, float(np.abs(th[k] - ref).max() / np.abs(ref).max()))
    # Alg. 1 from the DC angles vs flat, same iteration budget
    mm = {}
    for start in ("flat", "dc"):
        res = dict(va=torch.empty((K, g.n_bus), dtype=torch.float64, device=dev),
                   vm=torch.empty((K, g.n_bus), dtype=torch.float64, device=dev),
                   status=torch.empty(K, dtype=torch.int32, device=dev),
                   max_mismatch=torch.empty(K, dtype=torch.float64, device=dev))
        opts = dpf.SolveOpts(lr=LR, tol=TOL, check_every=CHECK_EVERY, max_iter=ITERS_PER_SOLVE,
                             dc_start=1 if start == "dc" else 0)
        with torch.cuda.stream(stream):
            dpf.dpf_solve_batch(y, ws, opts, stream=stream, n_case=K, outage=od, **res)
            stream.synchronize()
        m = res["max_mismatch"].cpu().numpy()
        mm[start] = {"p50": float(np.median(m)), "max": float(m.max()),
                     "converged": int((res["status"].cpu().numpy() == 0).sum())}
    iters_max = int(it.max())
    b = dc_bytes_per_iteration(g.n_bus, y.nnz, K)
    fl = dc_flops_per_iteration(g.n_bus, y.nnz, K, n_slack=int((g.bus_type == 2).sum()))
    peak, src = _peaks()
    print(json.dumps({
        "workload": "dc",
        "config": {"grid": "c3_n1_2kbus", "n_bus": int(g.n_bus), "cases": int(K), "tol_rel_residual": 1e-10,
                   "solver": "Jacobi-preconditioned CG on chip, one CTA per case, double-float vectors and "
                             "scalars (FP32 pairs)"},
        "wall_ms": 1e3 * wall,
        "cg_iterations_max": iters_max, "cg_iterations_p50": float(np.median(it)),
        "us_per_cg_iteration": 1e6 * wall / max(iters_max, 1),
        "roofline": {"bound": "instruction issue",
                     "two_launch_form": {"bytes_per_iteration": b, "floor_us_per_iteration": b / peak / 1e3,
                                         "peak_gbs": peak, "peak_source": src},
                     "flops": {"unit": "TFLOP/s", "achieved": fl * iters_max / wall / 1e12,
                               "algorithmic_flops_per_iteration": fl,
                               "note": "double-float arithmetic on the FP32 pipes (nominal FP64 rate "
                                       f"{FP64_NOMINAL_TFLOPS} TFLOP/s for comparison)"},
                     "note": "vectors and matrix stay on chip; each case stops by itself"},
        "max_rel_error_vs_oracle_sampled": err,
        "alg1_after_1000_iterations": mm,
    }), flush=True)
    ws.free()
    y.free()


def run_warmstart(args):
    """Iterations to 1e-6 p.u. from a flat start and from the solution of a
    neighbouring operating point (the paper's warm-start claim, Sec. 5.4.2),
    on the 30-bus grid, the one where Alg. 1 reaches 1e-6 (FP64, one case):
    the base loads solved flat, then loads x 1.01 / 1.02 / 1.05 solved flat
    and warm with Table 2's settings at several rates and with Table 3's
    settings for t > 0.  One JSON line."""
    import torch
    import gridgen
    from paper_2603_28203_gb300.build import LIB, build
    if not os.path.exists(LIB):
        build()
    import paper_2603_28203_gb300 as dpf
    from paper_2603_28203_gb300.timeseries import TABLE3_T1
    g = gridgen.config_grid("c1_30bus_fp64")
    y = dpf.dpf_build_ybus(g)
    ws = dpf.dpf_workspace_create(y, 1)
    dev = torch.device("cuda", 0)
    cap = args.warm_max_iter

    def solve(p, q, opts, start=None):
        r = {k: torch.zeros((1, g.n_bus), dtype=torch.float64, device=dev) for k in ("va", "vm")}
        r.update(iters=torch.zeros(1, dtype=torch.int32, device=dev),
                 status=torch.zeros(1, dtype=torch.int32, device=dev))
        if start is not None:
            r["va"].copy_(start["va"])
            r["vm"].copy_(start["vm"])
        dpf.dpf_solve_batch(y, ws, opts, n_case=1, p_spec=torch.tensor(p[None], dtype=torch.float64, device=dev),
                            q_spec=torch.tensor(q[None], dtype=torch.float64, device=dev), **r)
        torch.cuda.synchronize()
        return r

    def iters(r):
        return int(r["iters"][0]) if int(r["status"][0]) == 0 else None  # None: not converged within the cap

    t2 = dpf.SolveOpts(precision=dpf.FP64, lr=1e-2, max_iter=cap, check_every=1)
    base = solve(g.p_spec, g.q_spec, t2)
    rows = []
    t3 = {k: v for k, v in TABLE3_T1.items() if k != "max_iter"}
    for scale in (1.01, 1.02, 1.05):
        p, q = g.p_spec * scale, g.q_spec * scale
        row = {"load_scale": scale, "flat_table2_lr1e-2": iters(solve(p, q, t2))}
        for lr in (1e-2, 1e-3, 2.7e-4):
            o = dpf.SolveOpts(precision=dpf.FP64, lr=lr, max_iter=cap, check_every=1, flat_start=0)
            row[f"warm_table2_lr{lr:g}"] = iters(solve(p, q, o, base))
        o = dpf.SolveOpts(precision=dpf.FP64, max_iter=cap, check_every=1, flat_start=0, **t3)
        row["warm_table3_t>0"] = iters(solve(p, q, o, base))
        rows.append(row)
    print(json.dumps({"workload": "warmstart", "grid": "c1_30bus_fp64", "tol_pu": 1e-6, "precision": "fp64",
                      "iteration_cap": cap, "base_flat_iterations": iters(base), "rows": rows,
                      "note": "None = not converged within the cap"}), flush=True)
    ws.free()
    y.free()


def nr_bytes_per_step(n_bus, n_pos, n_pairs, n_case):
    """Bytes one Newton step of dpf_nr_solve must move (FP64 state, factor of
    `fb` bytes per block) for n_case active cases: k_nr_volt reads theta,
    |V| and writes V (32 B per bus); k_nr_eval gathers V (each value once)
    and writes I and the right-hand side (48); k_nr_check reads it (16);
    k_nr_assemble reads V, I, |V| (40 per bus) and writes every block of the
    filled pattern; k_nr_lu reads every block once as its own target and
    twice per block product, writes every block but the diagonals and the
    inverse diagonals, and reads/writes the right-hand side twice (64 per
    bus) plus one right-hand-side read per off-diagonal block in the two
    substitutions; k_nr_update reads dx, theta, |V| and writes theta, |V|
    (48).  The schedule (shared by all cases) is left out; so is the
    pivots' diagonal block that each L target re-forms (not needed by the
    arithmetic)."""
    def per_case(fb):
        bus = 32 + 48 + 16 + 40 + 64 + 48
        lu = fb * (n_pos + 2 * n_pairs) + fb * (n_pos - n_bus) + fb * n_bus + 16 * (n_pos - n_bus)
        return n_bus * bus + fb * n_pos + lu
    return {"fp64": n_case * per_case(32), "fp32": n_case * per_case(16)}


def run_nr(args):
    """Newton-Raphson (Alg. 2) on the GPU over the N-1 batch (dpf_nr_solve):
    all 2,379 cases from the flat start to 1e-6 and 1e-10 p.u. with the FP64
    and the FP32 factor, and the hybrid of Sec. 6 (Alg. 1 for a few hundred
    iterations, then Newton from its state).  Solves/s count converged cases
    only; cases the oracle's NR cannot solve either are listed.  The oracle's
    NR (scipy sparse LU) on a bounded sample of cases, one per host core, is
    the CPU baseline.  One JSON line."""
    import torch
    import oracle
    from oracle.ybus import grid_ybus
    from paper_2603_28203_gb300.build import LIB, build
    if not os.path.exists(LIB):
        build()
    import paper_2603_28203_gb300 as dpf
    g, outages = _workload()
    K = outages.size
    cores = len(os.sched_getaffinity(0))
    sample = [int(c) for c in np.random.default_rng(7).choice(outages, size=8 * cores, replace=False)]
    cpu = _oracle_nr_sample(sample, cores)
    dev = torch.device("cuda", 0)
    y = dpf.dpf_build_ybus(g)
    nr = dpf.dpf_nr_create(y, K)
    st = nr.stats()
    od = torch.tensor(outages.astype(np.int32), device=dev)
    peak, src = _peaks()

    def state():
        return dict(va=torch.zeros((K, g.n_bus), dtype=torch.float64, device=dev),
                    vm=torch.ones((K, g.n_bus), dtype=torch.float64, device=dev),
                    iters=torch.empty(K, dtype=torch.int32, device=dev),
                    status=torch.empty(K, dtype=torch.int32, device=dev),
                    max_mismatch=torch.empty(K, dtype=torch.float64, device=dev))

    def timed(fn, reps=3):
        best = None
        for _ in range(reps):
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            fn()
            e1.record()
            torch.cuda.synchronize()
            t = e0.elapsed_time(e1) / 1e3
            best = t if best is None else min(best, t)
        return best

    out = {}
    steps_bytes = nr_bytes_per_step(g.n_bus, st["n_pos"], st["n_pairs"], 1)
    for prec, pname in ((dpf.FP64, "fp64"), (dpf.FP32, "fp32")):
        if pname not in args.nr_precision.split(","):
            continue
        for tol in (1e-6, 1e-10):
            r = state()
            wall = timed(lambda: dpf.dpf_nr_solve(nr, precision=prec, tol=tol, max_iter=args.nr_max_iter,
                                                  n_case=K, outage=od, **r))
            it, stt, mm = (r[k].cpu().numpy() for k in ("iters", "status", "max_mismatch"))
            conv = stt == 0
            steps = int(it.sum())  # Newton steps taken over all cases
            out[f"{pname}_tol{tol:g}"] = {
                "wall_ms": 1e3 * wall, "converged": int(conv.sum()), "solves_per_s": float(conv.sum() / wall),
                "newton_steps_p50": float(np.median(it)), "newton_steps_max": int(it.max()),
                "not_converged_outages": [int(outages[k]) for k in np.flatnonzero(~conv)],
                "max_mismatch_converged": float(mm[conv].max()),
                "achieved_gbs_algorithmic": steps * steps_bytes[pname] / wall / 1e9,
                "hbm_frac": steps * steps_bytes[pname] / wall / 1e9 / peak,
            }
    # Sec. 6 hybrid: Alg. 1 (FP32 iterations, Table 2, lr 1e-2) then Newton from its state
    ws = dpf.dpf_workspace_create(y, K)
    hyb = {}
    for t_dpf in (100, 300):
        r = state()
        o = dpf.SolveOpts(lr=LR, max_iter=t_dpf, check_every=CHECK_EVERY, tol=TOL)

        def both():
            dpf.dpf_solve_batch(y, ws, o, n_case=K, outage=od, **r)
            dpf.dpf_nr_solve(nr, precision=dpf.FP64, tol=1e-10, max_iter=args.nr_max_iter, flat_start=False,
                             fallback=True, n_case=K, outage=od, **r)
        wall = timed(both, reps=2)
        it, stt = r["iters"].cpu().numpy(), r["status"].cpu().numpy()
        conv = stt == 0
        hyb[f"dpf{t_dpf}_then_nr"] = {"wall_ms": 1e3 * wall, "converged": int(conv.sum()),
                                      "solves_per_s": float(conv.sum() / wall),
                                      "newton_steps_p50": float(np.median(it)), "newton_steps_max": int(it.max())}
    # reported mismatch against the oracle's recomputation (FP32 factor, 1e-10)
    r = state()
    dpf.dpf_nr_solve(nr, precision=dpf.FP32, tol=1e-10, max_iter=args.nr_max_iter, n_case=K, outage=od, **r)
    va, vm, mm = (r[k].cpu().numpy() for k in ("va", "vm", "max_mismatch"))
    err = 0.0
    for k in (0, K // 2, K - 1):
        Yk = grid_ybus(g.without_branch(int(outages[k])))
        f, _ = oracle.mismatch(Yk, va[k], vm[k], g.p_spec, g.q_spec, g.bus_type)
        err = max(err, abs(float(np.abs(f).max()) - float(mm[k])))
    print(json.dumps({
        "workload": "nr",
        "config": {"grid": "c3_n1_2kbus", "n_bus": int(g.n_bus), "cases": int(K), "start": "flat",
                   "max_newton_steps": args.nr_max_iter},
        "pattern": st,
        "newton": out,
        "hybrid": hyb,
        "reported_vs_oracle_mismatch_max_abs_diff": err,
        "cpu_baseline": cpu,
        "note": "Alg. 1 (DPF) converges none of these cases to 1e-6 within 1,000 iterations (workload n1)",
    }), flush=True)
    ws.free()
    nr.free()
    y.free()


def _oracle_nr_worker(ell):
    import gridgen
    import oracle
    from oracle.ybus import grid_ybus
    g = gridgen.config_grid("c3_n1_2kbus")
    Y = grid_ybus(g.without_branch(int(ell)))
    t0 = time.perf_counter()
    r = oracle.nr_solve(Y, g.p_spec, g.q_spec, g.bus_type, g.vm_set, tol=1e-10, max_iter=20)
    return time.perf_counter() - t0, bool(r["converged"])


def _oracle_nr_sample(sample, cores):
    """The oracle's NR (Alg. 2 with scipy's sparse LU) on sampled N-1 cases,
    one process per host core (spawn)."""
    import multiprocessing as mp
    t0 = time.perf_counter()
    with mp.get_context("spawn").Pool(cores) as pool:
        res = pool.map(_oracle_nr_worker, sample)
    wall = time.perf_counter() - t0
    conv = sum(c for _, c in res)
    return {"value": conv / wall, "unit": "solves/s", "cores": cores, "kind": "oracle",
            "sample": f"{len(sample)} N-1 cases, oracle NR to 1e-10 (one case per core, spawn pool, "
                      f"{wall:.1f} s wall incl. pool start)",
            "seconds_per_case_median": float(np.median([t for t, _ in res]))}

# ---------------------------------------------------------------------------
# reference arm: the CPU oracle
# ---------------------------------------------------------------------------
def _oracle_steps_worker(args):
    """One host core: its warm-up cases untimed, then its timed cases (one per
    step); returns (case-iterations, seconds, converged) of the timed ones."""
    warm, timed, budget, start = args
    for ell in warm:
        _oracle_case((ell, budget, start))
    return _oracle_cases((timed, budget, start))


def run_reference(args):
    """The oracle on the benchmark's workload: each step every host core runs
    one warm-started N-1 case (distinct, seeded) through the oracle's Alg. 1
    loop with the same settings and budget; every core runs its warm-up and
    timed steps in one call, the run's time is the slowest core's.  solves/s
    counts the converged cases."""
    import multiprocessing as mp
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    g, outages = _workload()
    cores = len(os.sched_getaffinity(0))
    per = args.warmup + args.steps
    rng = np.random.default_rng(11)
    need = cores * per
    pick = [int(c) for c in rng.choice(outages, size=need, replace=need > outages.size)]
    jobs = [(pick[c * per: c * per + args.warmup], pick[c * per + args.warmup: (c + 1) * per], args.n1_budget,
             args.n1_start) for c in range(cores)]
    with mp.get_context("spawn").Pool(cores) as pool:
        pool.map(_oracle_base_init, range(cores))  # start-up and the base case, untimed
        res = pool.map(_oracle_steps_worker, jobs)
    n_it = sum(r[0] for r in res)
    t = max(r[1] for r in res)
    conv = sum(r[2] for r in res)
    v = conv / t
    cpu = dict(value=v, unit="solves/s", cores=cores, kind="oracle",
               sample=f"per step {cores} warm-started N-1 cases (one per core, distinct, seeded) through the FP64 "
                      f"numpy/scipy oracle ({'the DC outage shift, then ' if args.n1_start == 'dc' else ''}"
                      f"Alg. 1 loop to 1e-6 p.u. or {args.n1_budget} iterations); "
                      f"{args.steps} timed steps: {conv} of {cores * args.steps} cases converged, "
                      f"{n_it} case-iterations in {t:.1f} s (slowest core)",
               case_iterations_per_s=n_it / t)
    line = {
        "impl": "reference", "metric": METRIC, "value": v, "unit": "solves/s",
        "n_gpus": int(os.environ.get("WORLD_SIZE", "1")), "steps": args.steps, "warmup": args.warmup,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": "N-1 contingency batch: 2,000-bus synthetic grid, each case warm-started from the "
                               "base case" + (" shifted by its outage's DC angle change" if args.n1_start == "dc"
                                              else "") + " (the oracle on a bounded sample of its cases per step)",
                   "n1_start": args.n1_start,
                   "solve_definition": f"Alg. 1 from the (shifted) base case's solution until FP64 max mismatch <= "
                                       f"{TOL} p.u. (counted) or {args.n1_budget} iterations (not counted)"},
        "cpu_baseline": cpu,
        "e2e": {"value": v, "unit": "solves/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line))


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10, help="timed steps (whole batched solves)")
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="n1", choices=["n1", "flat", "scaling", "uneven", "timeseries", "paramid",
                                                         "dc", "warmstart", "c1batch", "nr"],
                    help="n1: the N-1 contingency batch (the benchmark line); flat: its flat-start FP32 "
                         "iteration rate alone; scaling: node/edge sweep; "
                         "uneven: 64-grid block-diagonal batch + parameter identification; "
                         "timeseries: the 10k-bus grid over a year of hourly snapshots; "
                         "paramid: branch identification against the oracle's operating points; "
                         "dc: the DC approximation of the N-1 batch (and Alg. 1 started from it); "
                         "warmstart: iterations from flat vs warm starts on the 30-bus grid; "
                         "c1batch: solves/s to 1e-6 on a batch of 30-bus load variants; "
                         "nr: Newton-Raphson on the GPU over the N-1 batch, and the DPF-then-Newton hybrid")
    ap.add_argument("--n1-start", default="dc", choices=["dc", "base"],
                    help="N-1 start: the base case's solution shifted by the outage's DC angle change, or unshifted")
    ap.add_argument("--n1-budget", type=int, default=None,
                    help="iterations of one N-1 solve (default: 3,500 with the DC shift, 4,000 without)")
    ap.add_argument("--profile-steps", type=int, default=100)
    ap.add_argument("--flat-iters", type=int, default=2000, help="timed flat-start FP32 iterations (sub-record)")
    ap.add_argument("--uneven-iters", type=int, default=300)
    ap.add_argument("--scaling-sizes", default="10000,100000,1000000", help="bus counts of the node sweep")
    ap.add_argument("--scaling-edges", default="5000,20000,80000", help="branches added to the 10k grid")
    ap.add_argument("--ts-hours", type=int, default=8760)
    ap.add_argument("--ts-precision", default="fp32r", choices=["fp32r", "fp32"])
    ap.add_argument("--warm-max-iter", type=int, default=50000)
    ap.add_argument("--c1-cases", type=int, default=8192)
    ap.add_argument("--nr-max-iter", type=int, default=10)
    ap.add_argument("--nr-precision", default="fp64,fp32", help="factor precisions the nr workload times")
    ap.add_argument("--pid-grids", type=int, default=16)
    ap.add_argument("--pid-steps", type=int, default=4000)
    ap.add_argument("--pid-lr", type=float, default=3e-3)
    ap.add_argument("--pid-precision", default="fp32", choices=["fp32", "fp64"])
    ap.add_argument("--pid-points", type=int, default=16, help="operating points of the identification")
    ap.add_argument("--pid-hours", default="first", choices=["first", "spread"],
                    help="candidate hours: the first 48, or 64 spread over the year")
    ap.add_argument("--uneven-pid-steps", type=int, default=10)
    ap.add_argument("--lanes", type=int, default=0)
    ap.add_argument("--warps", type=int, default=0)
    ap.add_argument("--row-blocks", type=int, default=0)
    ap.add_argument("--cpu-rounds", type=int, default=3, help="warm-started N-1 cases per host core (cpu_baseline)")
    ap.add_argument("--e2e-steps", type=int, default=2)
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-autotune", action="store_true")
    ap.add_argument("--no-plain", action="store_true")
    ap.add_argument("--no-pdl", action="store_true")
    ap.add_argument("--no-subrecords", action="store_true")
    ap.add_argument("--plain-cases", type=int, default=4)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    args = ap.parse_args()
    if args.n1_budget is None:
        args.n1_budget = n1_settings(args.n1_start)[2]
    if args.warmup < 3:
        ap.error("--warmup must be >= 3")
    if args.impl == "reference":
        run_reference(args)
    elif args.workload == "flat":
        run_flat(args)
    elif args.workload == "scaling":
        run_scaling(args)
    elif args.workload == "uneven":
        run_uneven(args)
    elif args.workload == "timeseries":
        run_timeseries(args)
    elif args.workload == "paramid":
        run_paramid(args)
    elif args.workload == "dc":
        run_dc(args)
    elif args.workload == "warmstart":
        run_warmstart(args)
    elif args.workload == "c1batch":
        run_c1batch(args)
    elif args.workload == "nr":
        run_nr(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
