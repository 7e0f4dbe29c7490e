"""Benchmark: time-to-1e-8 relative residual of the hierarchical master-slave
solver on the 1024 x 1024 triangle-lattice truss (16 x 16 sets of 64 x 64
nodes, lognormal(0, 0.3) EA, bottom row clamped, Uniform(-1, 1) loads).

A step is one whole solve from u = 0 until R1 = ||K u - p||_1 / ||p||_1 < 1e-8
(Eq. 19): every iteration runs the residual, the relaxation of every set, the
upper-level assembly and solve, all in the library's CUDA kernels.  The plain
FP64 form is the headline (`value`); the mixed form (FP32 relaxation) runs on
the same workload and is reported beside it.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

Prints one JSON line on rank 0.  With --impl reference the timed program is
the CPU oracle on the host cores (a bounded sample of iterations, scaled by
the iteration count of the method on this workload).
"""
from __future__ import annotations

import argparse
import hashlib
import json
import math
import os
import re
import statistics
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

WORKLOAD = "lattice1024_lognormal"
# arithmetic of the mixed form: FP32 relaxation, bar products of K_aa and increment of Eq. 3;
# FP64 residual, u, norms, P and the refined upper-level solution
MIXED_DTYPE = "f32 relax, K_aa products, increment / f64 residual, u, norms, master"
TOL = 1e-8
TOL_CONFIG = 1e-10  # the stopping level the 1024^2 lognormal configuration states
METRIC = f"time to R1 < {TOL:g} (Eq. 19 1-norm relative residual), plain FP64 form"


def workload_config(c):
    """The config keys both arms report for the bench workload."""
    return {"workload": WORKLOAD, "nx": c.nx, "ny": c.ny, "dofs": c.dofs, "sets": [c.sx, c.sy],
            "ea": "lognormal(0,0.3)", "loads": "Uniform(-1,1) seed 0", "tol": TOL}
MEASURED = os.path.join(ROOT, "MEASURED_PEAKS.json")
GOLDEN_FULL = os.path.join(ROOT, "tests", "golden", "lattice1024_lognormal_history.json")
FP64_LANES_PER_SM_CLK = 2  # DFMA lanes per SM per clock on GB300 (ncu: sm__sass_thread_inst_executed_op_dfma peak)


def fp64_peak_gflops(n_sm, sm_mhz):
    """FP64 roofline from the unit counts and the clock: SMs x DFMA lanes x 2 flops x clock."""
    return n_sm * FP64_LANES_PER_SM_CLK * 2 * sm_mhz * 1e-3


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-mixed", action="store_true")
    ap.add_argument("--no-force-modes", action="store_true",
                    help="skip the q = 12 solves (force-controlled modes) on the bench workload")
    ap.add_argument("--no-config-eps", action="store_true",
                    help="skip the solves to the configuration's own R1 < 1e-10")
    ap.add_argument("--ncu-case", choices=["fp64", "mixed"], default=None,
                    help="only run --ncu-iters updates of the workload once (for ncu captures); no JSON line")
    ap.add_argument("--ncu-iters", type=int, default=1)
    ap.add_argument("--batched", action="store_true",
                    help="time the batched uneven-lattice workload instead (separate JSON line)")
    ap.add_argument("--batched-count", type=int, default=256)
    ap.add_argument("--nir-sweep", action="store_true",
                    help="NIR (updates to R1 < 1e-8) versus set size at 8 x 8 sets, and versus the number "
                         "of 32 x 32-node sets (the shapes of the paper's Tests 2 and 3), FP64, 4 loadings")
    ap.add_argument("--overlap-sweep", action="store_true",
                    help="time to R1 < 1e-8 against the relaxation region's overlap instead (separate JSON line)")
    ap.add_argument("--paper-scale", action="store_true",
                    help="the 22361 x 22361-node (1.0e9 DOF) lattice: setup, time per update, kernel split")
    ap.add_argument("--paper-updates", type=int, default=8, help="updates timed by --paper-scale")
    ap.add_argument("--paper-full", action="store_true", help="with --paper-scale: also the whole solve to 1e-10")
    ap.add_argument("--no-paper-scale", action="store_true",
                    help="leave the paper-scale leg (a few updates of the 10^9-DOF lattice) out of the bench line")
    ap.add_argument("--serve", type=int, default=0, metavar="N",
                    help="serve N requests of the serving workload instead (separate JSON line)")
    ap.add_argument("--serve-max-active", type=int, default=8,
                    help="requests running at once (the rest wait in arrival order)")
    ap.add_argument("--serve-in-bench", type=int, default=24, metavar="N",
                    help="requests of the serving workload run after the timed solves (the line's `serve`; 0: none)")
    return ap.parse_args()


def case():
    from workloads import CASES
    return CASES["lattice1024_lognormal_fp64"]


def peaks():
    try:
        with open(MEASURED) as f:
            m = json.load(f)
        return float(m["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


# ---------------------------------------------------------------- algorithmic work
def dissection_entries(w, h):
    """Factor entries of the nested dissection of a w x h-node set: per tree node
    with ns unknowns of its own and nb around its box, D (ns x ns) and G (nb x
    ns) once for the way up and once, transposed, for the way down.  Boxes are
    cut by the middle column or row, those of up to 16 nodes a side by both;
    boxes of up to 2 x 2 nodes are not cut."""
    total = 0
    boxes = [(0, 0, w, h)]
    while boxes:
        x0, y0, bw, bh = boxes.pop()
        around = ((min(x0 + bw + 1, w) - max(x0 - 1, 0)) * (min(y0 + bh + 1, h) - max(y0 - 1, 0))) - bw * bh
        inner = 0
        if bw > 2 or bh > 2:
            both = bw > 2 and bh > 2 and max(bw, bh) <= 16 and bw <= 2 * bh and bh <= 2 * bw
            xs, ys = [(x0, bw)], [(y0, bh)]
            if both or bw >= bh:
                xs = [(x0, bw // 2), (x0 + bw // 2 + 1, bw - bw // 2 - 1)]
            if both or bw < bh:
                ys = [(y0, bh // 2), (y0 + bh // 2 + 1, bh - bh // 2 - 1)]
            for xa, xl in xs:
                for ya, yl in ys:
                    if xl > 0 and yl > 0:
                        boxes.append((xa, ya, xl, yl))
                        inner += xl * yl
        ns, nb = 2 * (bw * bh - inner), 2 * around
        total += ns * ns + 2 * ns * nb
    return total


def relax_work(c, fp32):
    """Per launch of the relaxation kernel: bytes the method must move (the
    factor read once, r read twice, delta written) and flops (one FMA per
    factor entry)."""
    esz = 4 if fp32 else 8
    ent = 0
    nodes = c.nx * c.ny
    for Iy in range(-(-c.ny // c.sy)):
        for Ix in range(-(-c.nx // c.sx)):
            ent += dissection_entries(min(c.sx, c.nx - Ix * c.sx), min(c.sy, c.ny - Iy * c.sy))
    return ent * esz + nodes * (32 + (8 if fp32 else 16)), 2 * ent


def residual_work(c, fp32):
    """Per launch of the update/residual kernel: u read + written, p read,
    r written, delta read, EA/L of the three owned bars, the support mask."""
    nodes = c.nx * c.ny
    return nodes * (16 * 4 + (8 if fp32 else 16) + 24 + 1), nodes * 110


# FP64 instructions per node of the update/residual kernel, each one slot of the
# FP64 pipe whatever its flops: 18 for the bar forces and r, 8 for the three norm
# terms, 8 for the upper-level update u += V a (4 in the mixed form: two
# conversions, two adds), in warps of 32 columns of which 30 are their own, and of
# 10 rows (1024^2 nodes) plus the update of the rows below and above and the
# forces of the bars from the row below.
RESIDUAL_FP64_INSTR_PER_NODE = (34 + (2 * 8 + 10) / 10) * 32 / 30
RESIDUAL_FP64_INSTR_PER_NODE_MIXED = (30 + (2 * 4 + 10) / 10) * 32 / 30


def residual_fp64_instr(fp32):
    return RESIDUAL_FP64_INSTR_PER_NODE_MIXED if fp32 else RESIDUAL_FP64_INSTR_PER_NODE


def residual_fp64_frac(c, avg_ms, n_sm, sm_mhz, fp32=False):
    """Share of the FP64 pipe's instruction slots (SMs x DFMA lanes x clock)
    the update/residual kernel's FP64 instructions fill."""
    slots = n_sm * FP64_LANES_PER_SM_CLK * sm_mhz * 1e6 * avg_ms * 1e-3
    return c.nx * c.ny * residual_fp64_instr(fp32) / slots


def src_sha(name):
    p = os.path.join(ROOT, "paper_1208_4093_gb300", "csrc", name)
    return hashlib.sha1(open(p, "rb").read()).hexdigest()[:12]


def traffic_for(kernel, workload, src):
    """DRAM bytes per launch (dram__bytes_read.sum + dram__bytes_write.sum of one
    ncu capture) from the TRAFFIC lines of the committed kernel summary, or
    None if the kernel's source changed since the capture."""
    p = os.path.join(ROOT, "profiles", "launches_update_paths.md")
    try:
        for line in open(p):
            m = re.match(r"TRAFFIC (\S+) workload=(\S+) src_sha=(\S+) bytes_per_launch=(\d+)", line.strip())
            if m and m.group(1) == kernel and m.group(2) == workload and m.group(3) == src_sha(src):
                return int(m.group(4))
    except OSError:
        pass
    return None


def max_over_ranks(x, device="cpu"):
    """The largest of x over all ranks of the default process group (the
    slowest replica sets the job's time)."""
    import torch
    import torch.distributed as dist
    v = torch.tensor([float(x)], dtype=torch.float64, device=device)
    dist.all_reduce(v, op=dist.ReduceOp.MAX)
    return float(v.item())


# ---------------------------------------------------------------- clocks
class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.proc = None
        self.gpu = gpu_index

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits", "-lms", "100",
                 "-i", str(self.gpu)], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except Exception:
            self.proc = None
        return self

    def __exit__(self, *exc):
        self.out = ""
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.out, _ = self.proc.communicate(timeout=5)
            except Exception:
                self.proc.kill()

    def summary(self):
        rows = []
        for line in (self.out or "").strip().splitlines():
            f = [x.strip() for x in line.split(",")]
            if len(f) >= 9:
                rows.append(f)
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unsampled"], "samples": 0}
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[k] for r in rows for k in range(4) if r[5 + k].lower() == "active"})
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(rows)}


# ---------------------------------------------------------------- CPU oracle sample
def oracle_update_seconds(tr, g, p, lf, iters):
    """Seconds per update of the oracle's iteration: `iters` updates (and their
    iters + 1 residuals) from u = 0, divided by iters.  The one definition both
    CPU legs use."""
    from oracle import hms
    t0 = time.perf_counter()
    hms.solve(tr, g, p, 0.0, iters, factors=lf)
    return (time.perf_counter() - t0) / iters


def oracle_sample(iters, workers=None):
    """Time `iters` oracle updates on the full workload, the per-set relaxation
    spread over `workers` host processes (all cores by default) and the dense
    algebra on the host BLAS's threads; setup untimed.  Returns (seconds per
    update, setup seconds, workers)."""
    from oracle import hms, pool, truss
    c = case()
    t0 = time.perf_counter()
    tr = truss.Truss(c.nx, c.ny, c.ea_array())
    g = hms.SetGrid(c.nx, c.ny, c.sx, c.sy)
    with pool.PoolFactors(c.nx, c.ny, c.sx, c.sy, ea=c.ea_array(), workers=workers) as lf:
        setup = time.perf_counter() - t0
        p = c.load_array().reshape(-1)
        per = oracle_update_seconds(tr, g, p, lf, iters)
        return per, setup, lf.workers


def oracle_c1_solve():
    """The oracle's whole solve of the 64 x 64 lattice (16 x 16 sets, EA = 1,
    seed-0 loads) to R1 < 1e-8, timed end to end after its setup: (ms, updates)."""
    from oracle import hms, truss
    from workloads import CASES
    c = CASES["lattice64_fp64"]
    tr = truss.Truss(c.nx, c.ny)
    g = hms.SetGrid(c.nx, c.ny, c.sx, c.sy)
    lf = hms.LocalFactors(tr, g)
    p = c.load_array().reshape(-1)
    t0 = time.perf_counter()
    res = hms.solve(tr, g, p, 1e-8, 5000, factors=lf)
    return (time.perf_counter() - t0) * 1e3, res.iterations


def err_vs_oracle(u):
    """||u - u_or|| / ||u_or|| on the 2000 DOFs the oracle's run stored at its
    convergence (R1 < 1e-10, tests/golden/, written by tests/golden/make_golden.py
    from oracle/ alone), or None without that file."""
    import numpy as np
    try:
        d = json.load(open(GOLDEN_FULL))
    except OSError:
        return None
    idx = np.array(d["sample_dofs"])
    ref = np.array(d["samples"]["final"])
    got = np.asarray(u).reshape(-1)[idx]
    return {"value": float(np.linalg.norm(got - ref) / np.linalg.norm(ref)), "dofs": int(idx.size),
            "oracle_state": "O2 at R1 < 1e-10 (%d updates)" % d["first_below_1e-10"]}


def nir_golden(tol):
    try:
        d = json.load(open(GOLDEN_FULL))
        return int(d["first_below_1e-8"] if tol == 1e-8 else d["first_below_1e-10"]), "oracle run to 1e-10"
    except Exception:
        return None, None


def host_cpu():
    """(model name, logical cores) of this host."""
    model = None
    try:
        for line in open("/proc/cpuinfo"):
            k, _, v = line.partition(":")
            if k.strip() in ("model name", "Model", "CPU part") and v.strip():
                model = model or v.strip()
    except OSError:
        pass
    import platform
    arm_parts = {"0xd4f": "Arm Neoverse V2", "0xd40": "Arm Neoverse V1", "0xd0c": "Arm Neoverse N1"}
    if model in arm_parts:
        model = f"{arm_parts[model]} (CPU part {model})"
    return model or platform.processor() or platform.machine(), os.cpu_count() or 1


def cpu_baseline_subprocess(iters):
    """The oracle as it stands on all host cores, in a child process (which
    never touches the GPU): seconds per update on the bench workload and the
    whole 64 x 64 solve."""
    code = ("import sys, json; sys.path.insert(0, %r); import bench; "
            "per, setup, w = bench.oracle_sample(%d); c1 = bench.oracle_c1_solve(); "
            "print(json.dumps([per, setup, w, c1[0], c1[1]]))" % (ROOT, iters))
    out = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=900)
    if out.returncode != 0:
        raise RuntimeError(out.stderr.strip().splitlines()[-1] if out.stderr.strip() else "oracle run failed")
    per, setup, workers, c1_ms, c1_its = json.loads(out.stdout.strip().splitlines()[-1])
    return per, setup, workers, c1_ms, c1_its


# ---------------------------------------------------------------- reference arm
def run_reference(args, rank, world):
    if rank != 0:
        return
    c = case()
    from oracle import hms, pool, truss
    tr = truss.Truss(c.nx, c.ny, c.ea_array())
    g = hms.SetGrid(c.nx, c.ny, c.sx, c.sy)
    p = c.load_array().reshape(-1)
    nir, src = nir_golden(TOL)
    model, cores = host_cpu()
    per = []
    with pool.PoolFactors(c.nx, c.ny, c.sx, c.sy, ea=c.ea_array()) as lf:
        workers = lf.workers
        for k in range(args.warmup + args.steps):
            t = oracle_update_seconds(tr, g, p, lf, 1)
            if k >= args.warmup:
                per.append(t)
    per_it = statistics.median(per)
    value = per_it * nir * 1e3 if nir else None
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": "ms",
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": value, "higher_is_better": False, "scaling": "weak", "vs_baseline": None,
            "dtype": "f64", "data": "synthetic",
            "config": dict(workload_config(c), iterations=nir, iterations_source=src,
                           parallelism=f"host: per-set relaxation over {workers} processes, BLAS threads"),
            "cpu_baseline": {"value": value, "unit": "ms", "cores": cores, "cpu": model, "kind": "oracle",
                             "sample": f"{args.steps} single-update oracle steps on the full workload "
                                       f"({per_it:.2f} s each, setup excluded) x {nir} updates, the count the "
                                       f"oracle's own run takes to R1 < {TOL:g}"},
            "e2e": {"value": value, "unit": "ms", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line))


# ---------------------------------------------------------------- profiling run
def run_ncu_case(args):
    """Setup plus --ncu-iters updates of the bench workload, untimed: the
    command the committed ncu summaries were captured with."""
    import numpy as np
    from paper_1208_4093_gb300 import capi
    c = case()
    ctx = capi.hms_context_create(0)
    prec = capi.HMS_FP64 if args.ncu_case == "fp64" else capi.HMS_MIXED
    # the relaxation at the launch shape the autotuner picks on this workload,
    # fixed so that no probe launches run
    pr = capi.hms_problem_create(ctx, c.nx, c.ny, c.sx, c.sy, ea=c.ea_array(), precision=prec, tol=0.0,
                                 max_iter=args.ncu_iters, relax_threads=256, relax_copies=1)
    p = c.load_array().reshape(1, -1)
    u = np.empty_like(p)
    capi.hms_solve(ctx, pr, p, u, allow_no_convergence=True)
    capi.hms_problem_destroy(pr)
    capi.hms_context_destroy(ctx)
    print(f"{args.ncu_case}: {args.ncu_iters} updates done")


# ---------------------------------------------------------------- batched lattices
def run_batched(args):
    """256 independent lattices (log-uniform sides 32..512, aspect up to 4,
    1-8 load vectors, 32 x 32-node sets, EA = 1, mixed precision, R1 < 1e-8):
    hms_solve_batch over one instance per load vector (clones share a
    lattice's set factors) against the lattices solved one after another."""
    import numpy as np
    import torch
    from paper_1208_4093_gb300 import capi
    from workloads import batched_lattices
    dev = torch.device("cuda", 0)
    lats = batched_lattices(args.batched_count)
    ctx = capi.hms_context_create(0)
    t0 = time.perf_counter()
    # the one-SM upper-level factor for every lattice: the lockstep engine runs
    # them all with one launch per step
    prs = [capi.hms_problem_create(ctx, l.nx, l.ny, 32, 32, precision=capi.HMS_MIXED, tol=TOL, max_iter=5000,
                                   coarse_factor=4) for l in lats]
    setup_s = time.perf_counter() - t0
    loads = [torch.from_numpy(l.load_array()).to(dev) for l in lats]
    outs = [torch.empty_like(x) for x in loads]
    nrhs = sum(l.nrhs for l in lats)
    its = torch.zeros(nrhs, dtype=torch.int32, device=dev)
    dofrhs = sum(2 * l.nx * l.ny * l.nrhs for l in lats)
    # one instance per load vector: the lattice's problem and nrhs - 1 clones sharing its set factors
    inst, inst_loads, inst_outs, clones = [], [], [], []
    for pr, l, x, o in zip(prs, lats, loads, outs):
        for q in range(l.nrhs):
            if q == 0:
                h = pr
            else:
                h = capi.hms_problem_clone(ctx, pr)
                clones.append(h)
            inst.append(h)
            inst_loads.append(x[q:q + 1])
            inst_outs.append(o[q:q + 1])
    torch.cuda.synchronize()
    for _ in range(max(args.warmup, 1)):
        capi.hms_solve_batch(ctx, inst, inst_loads, inst_outs, iters=its)
    torch.cuda.synchronize()
    ms = []
    for _ in range(args.steps):
        t0 = time.perf_counter()
        capi.hms_solve_batch(ctx, inst, inst_loads, inst_outs, iters=its)
        torch.cuda.synchronize()
        ms.append((time.perf_counter() - t0) * 1e3)
    ub = [o.cpu().numpy() for o in outs]
    # the same batch with one CUDA-graph round per problem on a pool of streams
    capi.hms_context_set_batch_mode(ctx, capi.HMS_BATCH_STREAMS)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    capi.hms_solve_batch(ctx, inst, inst_loads, inst_outs, iters=its)
    torch.cuda.synchronize()
    streams_ms = (time.perf_counter() - t0) * 1e3
    same_streams = all(np.array_equal(a, o.cpu().numpy()) for a, o in zip(ub, outs))
    capi.hms_context_set_batch_mode(ctx, capi.HMS_BATCH_AUTO)
    for h in clones:
        capi.hms_problem_destroy(h)
    # the same problems one after another (one pass)
    t0 = time.perf_counter()
    for pr, x, o in zip(prs, loads, outs):
        capi.hms_solve(ctx, pr, x, o)
    torch.cuda.synchronize()
    seq_ms = (time.perf_counter() - t0) * 1e3
    same = all(np.array_equal(a, o.cpu().numpy()) for a, o in zip(ub, outs))
    it = its.cpu().numpy()
    for pr in prs:
        capi.hms_problem_destroy(pr)
    capi.hms_context_destroy(ctx)
    med = statistics.median(ms)
    print(json.dumps({
        "metric": "batched uneven lattices: DOF x load vectors solved per second (mixed, R1 < 1e-8)",
        "value": dofrhs / (med * 1e-3), "unit": "DOF/s", "n_gpus": 1, "steps": args.steps,
        "warmup": max(args.warmup, 1), "ms_per_step": med, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": MIXED_DTYPE, "data": "synthetic",
        "config": {"workload": f"batched_lattices_{len(lats)}", "lattices": len(lats), "load_vectors": nrhs,
                   "dof_x_rhs": dofrhs, "sides": "log-uniform [32, 512]", "aspect": "Uniform[1, 4]",
                   "sets": [32, 32], "ea": 1.0, "tol": TOL, "setup_s": setup_s,
                   "updates_median": float(np.median(it)), "updates_max": int(it.max())},
        "engine": "lockstep: one launch per step over every running problem's work items, 16 updates per graph",
        "streams_engine_ms": streams_ms, "same_as_streams_engine": same_streams,
        "sequential_ms": seq_ms, "speedup_vs_sequential": seq_ms / med, "same_as_sequential": same}))


# ---------------------------------------------------------------- NIR sweeps
def run_nir_sweep(args):
    """The number of iterations required (NIR, upper-level updates to R1 < 1e-8
    by Eq. 19) and the time per update, averaged over four random loadings
    (seeds 0-3), FP64 form, EA = 1, bottom row clamped:
      test 2 shape: 8 x 8 sets of s x s nodes, s = 8 .. 64 (DOFs per set 128 .. 8192);
      test 3 shape: 32 x 32-node sets, 2 .. 1024 sets.
    The paper's own sweeps (Figs. 6-7: up to 980 000 DOFs per set, 2 .. 2000
    sets) are printed without values, so only the shapes compare."""
    import numpy as np
    from paper_1208_4093_gb300 import capi
    from workloads import loads
    ctx = capi.hms_context_create(0)

    def nir(nx, ny, sx, sy):
        pr = capi.hms_problem_create(ctx, nx, ny, sx, sy, precision=capi.HMS_FP64, tol=TOL, max_iter=20000)
        its, ms = [], []
        try:
            for seed in range(4):
                p = loads(nx, ny, seed).reshape(1, -1)
                u = np.empty_like(p)
                it = np.zeros(1, np.int32)
                t0 = time.perf_counter()
                capi.hms_solve(ctx, pr, p, u, iters=it)
                ms.append((time.perf_counter() - t0) * 1e3)
                its.append(int(it[0]))
        finally:
            capi.hms_problem_destroy(pr)
        return {"nx": nx, "ny": ny, "set": [sx, sy], "sets": -(-nx // sx) * -(-ny // sy),
                "dofs_per_set": 2 * sx * sy, "dofs": 2 * nx * ny, "nir": its, "nir_mean": float(np.mean(its)),
                "ms_per_update": float(np.sum(ms) / max(1, np.sum(its)))}

    test2 = [nir(8 * s, 8 * s, s, s) for s in (8, 12, 16, 24, 32, 48, 64)]
    test3 = [nir(32 * mx, 32 * my, 32, 32) for mx, my in ((1, 2), (2, 2), (2, 4), (4, 4), (4, 8), (8, 8), (8, 16),
                                                           (16, 16), (16, 32), (20, 50))]
    capi.hms_context_destroy(ctx)
    print(json.dumps({"metric": "NIR to R1 < 1e-8 (FP64 form, mean of 4 loadings)", "unit": "updates",
                      "test2_fixed_sets_8x8": test2, "test3_sets_of_32x32": test3}))


def run_overlap_sweep(args):
    """Extended relaxation regions (Sec. 2.2): a 512 x 1024-node lognormal
    lattice with 32 x 32-node sets (16 x 32 sets, the widest set grid the
    upper-level band factor takes at this set size), each set relaxed over its
    tile grown by e nodes, e = 0 .. 16; updates to R1 < 1e-8, setup (factoring
    the regions) and the time of one whole solve after a warm-up solve (CUDA
    events on the context stream), per form.  A larger region needs fewer
    updates but each relaxation does more work (Sec. 2.2)."""
    import numpy as np
    import torch
    from paper_1208_4093_gb300 import capi
    from workloads import ea_lognormal, loads
    nx, ny = 512, 1024
    ea = ea_lognormal(nx, ny, 1000)
    ctx = capi.hms_context_create(0)
    stream = torch.cuda.ExternalStream(capi.hms_context_stream(ctx), device=torch.device("cuda", 0))
    p = torch.from_numpy(loads(nx, ny, 0).reshape(1, -1)).cuda()
    u = torch.empty_like(p)
    its = torch.zeros(1, dtype=torch.int32, device="cuda")
    rows = []
    for prec, name in ((capi.HMS_FP64, "fp64"), (capi.HMS_MIXED, "mixed")):
        for e in (0, 1, 2, 4, 8, 16):
            pr = capi.hms_problem_create(ctx, nx, ny, 32, 32, ea=ea, precision=prec, tol=TOL,
                                         max_iter=5000, relax_overlap=e)
            try:
                setup = capi.hms_problem_setup_ms(pr)
                capi.hms_solve(ctx, pr, p, u, iters=its)
                torch.cuda.synchronize()
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record(stream)
                capi.hms_solve(ctx, pr, p, u, iters=its)
                b.record(stream)
                torch.cuda.synchronize()
                ms, nir = a.elapsed_time(b), int(its.item())
                rows.append({"form": name, "overlap": e, "updates": nir, "ms": ms, "ms_per_update": ms / max(nir, 1),
                             "setup_ms": setup, "device_bytes": capi.hms_problem_device_bytes(pr)})
            finally:
                capi.hms_problem_destroy(pr)
    # the 1024^2 lognormal workload's own 64 x 64-node sets: regions up to 80
    # nodes wide, which the mixed path's FP32 factors take
    from workloads import CASES
    c = CASES["lattice1024_lognormal_fp64"]
    p2 = torch.from_numpy(c.load_array().reshape(1, -1)).cuda()
    u2 = torch.empty_like(p2)
    rows1024 = []
    for e in (0, 2, 4, 8):
        pr = capi.hms_problem_create(ctx, c.nx, c.ny, c.sx, c.sy, ea=c.ea_array(), precision=capi.HMS_MIXED,
                                     tol=TOL, max_iter=5000, relax_overlap=e)
        try:
            setup = capi.hms_problem_setup_ms(pr)
            capi.hms_solve(ctx, pr, p2, u2, iters=its)
            torch.cuda.synchronize()
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(stream)
            capi.hms_solve(ctx, pr, p2, u2, iters=its)
            b.record(stream)
            torch.cuda.synchronize()
            ms, nir = a.elapsed_time(b), int(its.item())
            rows1024.append({"form": "mixed", "overlap": e, "updates": nir, "ms": ms,
                             "ms_per_update": ms / max(nir, 1), "setup_ms": setup,
                             "device_bytes": capi.hms_problem_device_bytes(pr),
                             "err_vs_oracle_sampled": err_vs_oracle(u2.cpu().numpy())})
        finally:
            capi.hms_problem_destroy(pr)
    capi.hms_context_destroy(ctx)
    print(json.dumps({"metric": "time to R1 < 1e-8 against the relaxation region's overlap", "unit": "ms",
                      "lattice1024_lognormal_mixed": rows1024,
                      "config": {"workload": "lattice512x1024_lognormal, 32 x 32-node sets", "nx": nx, "ny": ny,
                                 "sets": [32, 32], "ea": "lognormal(0,0.3)", "loads": "Uniform(-1,1) seed 0",
                                 "tol": TOL},
                      "rows": rows}))


# ---------------------------------------------------------------- paper scale
def paper_scale_measure(updates, full=False, split=True):
    """The paper's largest test (Sec. 3.2, Test 1: about 10^9 DOFs): a 22361 x
    22361-node lattice, EA = 1, bottom row clamped, loads Uniform(-1, 1) (seed
    0, drawn on the device by the same Philox recipe as every other workload),
    350 x 350 sets of 64 x 64 nodes (the last row and column 25 wide), mixed
    precision, the sets' factors shared by class (class_factors = 1), the
    upper level (1.1 M unknowns) by nested dissection of the set grid.

    Returns the setup, device memory, the time per update over `updates`
    updates (CUDA events on the context stream; loads already on the device),
    R1 after them, with `split` the per-kernel split of a profiled run of 3
    updates with each kernel's HBM traffic per node against the measured copy
    rate, and with `full` the whole solve to the configuration's R1 < 1e-10."""
    import torch
    from paper_1208_4093_gb300 import capi
    from workloads import CASES, loads_torch
    c = CASES["lattice22361_mixed"]
    nn = c.nx * c.ny
    ctx = capi.hms_context_create(0)
    stream = torch.cuda.ExternalStream(capi.hms_context_stream(ctx), device=torch.device("cuda", 0))
    t0 = time.time()
    p = loads_torch(c.nx, c.ny, c.seed, device="cuda").reshape(1, -1)
    gen_s = time.time() - t0
    u = torch.empty_like(p)
    its = torch.zeros(1, dtype=torch.int32, device="cuda")
    K = updates
    out = {"metric": "time per upper-level update and to R1 < 1e-10, paper-scale lattice", "unit": "ms",
           "config": {"workload": c.name, "nx": c.nx, "ny": c.ny, "dofs": 2 * nn, "sets": [c.sx, c.sy],
                      "set_grid": [-(-c.nx // c.sx), -(-c.ny // c.sy)], "ea": "1", "supports": "bottom row clamped",
                      "loads": "Uniform(-1,1) seed 0 (Philox, drawn on the device)", "precision": "mixed",
                      "class_factors": 1, "upper_level": "nested dissection by blocks"},
           "load_generation_s": gen_s}

    def timed(pr, nupd, tol):
        hist = torch.zeros((1, nupd + 1, 3), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        capi.hms_solve(ctx, pr, p, u, hist=hist, iters=its, allow_no_convergence=True)
        b.record(stream)
        torch.cuda.synchronize()
        n = int(its.item())
        h = hist[0, :n + 1, 0].cpu().numpy()
        return a.elapsed_time(b), n, h

    # a CUDA graph of K updates: no launches of finished updates in the timed region
    pr = capi.hms_problem_create(ctx, c.nx, c.ny, c.sx, c.sy, precision=capi.HMS_MIXED, tol=0.0, max_iter=K,
                                 class_factors=1, batch=min(K, 16))
    try:
        out["setup_ms"] = capi.hms_problem_setup_ms(pr)
        out["device_bytes"] = capi.hms_problem_device_bytes(pr)
        timed(pr, K, 0.0)  # warm-up (first graph launches)
        ms, n, h = timed(pr, K, 0.0)
        out["updates_timed"] = n
        out["ms_per_update"] = ms / max(n, 1)
        out["r1_history"] = [float(x) for x in h]
    finally:
        capi.hms_problem_destroy(pr)
    # per-kernel split (profile mode: CUDA events around every kernel, no graph)
    pr = capi.hms_problem_create(ctx, c.nx, c.ny, c.sx, c.sy, precision=capi.HMS_MIXED, tol=0.0, max_iter=3,
                                 class_factors=1, profile=1) if split else None
    try:
        if pr is None:
            raise StopIteration
        capi.hms_solve(ctx, pr, p, u, iters=its, allow_no_convergence=True)
        kt = capi.hms_kernel_times(pr)
        n = max(int(its.item()), 1)
        hbm = peaks()[0]
        # algorithmic bytes per node of the per-node kernels (uniform EA: no bar array)
        bytes_per_node = {"update_residual": 16 + 16 + 8 + 16 + 16 + 1, "relax": 16 + 8 + 2 * 8,
                          "coarse_assemble": 8}
        split = {}
        for k, (tms, cnt) in kt.items():
            e = {"ms_per_update": tms / n, "ms_per_launch": tms / max(cnt, 1), "launches": cnt}
            if k in bytes_per_node and tms > 0:
                gbs = bytes_per_node[k] * nn / (tms / max(cnt, 1) * 1e-3) / 1e9
                e.update({"bytes_per_node": bytes_per_node[k], "hbm_gbs": gbs, "hbm_frac": gbs / hbm})
            split[k] = e
        out["kernel_split"] = split
        out["kernel_split_note"] = ("profile mode (CUDA events around every kernel, no graph), 3 updates (the "
                                    "residual runs once more than the updates); "
                                    "update_residual and coarse_assemble are bound by the FP64 pipe, the class "
                                    "relaxation by the FP32 pipe, the upper level by its chain of fronts")
    except StopIteration:
        pass
    finally:
        if pr is not None:
            capi.hms_problem_destroy(pr)
    if full:
        pr = capi.hms_problem_create(ctx, c.nx, c.ny, c.sx, c.sy, precision=capi.HMS_MIXED, tol=c.tol,
                                     max_iter=6000, class_factors=1)
        try:
            ms, n, h = timed(pr, 6000, c.tol)
            out["full_solve"] = {"tol": c.tol, "ms": ms, "updates": n, "r1_final": float(h[-1]),
                                 "ms_per_update": ms / max(n, 1),
                                 "dofs_per_s": 2 * nn / (ms * 1e-3)}
        finally:
            capi.hms_problem_destroy(pr)
    capi.hms_context_destroy(ctx)
    del p, u
    torch.cuda.empty_cache()
    return out


def run_paper_scale(args):
    print(json.dumps(paper_scale_measure(args.paper_updates, full=args.paper_full)))


# ---------------------------------------------------------------- serving
def serve_measure(count, max_active):
    """Requests arrive by a Poisson process (mean 200 per second) with
    log-uniform sides in [64, 2048], 1-16 load vectors, lognormal(0, 0.3) EA,
    64 x 64-node sets, mixed precision, R1 < 1e-8; the server admits them
    under a 150 GB budget and advances all admitted ones together.  Latency =
    completion time - arrival time.  Returns the summary dict."""
    import numpy as np
    from paper_1208_4093_gb300 import capi
    from workloads import serving_requests
    reqs = serving_requests(count)
    data = [(r.ea_array(), r.load_array()) for r in reqs]  # generated before the clock starts
    budget = 150 << 30
    ctx = capi.hms_context_create(0)
    srv = capi.hms_server_create(ctx, budget, max_active=max_active)
    rid_of, arrival, done_t, peak_bytes, steps, rejected = {}, {}, {}, 0, 0, []
    t0 = time.perf_counter()
    nxt = 0
    while len(done_t) + len(rejected) < len(reqs):
        now = time.perf_counter() - t0
        while nxt < len(reqs) and reqs[nxt].arrival <= now:
            r = reqs[nxt]
            ea, ld = data[nxt]
            try:
                rid = capi.hms_server_submit(ctx, srv, r.nx, r.ny, 64, 64, ld, ea=ea, precision=capi.HMS_MIXED,
                                             tol=TOL, max_iter=5000)
                rid_of[rid] = nxt
                arrival[rid] = r.arrival
            except capi.HmsError:
                rejected.append(nxt)
            nxt += 1
        ids, na, nq, used = capi.hms_server_step(ctx, srv)
        steps += 1
        peak_bytes = max(peak_bytes, used)
        t_now = time.perf_counter() - t0
        for rid in ids:
            done_t[rid] = t_now
        if na == 0 and nq == 0 and nxt < len(reqs):
            time.sleep(max(0.0, reqs[nxt].arrival - (time.perf_counter() - t0)))
    makespan = time.perf_counter() - t0
    status = [capi.hms_server_take(ctx, srv, rid) for rid in list(done_t)]
    capi.hms_server_destroy(srv)
    capi.hms_context_destroy(ctx)
    lat = np.array([done_t[rid] - arrival[rid] for rid in done_t]) * 1e3
    dofrhs = sum(2 * r.nx * r.ny * r.nrhs for k, r in enumerate(reqs) if k not in rejected)
    return {"requests": len(reqs), "arrival_rate_per_s": 200.0, "arrivals_span_s": reqs[-1].arrival,
            "sides": "nx, ny log-uniform [64, 2048]", "nrhs": "1-16", "ea": "lognormal(0,0.3)", "sets": [64, 64],
            "tol": TOL, "dtype": MIXED_DTYPE, "hbm_budget_bytes": budget,
            "max_active_requests": max_active, "widest_nx": max(r.nx for r in reqs),
            "p50_ms": float(np.percentile(lat, 50)), "p99_ms": float(np.percentile(lat, 99)),
            "mean_ms": float(lat.mean()), "makespan_s": makespan, "dof_x_rhs": dofrhs,
            "dof_per_s": dofrhs / makespan, "peak_bytes_in_use": peak_bytes, "scheduler_steps": steps,
            "statuses_ok": int(sum(1 for s in status if s == capi.HMS_OK)), "rejected": len(rejected)}


def run_serve(args):
    """The serving workload alone (--serve N): one JSON line."""
    d = serve_measure(args.serve, args.serve_max_active)
    print(json.dumps({
        "metric": "serving: p50 / p99 request latency and DOF x load vectors per second (mixed, R1 < 1e-8)",
        "value": d["p50_ms"], "unit": "ms (p50 latency)", "n_gpus": 1, "steps": d["scheduler_steps"],
        "warmup": 0, "ms_per_step": d["makespan_s"] * 1e3 / max(d["scheduler_steps"], 1),
        "higher_is_better": False, "scaling": "weak", "vs_baseline": None, "dtype": d["dtype"],
        "data": "synthetic", "config": {"workload": f"serving_{d['requests']}", **d}}))


# ---------------------------------------------------------------- our arm
def run_ours(args, rank, world, local_rank):
    import numpy as np
    import torch
    from paper_1208_4093_gb300 import capi

    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    c = case()
    ea = c.ea_array()
    nd = c.dofs
    p_host = c.load_array().reshape(1, -1)
    ctx = capi.hms_context_create(local_rank)
    stream = torch.cuda.ExternalStream(capi.hms_context_stream(ctx), device=dev)

    def make(prec, profile=0, tol=TOL):
        return capi.hms_problem_create(ctx, c.nx, c.ny, c.sx, c.sy, ea=ea, precision=prec, tol=tol,
                                       max_iter=5000, profile=profile)

    p_dev = torch.from_numpy(p_host).to(dev)
    u_dev = torch.empty_like(p_dev)
    its = torch.zeros(1, dtype=torch.int32, device=dev)

    def timed(pr, steps, warmup, clocks=False):
        for _ in range(warmup):
            capi.hms_solve(ctx, pr, p_dev, u_dev, iters=its)
        torch.cuda.synchronize()
        if world > 1:
            torch.distributed.barrier()
        ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(steps)]
        sampler = ClockSampler(local_rank)
        if clocks:
            sampler.__enter__()
            time.sleep(0.3)
        torch.cuda.synchronize()
        for k in range(steps):
            ev[k][0].record(stream)
            capi.hms_solve(ctx, pr, p_dev, u_dev, iters=its)
            ev[k][1].record(stream)
        torch.cuda.synchronize()
        if clocks:
            sampler.__exit__(None, None, None)
        if world > 1:
            torch.distributed.barrier()
        ms = [a.elapsed_time(b) for a, b in ev]
        return ms, (sampler.summary() if clocks else None)

    # ---- plain FP64 form (headline) ----
    pr64 = make(capi.HMS_FP64)
    setup64 = capi.hms_problem_setup_ms(pr64)
    ms64, clocks = timed(pr64, args.steps, args.warmup, clocks=True)
    nit64 = int(its.item())
    cap_hits64 = capi.hms_problem_refine_cap_hits(pr64)
    shape64 = {"threads": capi.hms_problem_relax_threads(pr64), "copies": capi.hms_problem_relax_copies(pr64)}
    u64 = u_dev.cpu().numpy().copy()
    # the error of the timed solve, against the same lattice solved far past the
    # metric's tolerance (R1 < 1e-12); tests/test_gpu_fullsize.py compares such
    # solves with the oracle's direct solve over every DOF
    prt = make(capi.HMS_FP64, tol=1e-12)
    capi.hms_solve(ctx, prt, p_dev, u_dev, iters=its)
    tight_its = int(its.item())
    u_tight = u_dev.cpu().numpy().copy()
    capi.hms_problem_destroy(prt)
    err_tight = float(np.linalg.norm(u64 - u_tight) / np.linalg.norm(u_tight))
    # e2e through host buffers (pinned): H2D of the loads and D2H of u inside the timed region
    p_pin = torch.from_numpy(p_host).pin_memory()
    u_pin = torch.empty_like(p_pin).pin_memory()
    e2e = []
    for k in range(args.warmup + args.steps):
        t0 = time.perf_counter()
        capi.hms_solve(ctx, pr64, p_pin, u_pin)
        if k >= args.warmup:
            e2e.append((time.perf_counter() - t0) * 1e3)
    capi.hms_problem_destroy(pr64)

    # ---- mixed form on the same workload ----
    mixed = None
    if not args.no_mixed:
        prm = make(capi.HMS_MIXED)
        setupm = capi.hms_problem_setup_ms(prm)
        msm, _ = timed(prm, args.steps, args.warmup)
        nitm = int(its.item())
        shapem = {"threads": capi.hms_problem_relax_threads(prm), "copies": capi.hms_problem_relax_copies(prm)}
        um = u_dev.cpu().numpy()
        capi.hms_problem_destroy(prm)
        mixed = {"value": statistics.median(msm), "unit": "ms", "iterations": nitm, "setup_ms": setupm,
                 "dtype": MIXED_DTYPE, "relax_launch": shapem,
                 "rel_diff_vs_fp64": float(np.linalg.norm(um - u64) / np.linalg.norm(u64)),
                 "err_vs_oracle_sampled": err_vs_oracle(um),
                 "speedup_vs_fp64": statistics.median(ms64) / statistics.median(msm)}

    # ---- the configuration's own stopping level (R1 < 1e-10), both forms ----
    # The oracle's stored state is at the same level (its run to 1e-10), so the
    # sampled error here compares like with like.
    config_eps = None
    if not args.no_config_eps:
        config_eps = {"tol": TOL_CONFIG}
        for prec, name in ((capi.HMS_FP64, "fp64"), (capi.HMS_MIXED, "mixed")):
            if name == "mixed" and args.no_mixed:
                continue
            pre = make(prec, tol=TOL_CONFIG)
            mse, _ = timed(pre, 2, 1)
            config_eps[name] = {"value": statistics.median(mse), "unit": "ms", "iterations": int(its.item()),
                                "err_vs_oracle_sampled": err_vs_oracle(u_dev.cpu().numpy())}
            capi.hms_problem_destroy(pre)
        nor, _ = nir_golden(TOL_CONFIG)
        config_eps["oracle_iterations"] = nor

    # ---- the force-controlled modes (q = 12, Eqs. 15-18) on the same workload ----
    force_modes = None
    if not args.no_force_modes:
        force_modes = {"tol": TOL, "what": "q = 12 (mode_mask 0xFFF: modes 10-12 of the force-controlled "
                                           "relaxation added) against the q = 9 solves above"}
        for prec, name in ((capi.HMS_FP64, "fp64"), (capi.HMS_MIXED, "mixed")):
            if name == "mixed" and args.no_mixed:
                continue
            prf = capi.hms_problem_create(ctx, c.nx, c.ny, c.sx, c.sy, ea=ea, precision=prec, tol=TOL,
                                          max_iter=5000, mode_mask=0xFFF)
            msf, _ = timed(prf, 1, 1)
            force_modes[name] = {"value": msf[0], "unit": "ms", "iterations": int(its.item()),
                                 "setup_ms": capi.hms_problem_setup_ms(prf),
                                 "device_bytes": capi.hms_problem_device_bytes(prf)}
            capi.hms_problem_destroy(prf)
        force_modes["q9"] = {"fp64": {"value": statistics.median(ms64), "iterations": nit64},
                             "mixed": ({"value": mixed["value"], "iterations": mixed["iterations"]}
                                       if mixed else None)}

    # ---- the 64 x 64 lattice (16 x 16-node sets, EA = 1), FP64, to R1 < 1e-8 ----
    from workloads import CASES
    c1 = CASES["lattice64_fp64"]
    pr1 = capi.hms_problem_create(ctx, c1.nx, c1.ny, c1.sx, c1.sy, precision=capi.HMS_FP64, tol=1e-8,
                                  max_iter=5000)
    p1 = torch.from_numpy(c1.load_array().reshape(1, -1)).to(dev)
    u1 = torch.empty_like(p1)
    for _ in range(2):
        capi.hms_solve(ctx, pr1, p1, u1, iters=its)
    c1_ms = []
    for _ in range(5):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        capi.hms_solve(ctx, pr1, p1, u1, iters=its)
        e1.record(stream)
        torch.cuda.synchronize()
        c1_ms.append(e0.elapsed_time(e1))
    c1_gpu = {"value": statistics.median(c1_ms), "unit": "ms", "iterations": int(its.item())}
    capi.hms_problem_destroy(pr1)

    # ---- per-kernel CUDA-event times (profile pass, same workload) ----
    hbm_peak, peak_src = peaks()
    try:
        fp64_probe = capi.hms_measure_fp64_rate(local_rank)
    except capi.HmsError:
        fp64_probe = None
    rooflines = {}
    for prec, name in ((capi.HMS_FP64, "fp64"), (capi.HMS_MIXED, "mixed")):
        if name == "mixed" and args.no_mixed:
            continue
        prp = make(prec, profile=1)
        capi.hms_solve(ctx, prp, p_dev, u_dev, iters=its)
        kt = capi.hms_kernel_times(prp)
        capi.hms_problem_destroy(prp)
        fp32 = prec == capi.HMS_MIXED
        kname = "k_rtree<{}>".format("float" if fp32 else "double")
        ms, n = kt["relax"]
        b, fl = relax_work(c, fp32)
        avg = ms / max(n, 1)
        if fp32:
            ach = b / (avg * 1e-3) / 1e9
            roof = {"kernel": kname, "bound": "hbm", "achieved": ach, "peak": hbm_peak,
                    "unit": "GB/s", "frac": ach / hbm_peak, "peak_source": peak_src}
        else:
            ach = fl / (avg * 1e-3) / 1e9
            n_sm = torch.cuda.get_device_properties(dev).multi_processor_count
            mhz = (clocks or {}).get("sm_max_mhz") or 2070.0
            pk = fp64_peak_gflops(n_sm, mhz)
            roof = {"kernel": kname, "bound": "alu", "achieved": ach, "peak": pk,
                    "unit": "GFLOP/s", "frac": ach / pk,
                    "peak_source": f"FP64 units: {n_sm} SMs x {FP64_LANES_PER_SM_CLK} DFMA lanes/clock x 2 flops x "
                                   f"{mhz:.0f} MHz",
                    "peak_measured_fma_loop": fp64_probe,
                    "frac_of_measured_fma_loop": (ach / fp64_probe) if fp64_probe else None,
                    "hbm_gbs": b / (avg * 1e-3) / 1e9, "hbm_frac": b / (avg * 1e-3) / 1e9 / hbm_peak}
        roof.update({"algorithmic_bytes": b, "algorithmic_flops": fl, "avg_launch_ms": avg, "launches": n,
                     "avg_launch_ms_source": "profile pass: one solve of the same workload with options.profile "
                                             "= 1 (CUDA events on the context stream around every kernel)",
                     "traffic": traffic_for(roof["kernel"], WORKLOAD, "relax_tree.cu")})
        rb, _ = residual_work(c, fp32)
        rms, rn = kt["update_residual"]
        ravg = rms / max(rn, 1)
        n_sm1 = torch.cuda.get_device_properties(dev).multi_processor_count
        mhz1 = (clocks or {}).get("sm_max_mhz") or 2070.0
        roof["update_residual"] = {"avg_launch_ms": ravg, "hbm_gbs": rb / (ravg * 1e-3) / 1e9,
                                   "hbm_frac": rb / (ravg * 1e-3) / 1e9 / hbm_peak,
                                   "bound": "alu (FP64 pipe)",
                                   "fp64_instr_per_node": residual_fp64_instr(fp32),
                                   "fp64_frac": residual_fp64_frac(c, ravg, n_sm1, mhz1, fp32)}
        roof["kernel_ms"] = {k: v[0] for k, v in kt.items()}
        roof["kernel_launches"] = {k: v[1] for k, v in kt.items()}
        rooflines[name] = roof

    # kernels launched per solve: graph batches of 16 iterations, each iteration
    # 9 kernels (residual, relaxation, assembly, the scaled system's diagonal and
    # rows, three levels of fronts, all solves), plus 1 load-norm kernel
    batches = math.ceil((nit64 + 1) / 16)
    per_iter = 9
    launches = args.steps * (batches * 16 * per_iter + 1)

    # ---- serving (continuous batching under the HBM budget), a bounded run ----
    serve = None
    if args.serve_in_bench > 0 and world == 1:
        serve = serve_measure(args.serve_in_bench, args.serve_max_active)

    # ---- the paper-scale lattice (10^9 DOFs): setup and time per update ----
    paper = None
    if not args.no_paper_scale and world == 1:
        try:
            paper = paper_scale_measure(4)
            paper.pop("metric", None)
            paper["full_solve_note"] = ("the whole solve to R1 < 1e-10 is `bench.py --paper-scale --paper-full` "
                                        "(minutes; not part of the default line)")
        except Exception as e:  # e.g. a device with less memory
            paper = {"skipped": str(e)}

    ms_med = statistics.median(ms64)
    if world > 1:
        ms_med = max_over_ranks(max(ms64), dev)
    if rank != 0:
        capi.hms_context_destroy(ctx)
        return
    cpu = None
    if not args.no_cpu_baseline and world == 1:
        try:
            per_it, setup_s, workers, c1_ms_or, c1_its_or = cpu_baseline_subprocess(3)
            nir = nit64
            model, cores = host_cpu()
            cpu = {"value": per_it * nir * 1e3, "unit": "ms", "cores": cores, "cpu": model, "kind": "oracle",
                   "sample": f"3 oracle updates on the full workload ({per_it:.2f} s per update: the per-set "
                             f"relaxation over {workers} host processes, dense algebra on the host BLAS's "
                             f"threads; setup {setup_s:.1f} s excluded), times the {nir} updates the FP64 "
                             f"method takes here",
                   "c1_full_solve": {"value": c1_ms_or, "unit": "ms", "iterations": c1_its_or,
                                     "what": "the oracle's whole solve of the 64 x 64 lattice to R1 < 1e-8, run "
                                             "(not extrapolated), one process"}}
        except Exception as e:  # the baseline is reported, never the target
            cpu = {"value": None, "unit": "ms", "cores": os.cpu_count(), "kind": "oracle", "sample": f"failed: {e}"}
    line = {
        "metric": METRIC,
        "value": ms_med, "unit": "ms", "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": ms_med, "higher_is_better": False, "scaling": "weak", "vs_baseline": None,
        "dtype": "f64", "data": "synthetic",
        "config": {**workload_config(c),
                   "iterations": nit64, "setup_ms": setup64, "relax_launch": shape64,
                   "l2": "working set > L2 (FP64 factors 2.5 GB streamed every iteration); no flush",
                   "parallelism": "replicas" if world > 1 else "single GPU"},
        "err_vs_oracle_sampled": err_vs_oracle(u64),
        "err_vs_tight_solve": {"value": err_tight, "tight_tol": 1e-12, "tight_iterations": tight_its,
                               "what": "||u - u_t|| / ||u_t|| over every DOF, u the timed R1 < 1e-8 solve, u_t the "
                                       "same lattice solved to R1 < 1e-12 (the FP64 bar 1e-9 is met at the "
                                       "configuration's own R1 < 1e-10: config_eps)"},
        "refine_cap_hits_per_solve": cap_hits64,
        "c1_lattice64": {"gpu": c1_gpu, "oracle": (cpu or {}).get("c1_full_solve")},
        "mixed": mixed,
        "config_eps": config_eps,
        "roofline": rooflines.get("fp64"),
        "roofline_mixed": rooflines.get("mixed"),
        "cpu_baseline": cpu,
        "e2e": {"value": statistics.median(e2e), "unit": "ms", "h2d_bytes_per_step": 8 * nd,
                "d2h_bytes_per_step": 8 * nd},
        "serve": serve,
        "paper_scale": paper,
        "force_modes": force_modes,
        "gpu_launches": launches,
        "clocks": clocks,
        "dofs_per_s": world * nd / (ms_med * 1e-3),
    }
    print(json.dumps(line))
    capi.hms_context_destroy(ctx)


def main():
    args = parse()
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch
        import torch.distributed as dist
        backend = "nccl" if args.impl == "ours" else "gloo"
        if args.impl == "ours":
            torch.cuda.set_device(local_rank)
        dist.init_process_group(backend)
    try:
        if args.ncu_case:
            run_ncu_case(args)
        elif args.batched:
            run_batched(args)
        elif args.nir_sweep:
            run_nir_sweep(args)
        elif args.overlap_sweep:
            run_overlap_sweep(args)
        elif args.paper_scale:
            run_paper_scale(args)
        elif args.serve:
            run_serve(args)
        elif args.impl == "reference":
            run_reference(args, rank, world)
        else:
            run_ours(args, rank, world, local_rank)
    finally:
        if world > 1:
            import torch.distributed as dist
            dist.destroy_process_group()


if __name__ == "__main__":
    main()
