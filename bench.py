#!/usr/bin/env python3
"""Throughput of the batched CMA-ES generation loop on GB300.

Workload (default, `batch256`): 256 concurrent IPOP-CMA-ES searches of uneven
size in one batch: n drawn from {50, 200, 500, 1000, 2000}, lambda = (4 +
floor(3 ln n)) 2^k with k drawn from 0..8, objectives alternating between a
rotated ellipsoid (cond 1e6) and a rotated Rastrigin; every search restarts at
its own population size when a stop test fires (the K-Distributed layout of
§3.2.3, where all population levels run side by side). One step = one
generation of every search = 264,864 candidates sampled, evaluated and used in
the update (rank, recombination, paths, step size, rank-one + rank-mu
covariance update), plus the lazy FP64 eigendecomposition where due and the
stop tests. Inputs are seeded synthetic instances (no BBOB data).

Prints one JSON line (rank 0). Timing: W warm-up generations, then K timed
generations, each bracketed by CUDA events on the launch stream, with a
256 MiB write between timed generations to flush L2. The per-phase and
per-kernel-stage device times come from a separate profiled handle that runs
the same generations (the timed handle runs without profiling); `e2e` is a
third handle, again over the same generations, timed on the host through the
public API (cmaes_step_batch, then every search's best point and value read
back with cmaes_best), with the same L2 flush between steps (outside the
timed region).

--impl reference times the FP64 CPU oracle on this host's cores on the same
workload (test infrastructure; it is the method's plain restatement).
"""
import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "candidates/sec sampled+evaluated+updated; mixed vs plain FP64 GPU; % roofline"
UNIT = "candidates/s"
SEED = 20240918
WORKLOADS = ("batch256", "batch32", "rastrigin-n100-kdist", "ellipsoid-n1000", "ellipsoid-n4096",
             "ellipsoid-n10", "rastrigin-n100-ipop")


def parse_args():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["engine", "reference"], default="engine")
    ap.add_argument("--workload", choices=WORKLOADS, default="batch256")
    ap.add_argument("--precision", choices=["fp64", "tf32", "bf16"], default="tf32",
                    help="headline path; the plain FP64 path is measured beside it")
    ap.add_argument("--paths", default="fp64",
                    help="comma-separated other precisions measured beside the headline ('' for none)")
    ap.add_argument("--eig-method", choices=["auto", "jacobi", "tridiagonal"], default="auto")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-extra", action="store_true",
                    help="skip the extra n = 100 K-Distributed line")
    ap.add_argument("--cpu-seconds", type=float, default=15.0)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    return ap.parse_args()


def dist_env():
    from paper_2409_11765_gb300 import dist as D
    return D.env()


def workload(name):
    from paper_2409_11765_gb300 import workloads as W
    if name == "batch256":
        return W.batch256()
    if name == "batch32":
        return W.batch32()
    if name == "rastrigin-n100-kdist":
        return W.rastrigin_n100_ipop(concurrent=True)
    if name == "rastrigin-n100-ipop":
        return W.rastrigin_n100_ipop(concurrent=False)
    if name == "ellipsoid-n1000":
        return W.ellipsoid_n1000()
    if name == "ellipsoid-n4096":
        return W.ellipsoid_n4096()
    return W.ellipsoid_n10()


def workload_config(wl, precision, eig_method):
    ns = sorted({s.n for s in wl.searches})
    kinds = sorted({s.problem.kind for s in wl.searches})
    names = {1: "rotated ellipsoid", 2: "rotated Rastrigin", 3: "sphere"}
    return {"workload": wl.name, "searches": len(wl.searches), "n": ns,
            "lambda_min": min(s.lam for s in wl.searches),
            "lambda_max": max(s.lam for s in wl.searches),
            "candidates_per_step": wl.candidates_per_generation,
            "objectives": [names[k] for k in kinds],
            "restarts": "each search at its own lambda" if not wl.ipop_double else "lambda doubled",
            "precision": precision,
            "gemms": {"fp64": "FP64 CUDA cores",
                      "tf32": "tcgen05 kind::tf32 (objective, rank-mu: 3-term split)",
                      "bf16": "tcgen05 kind::f16 bf16 (objective, rank-mu: 3-term split)"}[precision],
            "eig": "FP64, lazy cadence; " + {0: "tridiagonal route above n = 160, Jacobi route below",
                                            1: "warm-started Jacobi route",
                                            2: "Householder tridiagonal route"}[eig_method],
            "l2": "256 MiB write between timed generations", "seed": SEED}


# ----------------------------- CPU oracle ----------------------------------
def oracle_searches(wl):
    from oracle import cmaes
    sts, probs = [], []
    for s in wl.searches:
        sts.append(cmaes.State(s.n, s.lam, s.sigma0, s.x0.copy(), s.sigma0))
        p = s.problem
        probs.append(cmaes.Problem(p.kind, p.xstar, p.Q, p.lamdiag))
    opts = cmaes.Options(f_target=wl.f_target, box_lo=wl.box_lo, box_hi=wl.box_hi,
                         max_restarts=wl.max_restarts if wl.max_restarts < 255 else 10 ** 9,
                         ipop_double=wl.ipop_double)
    return sts, probs, opts


def oracle_sample(wl, seconds):
    """The oracle as it stands on this host's cores: generations of the batch's
    searches in order (search by search) until `seconds` have passed.
    Returns (candidates, searches done, generations, elapsed)."""
    from oracle import cmaes
    sts, probs, opts = oracle_searches(wl)
    t0 = time.perf_counter()
    cand = 0
    gens = 0
    done_searches = 0
    while True:
        for i, (st, pr) in enumerate(zip(sts, probs)):
            if not st.done:
                cand += st.lam
                cmaes.generation(st, SEED, i, pr, opts)
            if gens == 0:
                done_searches = i + 1
            if time.perf_counter() - t0 >= seconds:
                return cand, done_searches, gens + (1 if done_searches == len(sts) else 0), \
                    time.perf_counter() - t0
        gens += 1


def cpu_baseline(wl, seconds):
    cand, ns, gens, el = oracle_sample(wl, seconds)
    return {"value": cand / el, "unit": UNIT, "cores": os.cpu_count(), "kind": "oracle",
            "sample": "%d candidates of the batch's first generations in %.1f s (%d of %d searches "
                      "of generation 0 done%s); numpy FP64, BLAS threads = host cores"
                      % (cand, el, ns, len(wl.searches),
                         ", %d full generations" % gens if gens else "")}


def run_reference(args):
    rank, _, world = dist_env()
    if rank != 0:
        return
    wl = workload(args.workload)
    per_step = max(args.cpu_seconds / max(args.steps, 1), 1.0)
    times, cands = [], []
    for _ in range(args.steps):
        cand, _, _, el = oracle_sample(wl, per_step)
        times.append(el)
        cands.append(cand)
    value = sum(cands) / sum(times)
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": 0,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * sum(times) / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": workload_config(wl, "fp64", 0),
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": os.cpu_count(),
                             "kind": "oracle",
                             "sample": "each step: the batch's searches in order for %.1f s "
                                       "(%d candidates per step on average)"
                                       % (per_step, sum(cands) // max(len(cands), 1))},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


# ------------------------------- clocks -------------------------------------
class ClockSampler:
    QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.f = tempfile.NamedTemporaryFile("w+", suffix=".csv", delete=False)
        try:
            self.p = subprocess.Popen(["nvidia-smi", "-i", str(gpu_index),
                                       "--query-gpu=" + self.QUERY, "--format=csv,noheader,nounits",
                                       "-lms", "200"], stdout=self.f, stderr=subprocess.DEVNULL)
        except OSError:
            self.p = None

    def stop(self):
        if self.p is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.p.terminate()
        try:
            self.p.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.p.kill()
        self.f.flush()
        self.f.seek(0)
        rows = [r.split(",") for r in self.f.read().strip().splitlines() if r.strip()]
        os.unlink(self.f.name)
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for r in rows:
            r = [x.strip() for x in r]
            if len(r) < 9:
                continue
            try:
                sm.append(float(r[1]))
                smax.append(float(r[2]))
            except ValueError:
                continue
            for nm, v in zip(names, r[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(smax) if smax else None, "reasons": sorted(reasons),
                "samples": len(sm)}


# ------------------------------ GPU engine ----------------------------------
PREC = {"fp64": 0, "tf32": 1, "bf16": 2}
DTYPE = {"fp64": "f64", "tf32": "tf32+f64", "bf16": "bf16+f64"}

# DRAM bytes per step of the dominant stage from one ncu capture, valid only
# for the sources of that stage's kernels as they were measured (a SHA-256 of
# the code without comments, stage_sources_sha): after any change to them the
# roofline's traffic is null until it is measured again.
#   reduction: dram__bytes_read.sum + dram__bytes_write.sum of the six launches of
#   k_trd_reduce a generation of the 256-search batch has (one pass each), the mean
#   of the ten timed generations of two handles.
KERNEL_TRAFFIC = {
    "reduction": {"bytes_per_step": 1.878e12, "workload": "batch256-n50..2000", "sources_sha256_16": "1de10db170175c3d"},
}

# The code each stage's kernels are built from: the reduction's source up to
# its host part (its kernel and every helper it calls) and the headers it
# includes.
STAGE_SOURCES = {
    "reduction": {"prefix": ("kernels_eig_trd_reduce.cu", "using RedFn ="),
                  "headers": ("device_common.cuh", "ozaki.cuh", "trd_common.cuh", "engine.h")},
}


def _strip_comments(text):
    """The code without comments and blank lines (string and character
    literals kept whole, so that "//" inside them is not a comment)."""
    import re
    token = re.compile(r'"(?:\\.|[^"\\\n])*"|\'(?:\\.|[^\'\\\n])*\'|//[^\n]*|/\*.*?\*/', re.S)
    code = token.sub(lambda m: m.group(0) if m.group(0)[0] in "\"'" else " ", text)
    lines = [ln.rstrip() for ln in code.splitlines()]
    return "\n".join(ln for ln in lines if ln.strip())


def stage_sources_sha(stage):
    """Hash of the code a stage's kernels are built from (STAGE_SOURCES):
    a change to it voids the recorded traffic, a change to a comment or to
    another stage's kernels does not."""
    import hashlib
    spec = STAGE_SOURCES.get(stage)
    if spec is None:
        return None
    csrc = os.path.join(ROOT, "paper_2409_11765_gb300", "csrc")
    h = hashlib.sha256()
    fname, marker = spec["prefix"]
    text = open(os.path.join(csrc, fname), encoding="utf-8").read()
    cut = text.find(marker)
    h.update(_strip_comments(text[:cut] if cut >= 0 else text).encode())
    for f in spec["headers"]:
        h.update(_strip_comments(open(os.path.join(csrc, f), encoding="utf-8").read()).encode())
    return h.hexdigest()[:16]


def make_handle(wl, prec, eig_method, rank):
    import paper_2409_11765_gb300 as eng
    from paper_2409_11765_gb300 import dist as D
    opt = eng.cmaes_default_options(precision=PREC[prec], f_target=wl.f_target,
                                    box_lo=wl.box_lo, box_hi=wl.box_hi,
                                    max_restarts=min(wl.max_restarts, 255),
                                    ipop_double=1 if wl.ipop_double else 0, eig_method=eig_method)
    h = eng.cmaes_create_batch([s.n for s in wl.searches], [s.lam for s in wl.searches],
                               [s.x0 for s in wl.searches], [s.sigma0 for s in wl.searches],
                               D.rank_seed(SEED, rank), opt)
    for i, s in enumerate(wl.searches):
        p = s.problem
        eng.cmaes_set_problem(h, i, p.kind, p.Q, p.lamdiag, p.xstar)
    return h


def decomposition_work(eng, h, wl, before):
    """Decompositions of each dimension done since `before` (cmaes_eig_stats)."""
    out = {}
    for i, s in enumerate(wl.searches):
        k = eng.cmaes_eig_stats(h, i)["decompositions"] - before[i]
        if k:
            out[s.n] = out.get(s.n, 0) + k
    return out


def measure(args, wl, prec, world, rank, dist, want_clocks, eig_method, secondary=False):
    import torch
    import paper_2409_11765_gb300 as eng
    from paper_2409_11765_gb300 import dist as D
    count = len(wl.searches)
    ns = [s.n for s in wl.searches]
    stream = torch.cuda.Stream()
    torch.cuda.set_stream(stream)
    sptr = stream.cuda_stream
    flush = torch.empty(256 * 1024 * 1024, dtype=torch.uint8, device="cuda")
    res = {}

    # 1. timed handle: device time of K generations, no profiling
    h = make_handle(wl, prec, eig_method, rank)
    try:
        for _ in range(args.warmup):
            eng.cmaes_step_batch(h, 1, sptr)
        torch.cuda.synchronize()
        before = [eng.cmaes_eig_stats(h, i)["decompositions"] for i in range(count)]
        launches0 = eng.cmaes_kernel_launches(h)
        starts = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
        ends = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
        sampler = None
        if want_clocks:
            vis = os.environ.get("CUDA_VISIBLE_DEVICES")
            local = int(os.environ.get("LOCAL_RANK", "0"))
            gpu_index = vis.split(",")[local] if vis else str(local)
            sampler = ClockSampler(gpu_index)
            time.sleep(0.3)
        if dist is not None:
            dist.barrier()
        torch.cuda.synchronize()
        for k in range(args.steps):
            flush.fill_(k & 255)
            starts[k].record(stream)
            eng.cmaes_step_batch(h, 1, sptr)
            ends[k].record(stream)
        torch.cuda.synchronize()
        if dist is not None:
            dist.barrier()
        res["clocks"] = sampler.stop() if sampler else None
        res["gpu_launches"] = int(eng.cmaes_kernel_launches(h) - launches0)
        eng.cmaes_sync(h)
        step_ms = [a.elapsed_time(b) for a, b in zip(starts, ends)]
        total_ms = D.max_over_ranks(sum(step_ms), dist, device="cuda")
        res["decompositions"] = decomposition_work(eng, h, wl, before)
    finally:
        eng.cmaes_destroy(h)
    cand = wl.candidates_per_generation
    res["value"] = D.whole_job_rate(cand, args.steps, world, total_ms)
    res["ms_per_step"] = total_ms / args.steps
    res["step_ms"] = step_ms

    if secondary:  # a path measured beside the headline: device time only
        torch.cuda.set_stream(torch.cuda.default_stream())
        del flush
        torch.cuda.empty_cache()
        return res
    # 2. profiled handle: the same generations with per-phase and per-stage events
    h = make_handle(wl, prec, eig_method, rank)
    try:
        for _ in range(args.warmup):
            eng.cmaes_step_batch(h, 1, sptr)
        torch.cuda.synchronize()
        eng.cmaes_phase_times(h, reset=True)
        eng.cmaes_eig_stage_times(h, reset=True)
        eng.cmaes_set_profiling(h, True)
        for k in range(args.steps):
            flush.fill_(k & 255)
            eng.cmaes_step_batch(h, 1, sptr)
        torch.cuda.synchronize()
        phase_ms, _ = eng.cmaes_phase_times(h, reset=True)
        stage_ms = eng.cmaes_eig_stage_times(h, reset=True)
        eng.cmaes_set_profiling(h, False)
    finally:
        eng.cmaes_destroy(h)
    res["phases_ms_per_step"] = {k: v / args.steps for k, v in phase_ms.items()}
    res["eig_stages_ms_per_step"] = {k: v / args.steps for k, v in stage_ms.items()}

    # 3. e2e handle: the same generations through the public API, host-timed
    if not args.no_e2e:
        h = make_handle(wl, prec, eig_method, rank)
        try:
            for _ in range(args.warmup):
                eng.cmaes_step_batch(h, 1, sptr)
            torch.cuda.synchronize()
            el = 0.0
            for k in range(args.steps):
                flush.fill_(k & 255)
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                eng.cmaes_step_batch(h, 1, sptr)
                for i in range(count):
                    eng.cmaes_best(h, i, ns[i])
                el += time.perf_counter() - t0
        finally:
            eng.cmaes_destroy(h)
        res["e2e"] = {"value": cand * args.steps * world / el, "unit": UNIT,
                      "h2d_bytes_per_step": 0, "d2h_bytes_per_step": sum(8 * m + 8 for m in ns)}
    torch.cuda.set_stream(torch.cuda.default_stream())
    del flush
    torch.cuda.empty_cache()
    return res


def stage_flops(decomps):
    """Algorithmic FP64 flops of the eigendecompositions per stage, from the
    decompositions done. The Householder reduction has none in its steps (its
    bound is reduction_roof's). Back-transformation: 2 n^3 (dormtr's count) for
    n <= 256, where it runs in FP64; above, on the tensor cores (0 FP64 flops).
    The eigenvalue and eigenvector stages are O(n^2) per decomposition and the
    Newton-Schulz orthogonalisation is not part of the minimal method (0)."""
    bt = sum(k * 2.0 * n ** 3 for n, k in decomps.items() if n <= 256)
    return {"backtransform": bt, "eigenvalues": 0.0, "eigenvectors": 0.0, "orthogonalisation": 0.0}


# 32 x 32 + 64-bit integer multiply-adds a clock and SM, measured.
IMAD_PER_CLOCK = 28.0
# What the reduction's resident CTAs hold in shared memory, bytes an SM.
REDUCTION_SMEM = 200e3


def reduction_roof(wl, decomps, steps, hbm_gbs, sms, sm_mhz):
    """The bound of the tridiagonal reduction: (bound, work per step, rate, unit).
    Each step reads and writes the whole trailing matrix and does nine integer
    multiply-adds an element, n^3 / 3 elements in all. Where the matrices of the
    workload do not fit the SMs' shared memory it is 16 bytes an element of HBM
    bandwidth (the multiply-adds then take less than half of that time), else the
    multiply-adds. The decompositions of n <= 160 (the Jacobi route) do not count."""
    elements = sum(k * n ** 3 / 3.0 for n, k in decomps.items() if n > 160) / steps
    held = sum(8.0 * s.n ** 2 for s in wl.searches if s.n > 160)
    if held > REDUCTION_SMEM * sms:
        return "hbm", 16.0 * elements, hbm_gbs * 1e9, "GB/s"
    return "alu", 9.0 * elements, IMAD_PER_CLOCK * sms * sm_mhz * 1e6, "G integer multiply-adds/s"


def phase_flops(wl, prec):
    """Algorithmic flops per step of the GEMM-shaped phases."""
    split = 1 if prec == "fp64" else 3
    samp = sum(2.0 * s.lam * s.n * s.n for s in wl.searches)
    obj = sum(2.0 * s.lam * s.n * s.n for s in wl.searches if s.problem.kind != 3) * split
    cov = sum((s.lam // 2) * s.n * (s.n + 1.0) for s in wl.searches) * split
    return {"sample": samp, "objective": obj, "cov": cov}


def run_engine(args):
    import torch
    rank, local_rank, world = dist_env()
    torch.cuda.set_device(local_rank)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local_rank))
    import paper_2409_11765_gb300 as eng
    from paper_2409_11765_gb300 import _build
    if rank == 0 or world == 1:
        _build.build()
    if dist is not None:
        dist.barrier()
    eig_method = {"auto": 0, "jacobi": 1, "tridiagonal": 2}[args.eig_method]
    wl = workload(args.workload)
    head = args.precision
    runs = {head: measure(args, wl, head, world, rank, dist, True, eig_method)}
    for other in [p for p in args.paths.split(",") if p]:
        if other != head:
            runs[other] = measure(args, wl, other, world, rank, dist, False, eig_method, secondary=True)
    r = runs[head]
    extra = None
    if not args.no_extra and args.workload != "rastrigin-n100-kdist":
        wk = workload("rastrigin-n100-kdist")
        a2 = argparse.Namespace(**vars(args))
        a2.steps, a2.warmup, a2.no_e2e = 50, 5, True
        x = measure(a2, wk, head, world, rank, dist, False, eig_method, secondary=True)
        extra = {"workload": wk.name, "value": x["value"], "ms_per_step": x["ms_per_step"],
                 "steps": a2.steps, "warmup": a2.warmup}

    # roofline of the dominant kernel stage of the headline run
    fp64_peak = eng.probe_fma_tflops(64)
    peaks = {}
    try:
        peaks = json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))
    except (OSError, ValueError):
        pass
    steps = args.steps
    cands = dict(r["eig_stages_ms_per_step"])
    for k in ("sample", "objective", "update", "cov", "stop"):
        cands[k] = r["phases_ms_per_step"][k]
    eig_other = r["phases_ms_per_step"]["eig"] - sum(r["eig_stages_ms_per_step"].values())
    cands["eig_other"] = max(eig_other, 0.0)
    dom = max(cands, key=cands.get)
    flops = stage_flops(r["decompositions"])
    flops = {k: v / steps for k, v in flops.items()}
    flops.update(phase_flops(wl, head))
    dom_ms = cands[dom]
    achieved = flops.get(dom, 0.0) / (dom_ms * 1e-3) / 1e12 if dom_ms > 0 else 0.0
    if dom in ("reduction", "backtransform", "eigenvalues", "eigenvectors", "orthogonalisation",
               "eig_other", "update", "stop") or head == "fp64":
        bound, peak, src = "alu", fp64_peak, "FP64 FMA rate measured live by the engine's probe"
    else:
        bf16 = peaks.get("bf16_tflops", 1908.7)
        peak = bf16 * (0.5 if head == "tf32" else 1.0)
        bound, src = "tensor", ("MEASURED_PEAKS.json bf16 x nominal tf32/bf16 ratio 0.5"
                                if head == "tf32" else "MEASURED_PEAKS.json bf16")
    unit = "TFLOP/s"
    work = {"algorithmic_flops_per_step": flops.get(dom, 0.0)}
    if dom == "reduction":
        sms = torch.cuda.get_device_properties(local_rank).multi_processor_count
        bound, amount, rate, unit = reduction_roof(wl, r["decompositions"], steps, peaks.get("hbm_gbs", 6800.0), sms,
                                                   r["clocks"]["sm_mhz"] or 2070.0)
        peak, achieved = rate / 1e9, amount / (dom_ms * 1e-3) / 1e9
        src = ("MEASURED_PEAKS.json hbm_gbs" if bound == "hbm"
               else "%g integer multiply-adds a clock and SM at the median clock" % IMAD_PER_CLOCK)
        work = {"algorithmic_bytes_per_step" if bound == "hbm" else "algorithmic_multiply_adds_per_step": amount}
    traffic = None
    kt = KERNEL_TRAFFIC.get(dom)
    if kt and kt["workload"] == wl.name and stage_sources_sha(dom) == kt["sources_sha256_16"]:
        traffic = kt["bytes_per_step"]
    roofline = {"bound": bound, "achieved": achieved, "peak": peak, "unit": unit,
                "frac": achieved / peak if peak else None, "traffic": traffic, "kernel": dom,
                "peak_source": src, **work, "kernel_ms_per_step": dom_ms}
    if rank != 0:
        if dist is not None:
            dist.destroy_process_group()
        return
    line = {"metric": METRIC, "value": r["value"], "unit": UNIT, "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": r["ms_per_step"],
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": DTYPE[head], "data": "synthetic", "config": workload_config(wl, head, eig_method),
            "roofline": roofline, "e2e": r.get("e2e"), "gpu_launches": r["gpu_launches"],
            "clocks": r["clocks"], "phases_ms_per_step": r["phases_ms_per_step"],
            "eig_stages_ms_per_step": r["eig_stages_ms_per_step"],
            "decompositions_per_step": {str(n): k / steps for n, k in sorted(r["decompositions"].items())},
            "step_ms": r["step_ms"]}
    for other, o in runs.items():
        if other != head:
            line[other + "_path"] = {"value": o["value"], "ms_per_step": o["ms_per_step"]}
    if "fp64_path" in line and head != "fp64":
        line["mixed_over_fp64"] = r["value"] / line["fp64_path"]["value"]
    if extra:
        line["kdist_n100"] = extra
    if not args.no_cpu_baseline and world == 1:
        line["cpu_baseline"] = cpu_baseline(wl, args.cpu_seconds)
    print(json.dumps(line), flush=True)
    if dist is not None:
        dist.destroy_process_group()


def main():
    args = parse_args()
    if args.impl == "reference":
        run_reference(args)
    else:
        run_engine(args)


if __name__ == "__main__":
    main()
