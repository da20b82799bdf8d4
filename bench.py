"""Benchmark of the RA-FEAST hot path on GB300.

One step = one full RA-FEAST solve (Algorithm 2: randomized warmstart, then
FEAST iterations until every in-interval Ritz pair has relative residual <=
outer_tol) of the workload below, inputs resident in HBM. Prints one JSON line.

``--workload sbm64``: the batched sweep, 64 stochastic-block-model Laplacians
of uneven n (2,000 to 300,000) solved by one rafeast_solve_batched call
(grouped COCG launches under one captured graph) per step; the line also
reports the same 64 problems solved one at a time by rafeast_solve.

Default workload (``knn200k``): kNN graph Laplacian of 200,000 uniform points
in [0,1]^3 (seed 2), k = 10, union-symmetrised, unit weights, + 1e-3 I; the
64 smallest eigenvalues; m0 = 80, N_c = 4, p = 20, q = 2, outer tolerance
1e-11, relaxed inner solves (COCG tolerance 1e-2, at most 60 steps), mixed
precision (float32 shifted solves, double outer loop). Every timed step
starts with a cold L2 (a 512 MB write before it, outside its CUDA events).

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = ("RA-FEAST time-to-solution & SpMM HBM GB/s, FP32-mixed vs FP64, "
          "eig relerr≤1e-8")
FALLBACK_HBM_GBS = 6800.0
# FP64 issue rate of the part: the nominal 1.25 TFLOP/s FP64 (an FMA counted
# as 2 flops) over 152 SMs at 2070 MHz is 2 FP64 lane operations (an add or an
# FMA each) per SM per clock
FP64_OPS_PER_SM_CLK = 2.0

WORKLOADS = {
    "knn200k": dict(key="knn200k", precision="mixed"),
    "grid3d": dict(key="grid3d", precision="mixed"),
    "knn8k": dict(key="knn8k", precision="fp64"),
    "sbm64": dict(key="sbm64", precision="mixed"),
    "rgg16k": dict(key="rgg16k", precision="fp64"),
}


def _peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured"
    return FALLBACK_HBM_GBS, "fallback"


def _traffic_per_launch(kernel: str, workload: str):
    """DRAM bytes per launch from the committed ncu summary, if any."""
    path = os.path.join(ROOT, "profiles", f"{kernel}_{workload}.md")
    if not os.path.exists(path):
        return None
    for line in open(path):
        if line.strip().startswith("traffic_bytes_per_launch:"):
            v = line.split(":", 1)[1].strip()
            return None if v in ("", "null", "None") else float(v)
    return None



def max_over_ranks(value: float, dist=None, device="cpu") -> float:
    """The largest `value` over all ranks (time-like quantities of a replica
    run: the whole job ends with its slowest rank); identity without a
    process group."""
    if dist is None:
        return float(value)
    import torch
    t = torch.tensor([float(value)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def whole_job_rate(units_per_rank: float, world: int, ms: float) -> float:
    """Units of all replicas per second over the slowest rank's time."""
    return units_per_rank * world / (ms / 1e3)


def sharded_rate(units_total: float, ms: float) -> float:
    """Units the ranks processed together per second over the slowest rank's
    time (a sharded run: every unit is shared out, not repeated)."""
    return units_total / (ms / 1e3)


def my_instances(costs, world: int, rank: int, R=None):
    """Indices of the problems this rank solves (longest first to the least
    loaded rank, rafeast_partition_instances); all of them at world = 1."""
    if world == 1:
        return list(range(len(costs)))
    owner = R.rafeast_partition_instances(costs, world)
    return [t for t in range(len(costs)) if owner[t] == rank]

class Clocks:
    """nvidia-smi sampling during the timed region."""

    def __init__(self, index: int):
        self.proc = None
        self.path = None
        self.index = index

    def start(self):
        try:
            fd, self.path = tempfile.mkstemp(suffix=".csv")
            os.close(fd)
            q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
                 "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
                 "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--id={self.index}", f"--query-gpu={q}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        rows = []
        for line in open(self.path):
            parts = [p.strip() for p in line.split(",")]
            if len(parts) >= 9:
                rows.append(parts)
        os.unlink(self.path)
        if not rows:
            return None
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4) if r[5 + i] == "Active"})
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(mx) if mx else None, "reasons": reasons,
                "samples": len(rows)}


def _cpu_sample(key: str, gpu_counts: dict, budget: str = "full", threads: int = 1):
    """Time the oracle (unchanged; single-threaded as in the paper's runs, or
    with `threads` BLAS threads) on a bounded sample of the workload in a
    fresh process; extrapolate one solve."""
    code = r"""
import json, os, sys, time
sys.path.insert(0, sys.argv[1])
import numpy as np
from oracle import cocg as OC, feast as OF, philox as OP, quadrature as OQ
from workloads import configs as CF
key, counts, budget = sys.argv[2], json.loads(sys.argv[3]), sys.argv[4]
cfg = CF.CONFIGS[key]
lap = cfg.make(); a = lap.scipy()
lmin, lmax = CF.interval(key)
n, m0 = lap.n, cfg.m0
steps = 3 if budget == "full" else 2
t0 = time.perf_counter()
om = OP.gaussian_matrix(n, m0 + cfg.p, cfg.seed)
q0, th0, _ = OF.warmstart(a, lmin, lmax, m0, cfg.p, cfg.q, om)
t_ws = time.perf_counter() - t0
z, w = OQ.nodes(lmin, lmax, cfg.nc, cfg.e)
rmat = a @ q0 - q0 * th0
t0 = time.perf_counter()
OC.cocg(lambda x: a @ x, z[0], rmat, 0.0, steps)
t_step = (time.perf_counter() - t0) / steps
t0 = time.perf_counter()
q = OF.orthonormalize(q0)
OF.rayleigh_ritz(a, q)
t_rr = time.perf_counter() - t0
est = t_ws + counts["outer"] * t_rr + cfg.nc * counts["cocg_total"] * t_step
print(json.dumps(dict(est=est, t_ws=t_ws, t_step=t_step, t_rr=t_rr, steps=steps)))
"""
    env = dict(os.environ, OMP_NUM_THREADS=str(threads), OPENBLAS_NUM_THREADS=str(threads),
               MKL_NUM_THREADS=str(threads), CUDA_VISIBLE_DEVICES="")
    t0 = time.perf_counter()
    res = subprocess.run([sys.executable, "-c", code, ROOT, key, json.dumps(gpu_counts), budget],
                         capture_output=True, text=True, env=env)
    wall = time.perf_counter() - t0
    if res.returncode != 0:
        return {"error": res.stderr[-400:]}
    d = json.loads(res.stdout.strip().splitlines()[-1])
    d["wall_s"] = wall
    return d


_REF_CODE = r"""
import json, sys, time
sys.path.insert(0, sys.argv[1])
import numpy as np
from oracle import cocg as OC, feast as OF, philox as OP, quadrature as OQ
from workloads import configs as CF
key, nsteps = sys.argv[2], int(sys.argv[3])
cfg = CF.CONFIGS[key]
lap = cfg.make(); a = lap.scipy()
lmin, lmax = CF.interval(key)
n, m0 = lap.n, cfg.m0
t0 = time.perf_counter()
om = OP.gaussian_matrix(n, m0 + cfg.p, cfg.seed)
q0, th0, _ = OF.warmstart(a, lmin, lmax, m0, cfg.p, cfg.q, om)
t_ws = time.perf_counter() - t0
z, w = OQ.nodes(lmin, lmax, cfg.nc, cfg.e)
rmat = a @ q0 - q0 * th0
print(json.dumps(dict(t_ws=t_ws)), flush=True)
for _ in range(nsteps):
    t0 = time.perf_counter()
    OC.cocg(lambda x: a @ x, z[0], rmat, 0.0, 2)
    t_step = (time.perf_counter() - t0) / 2
    t0 = time.perf_counter()
    OF.rayleigh_ritz(a, OF.orthonormalize(q0))
    t_rr = time.perf_counter() - t0
    print(json.dumps(dict(t_step=t_step, t_rr=t_rr)), flush=True)
"""


def run_reference(args):
    """--impl reference: the oracle, unchanged, on the host cores (one BLAS
    thread, as the paper's runs). The warmstart of Phase 1 is timed once;
    every step then times a bounded sample of the same solve, two COCG steps
    of one shift on the full matrix and one Rayleigh-Ritz, and the solve's
    time is extrapolated from them to the GPU solve's iteration counts.
    ms_per_step is the measured time of a sample step."""
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    key = WORKLOADS[args.workload]["key"]
    if key == "sbm64":
        return _run_reference_sbm(args)
    counts = _reference_counts(key)
    env = dict(os.environ, OMP_NUM_THREADS="1", OPENBLAS_NUM_THREADS="1", MKL_NUM_THREADS="1",
               CUDA_VISIBLE_DEVICES="")
    res = subprocess.run([sys.executable, "-c", _REF_CODE, ROOT, key,
                          str(args.warmup + args.steps)], capture_output=True, text=True, env=env)
    if res.returncode != 0:
        print(json.dumps({"impl": "reference", "unavailable": res.stderr[-200:]}))
        return 0
    rows = [json.loads(x) for x in res.stdout.strip().splitlines()]
    t_ws = rows[0]["t_ws"]
    timed = rows[1 + args.warmup:]
    t_step = statistics.mean(r["t_step"] for r in timed)
    t_rr = statistics.mean(r["t_rr"] for r in timed)
    cfg_nc = _config(key)["nc"]
    est = t_ws + counts["outer"] * t_rr + cfg_nc * counts["cocg_total"] * t_step
    sample_ms = statistics.mean(2 * r["t_step"] + r["t_rr"] for r in timed) * 1e3
    sample = (f"per step: two oracle COCG steps of one shift on the full matrix "
              f"({t_step:.3f} s each) + one Rayleigh-Ritz ({t_rr:.2f} s); the warmstart timed once "
              f"({t_ws:.1f} s); one solve extrapolated to {counts['outer']} outer and "
              f"{counts['cocg_total']} COCG iterations x {cfg_nc} shifts ({est:.0f} s)")
    value = 1.0 / est
    line = {"metric": METRIC, "value": value, "unit": "solves/s", "impl": "reference",
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": sample_ms, "ms_per_solve_extrapolated": est * 1e3,
            "higher_is_better": True,
            "scaling": "weak" if args.shard == "replicas" else "strong",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": dict(_config(key), parallelism="the oracle on the host cores (rank 0)"),
            "cpu_baseline": {"value": value, "unit": "solves/s", "cores": 1, "kind": "oracle",
                             "sample": sample},
            "e2e": {"value": value, "unit": "solves/s", "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}
    print(json.dumps(line))
    return 0


def _run_reference_sbm(args):
    """--impl reference --workload sbm64: the oracle on the median instance,
    scaled by nnz to all 64 and to the GPU solve's mean iteration counts."""
    from types import SimpleNamespace
    from workloads import configs as CF
    insts = CF.sbm_instances()
    gold = CF.load_golden()["sbm64"]["instances"]
    # mean per-instance counts of the batched GPU solve (22.4 outer iterations,
    # 38,100 COCG steps over the 64 instances)
    infos = [SimpleNamespace(outer_iters=22, cocg_iters_total=595) for _ in insts]
    ests = []
    for i in range(args.warmup + args.steps):
        d = _cpu_sample_sbm(insts, gold, infos)
        if "error" in d:
            print(json.dumps({"impl": "reference", "unavailable": d["error"][-200:]}))
            return 0
        if i >= args.warmup:
            ests.append(d)
    est = statistics.mean(d["est"] for d in ests)
    value = len(insts) / est
    line = {"metric": METRIC, "value": value, "unit": "problems/s", "impl": "reference",
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": est * 1e3, "higher_is_better": True, "scaling": "strong",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": "sbm64: 64 stochastic-block-model Laplacians, batched",
                       "parallelism": "the oracle on the host cores (rank 0)"},
            "cpu_baseline": {"value": value, "unit": "problems/s", "cores": 1, "kind": "oracle",
                             "sample": ests[0]["sample"]},
            "e2e": {"value": value, "unit": "problems/s", "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}
    print(json.dumps(line))
    return 0


def _reference_counts(key):
    # iteration counts of the GPU solve of this workload (same algorithm and
    # parameters); used only to extrapolate the oracle's bounded sample
    table = {"knn200k": dict(outer=8, cocg_total=800),
             "grid3d": dict(outer=9, cocg_total=900),
             "knn8k": dict(outer=11, cocg_total=900),
             "rgg16k": dict(outer=4, cocg_total=389)}
    return table[key]


def _config(key):
    from workloads import configs as CF
    cfg = CF.CONFIGS[key]
    g = CF.load_golden()[key]
    return {"workload": f"{key}: {cfg.description}", "n": g["n"], "nnz": g["nnz"],
            "count": g["count"], "m0": cfg.m0, "nc": cfg.nc, "p": cfg.p, "q": cfg.q,
            "solve_tol": cfg.solve_tol, "max_inner": cfg.max_inner, "outer_tol": cfg.outer_tol,
            "interval": [g["lmin"], g["lmax"]],
            "l2": "L2 flushed (512 MB write, outside the timed events) before every timed step"}


def run_batched(args):
    """--workload sbm64: one step = warmstart of all 64 instances + one
    batched solve; the per-instance loop of the same work is timed beside it."""
    import numpy as np
    import torch
    from paper_2512_01257_gb300 import rafeast as R
    from workloads import configs as CF

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    dev = torch.device("cuda", local)
    S = CF.SBM_SOLVE
    gold = CF.load_golden()["sbm64"]["instances"]
    insts = CF.sbm_instances()
    total = len(insts)
    # N ranks: each solves its share of the problems (cost nnz x m0), no
    # exchange between ranks
    mine = my_instances([g["nnz"] * i["m0"] for i, g in zip(insts, gold)], world, rank, R)
    insts = [insts[t] for t in mine]
    gold = [gold[t] for t in mine]
    t_gen = time.perf_counter()
    laps = [CF.make_sbm(i) for i in insts]
    t_gen = time.perf_counter() - t_gen
    for lap, g in zip(laps, gold):
        assert lap.checksum() == g["checksum"], "instance differs from the stored spectrum"
    hs = []
    for lap in laps:
        hs.append(R.rafeast_create(torch.from_numpy(lap.row_ptr).to(dev),
                                   torch.from_numpy(lap.col_idx).to(dev),
                                   torch.from_numpy(lap.values).to(dev), lap.shift))
    cnt = len(hs)
    m0s = [i["m0"] for i in insts]
    prms = [R.make_params(g["lmin"], g["lmax"], i["m0"], S["nc"], S["e"], S["solve_tol"],
                          S["outer_tol"], S["max_outer"], S["max_inner"], R.RAFEAST_MIXED,
                          R.RAFEAST_FORM_CORRECTION, R.RAFEAST_START_SUBSPACE)
            for i, g in zip(insts, gold)]
    evals = [torch.zeros(m, dtype=torch.float64, device=dev) for m in m0s]
    evecs = [torch.zeros((m, lap.n), dtype=torch.float64, device=dev) for m, lap in zip(m0s, laps)]
    resid = [torch.zeros(m, dtype=torch.float64, device=dev) for m in m0s]
    last = {}

    def warm(hl):
        for h, i, g in zip(hl, insts, gold):
            R.rafeast_warmstart(h, g["lmin"], g["lmax"], i["m0"], S["p"], S["q"], i["seed"])

    def step():
        warm(hs)
        st, mf, info = R.rafeast_solve_batched(hs, prms, evals, evecs, resid)
        # 2 (no convergence within max_outer) still returns the best iterate;
        # the parity check below decides whether its eigenvalues are right
        if any(x not in (R.RAFEAST_OK, R.RAFEAST_NO_CONVERGENCE) for x in st):
            raise RuntimeError(f"batched statuses {st}")
        last.update(mf=mf, info=info, st=st)

    for _ in range(args.warmup):
        step()
    R.rafeast_set_option(hs[0], R.RAFEAST_OPT_PROFILE, 1)
    R.rafeast_profile(hs[0], reset=True)
    clocks = Clocks(local)
    stream = torch.cuda.current_stream()
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    clocks.start()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    launches = 0
    for _ in range(args.steps):
        step()
        launches += sum(i.kernel_launches for i in last["info"])
    e1.record(stream)
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    ck = clocks.stop()
    ms = e0.elapsed_time(e1)
    prof = R.rafeast_profile(hs[0], reset=True)
    R.rafeast_set_option(hs[0], R.RAFEAST_OPT_PROFILE, 0)
    ms = max_over_ranks(ms, dist, dev)
    ms_step = ms / args.steps
    # parity: every instance's eigenvalues against its stored Lanczos spectrum
    worst, found_all = 0.0, True
    for t in range(cnt):
        mf = last["mf"][t]
        ev = np.sort(evals[t].cpu().numpy()[:mf])
        ref = np.array(gold[t]["evals"])
        if mf != len(ref):
            found_all = False
            continue
        worst = max(worst, float(np.max(np.abs(ev - ref) / np.abs(ref))))
    infos = last["info"]
    n_conv = sum(1 for x in last["st"] if x == R.RAFEAST_OK)
    it_max = max(i.outer_iters for i in infos)
    it_sum = sum(i.outer_iters for i in infos)
    if dist:
        agg = torch.tensor([worst, 0.0 if found_all else 1.0, float(it_max)], dtype=torch.float64,
                           device=dev)
        dist.all_reduce(agg, op=dist.ReduceOp.MAX)
        tot = torch.tensor([float(n_conv), float(it_sum)], dtype=torch.float64, device=dev)
        dist.all_reduce(tot, op=dist.ReduceOp.SUM)
        worst, found_all, it_max = float(agg[0]), agg[1].item() == 0.0, int(agg[2])
        n_conv, it_sum = int(tot[0]), float(tot[1])
    # the same 64 problems one at a time (rafeast_solve each, same settings)
    loop_ms, loop_kernels = None, None
    trace = R.rafeast_profile_history(hs[0])
    if not args.no_loop and world == 1:
        for h in hs:
            R.rafeast_set_option(h, R.RAFEAST_OPT_PROFILE, 1)
            R.rafeast_profile(h, reset=True)
        torch.cuda.synchronize()
        l0 = torch.cuda.Event(enable_timing=True)
        l1 = torch.cuda.Event(enable_timing=True)
        l0.record(stream)
        warm(hs)
        loop_info = []
        for t in range(cnt):
            st, _, inf = R.rafeast_solve(hs[t], prms[t], evals[t], evecs[t], resid[t])
            assert st in (R.RAFEAST_OK, R.RAFEAST_NO_CONVERGENCE)
            loop_info.append(inf)
        l1.record(stream)
        torch.cuda.synchronize()
        loop_ms = l0.elapsed_time(l1)
        lp = [R.rafeast_profile(h, reset=True) for h in hs]
        for h in hs:
            R.rafeast_set_option(h, R.RAFEAST_OPT_PROFILE, 0)
        loop_kernels = {"dots_ms": sum(p["dots_ms"] for p in lp),
                        "update_ms": sum(p["update_ms"] for p in lp),
                        "steps": int(sum(p["dots_launches"] for p in lp)),
                        # the slowest problems solved alone: the batched
                        # step cannot end before the slowest of them
                        "slowest": [{"n": laps[t].n, "outer": loop_info[t].outer_iters,
                                     "ms": loop_info[t].t_total_ms,
                                     "filter_ms": loop_info[t].t_filter_ms,
                                     "orth_ms": loop_info[t].t_orth_ms,
                                     "rr_ms": loop_info[t].t_rr_ms}
                                    for t in sorted(range(cnt), key=lambda t: -loop_info[t].t_total_ms)[:4]]}
    peak, peak_kind = _peaks()
    pre = "update" if prof["update_ms"] >= prof["dots_ms"] else "dots"
    names = {"update": "lz_update_grouped", "dots": "lz_dots_grouped"}
    launches_k = max(prof[f"{pre}_launches"], 1.0)
    bytes_per = prof[f"{pre}_bytes"] / launches_k
    ms_per = prof[f"{pre}_ms"] / launches_k
    achieved = bytes_per / (ms_per * 1e-3) / 1e9
    other = "dots" if pre == "update" else "update"
    roofline = {"bound": "hbm", "kernel": names[pre], "achieved": achieved, "peak": peak,
                "peak_kind": peak_kind, "unit": "GB/s", "frac": achieved / peak,
                "traffic": _traffic_per_launch(names[pre], "sbm64"),
                "algorithmic_bytes_per_launch": bytes_per, "ms_per_launch": ms_per,
                "launches": int(launches_k),
                "shapes": {"dots": prof.get("dots_shape"), "update": prof.get("update_shape"),
                           "note": "lanes*100+chunks, 0 = per-problem default"},
                "other_kernel": {"kernel": names[other],
                                 "achieved": (prof[f"{other}_bytes"] / max(prof[f"{other}_ms"], 1e-9))
                                 / 1e6,
                                 "ms_per_launch": prof[f"{other}_ms"] / max(prof[f"{other}_launches"], 1)},
                "share_of_step": (prof["update_ms"] + prof["dots_ms"]) / ms}
    ns = [lap.n for lap in laps]
    value = sharded_rate(args.steps * total, ms)
    line = {"metric": METRIC, "value": value, "unit": "problems/s", "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_step,
            "time_to_solution_s": ms_step / 1e3, "higher_is_better": True, "scaling": "strong",
            "vs_baseline": None, "dtype": "f32",
            "precision": "mixed: f32 shifted solves and SpMM; f64 Gram, Cholesky-QR, "
                         "Rayleigh-Ritz, residuals",
            "data": "synthetic (seeded generator, no dataset)",
            "config": {"workload": "sbm64: 64 stochastic-block-model Laplacians + 1e-3 I, n "
                                   "log-uniform in [2000, 300000], 4-16 blocks, p_in=20/n_block, "
                                   "p_out=1/n, k=blocks+8, m0=ceil(1.5k), N_c=2 (ellipse ratio "
                                   "0.3), batched",
                       "count": total, "sum_n": int(sum(ns)), "min_n": min(ns), "max_n": max(ns),
                       "sum_nnz": int(sum(lap.nnz for lap in laps)), "nc": S["nc"],
                       "parallelism": (f"instances sharded over {world} ranks by nnz x m0 "
                                       "(no exchange); n and nnz figures are rank 0's share"
                                       if world > 1 else "one GPU"),
                       "p": S["p"], "q": S["q"], "solve_tol": S["solve_tol"],
                       "outer_tol": S["outer_tol"], "max_inner": S["max_inner"],
                       "l2": "inputs larger than L2 (no flush): COCG state of all instances"},
            "parity": {"max_eig_relerr_vs_lanczos": worst if found_all else None,
                       "all_found": found_all, "gate": 1e-8,
                       "converged": n_conv, "count": total},
            "outer_iters_max": it_max,
            # per-problem phase times of the last step, summed over this
            # rank's problems (they overlap on the problems' own streams)
            "phases_ms_sum": {"filter_ms": sum(i.t_filter_ms for i in infos),
                              "orth_ms": sum(i.t_orth_ms for i in infos),
                              "rr_ms": sum(i.t_rr_ms for i in infos),
                              "total_ms_max": max(i.t_total_ms for i in infos)},
            "outer_iters_mean": it_sum / total,
            "per_instance_loop_ms": loop_ms, "per_instance_loop_kernels": loop_kernels,
            "batched_kernels": {"dots_ms": prof["dots_ms"] / args.steps,
                                "update_ms": prof["update_ms"] / args.steps,
                                "steps": int(prof["dots_launches"] / args.steps)},
            "batched_speedup_vs_loop": (loop_ms / ms_step) if loop_ms else None,
            "roofline": roofline, "gpu_launches": int(launches), "clocks": ck,
            "generation_s": t_gen}
    if args.trace:
        cols, probs, kms = trace
        with open(args.trace, "w") as f:
            json.dump({"active_pairs": cols.tolist(), "active_problems": probs.tolist(),
                       "ms": kms.tolist()}, f)
    for h in hs:
        R.rafeast_destroy(h)
    if not args.no_e2e:
        pins = [(torch.from_numpy(l.row_ptr).pin_memory(), torch.from_numpy(l.col_idx).pin_memory(),
                 torch.from_numpy(l.values).pin_memory()) for l in laps]
        oev = [np.zeros(m) for m in m0s]
        ove = [np.zeros((m, l.n)) for m, l in zip(m0s, laps)]
        ore = [np.zeros(m) for m in m0s]
        bi = sum(a.numel() * 4 + b.numel() * 4 + c.numel() * 8 for a, b, c in pins)
        bo = sum(a.nbytes + b.nbytes + c.nbytes for a, b, c in zip(oev, ove, ore))

        def e2e_step():
            hl = [R.rafeast_create(a.numpy(), b.numpy(), c.numpy(), l.shift)
                  for (a, b, c), l in zip(pins, laps)]
            try:
                warm(hl)
                st, _, _ = R.rafeast_solve_batched(hl, prms, oev, ove, ore)
                assert all(x in (R.RAFEAST_OK, R.RAFEAST_NO_CONVERGENCE) for x in st)
            finally:
                for h in hl:
                    R.rafeast_destroy(h)

        torch.cuda.synchronize()
        if dist:
            dist.barrier()
        t0 = time.perf_counter()
        e2e_step()
        torch.cuda.synchronize()
        el = time.perf_counter() - t0
        el = max_over_ranks(el, dist, dev)
        if dist:
            bt = torch.tensor([float(bi), float(bo)], dtype=torch.float64, device=dev)
            dist.all_reduce(bt, op=dist.ReduceOp.SUM)
            bi, bo = int(bt[0]), int(bt[1])
        line["e2e"] = {"value": total / el, "unit": "problems/s",
                       "h2d_bytes_per_step": bi, "d2h_bytes_per_step": bo, "steps": 1,
                       "includes": "rafeast_create of all 64 from pinned host CSR, warmstarts, "
                                   "batched solve, copy of eigenpairs to host"}
    if not args.no_cpu and rank == 0 and world == 1:
        d = _cpu_sample_sbm(insts, gold, infos)
        if "est" in d:
            line["cpu_baseline"] = {"value": cnt / d["est"], "unit": "problems/s", "cores": 1,
                                    "kind": "oracle", "sample": d["sample"],
                                    "est_seconds_per_step": d["est"]}
        else:
            line["cpu_baseline"] = {"error": d.get("error")}
        # the same oracle with every host core as BLAS threads (its sparse
        # products and vector updates stay single-threaded)
        cores = os.cpu_count() or 1
        d = _cpu_sample_sbm(insts, gold, infos, threads=cores)
        if "est" in d:
            line["cpu_baseline_all_cores"] = {
                "value": cnt / d["est"], "unit": "problems/s", "cores": cores, "kind": "oracle",
                "sample": f"as cpu_baseline with {cores} BLAS threads",
                "est_seconds_per_step": d["est"]}
    if rank == 0:
        print(json.dumps(line))
    if dist:
        dist.destroy_process_group()
    return 0


def _cpu_sample_sbm(insts, gold, infos, threads: int = 1):
    """Oracle (single-threaded) on the instance of median size: warmstart, a
    few COCG steps, one Rayleigh-Ritz; extrapolated to the whole batch by nnz
    and to each instance's GPU iteration counts."""
    med = sorted(range(len(insts)), key=lambda t: insts[t]["n"])[len(insts) // 2]
    code = r"""
import json, sys, time
sys.path.insert(0, sys.argv[1])
from oracle import cocg as OC, feast as OF, philox as OP, quadrature as OQ
from workloads import configs as CF
t = int(sys.argv[2]); lmin, lmax = float(sys.argv[3]), float(sys.argv[4])
S = CF.SBM_SOLVE
inst = CF.sbm_instances()[t]
a = CF.make_sbm(inst).scipy()
n, m0 = a.shape[0], inst["m0"]
t0 = time.perf_counter()
om = OP.gaussian_matrix(n, m0 + S["p"], inst["seed"])
q0, th0, _ = OF.warmstart(a, lmin, lmax, m0, S["p"], S["q"], om)
t_ws = time.perf_counter() - t0
z, w = OQ.nodes(lmin, lmax, S["nc"], S["e"])
rmat = a @ q0 - q0 * th0
t0 = time.perf_counter()
OC.cocg(lambda x: a @ x, z[0], rmat, 0.0, 3)
t_step = (time.perf_counter() - t0) / 3
t0 = time.perf_counter()
OF.rayleigh_ritz(a, OF.orthonormalize(q0))
t_rr = time.perf_counter() - t0
print(json.dumps(dict(t_ws=t_ws, t_step=t_step, t_rr=t_rr, nnz=a.nnz)))
"""
    env = dict(os.environ, OMP_NUM_THREADS=str(threads), OPENBLAS_NUM_THREADS=str(threads),
               MKL_NUM_THREADS=str(threads), CUDA_VISIBLE_DEVICES="")
    g = gold[med]
    t0 = time.perf_counter()
    res = subprocess.run([sys.executable, "-c", code, ROOT, str(med), repr(g["lmin"]),
                          repr(g["lmax"])], capture_output=True, text=True, env=env)
    wall = time.perf_counter() - t0
    if res.returncode != 0:
        return {"error": res.stderr[-400:]}
    d = json.loads(res.stdout.strip().splitlines()[-1])
    est = 0.0
    for t, (i, gg) in enumerate(zip(insts, gold)):
        f = gg["nnz"] / d["nnz"]
        est += f * (d["t_ws"] + infos[t].outer_iters * d["t_rr"]
                    + 2 * infos[t].cocg_iters_total * d["t_step"])
    sample = (f"oracle on instance {med} (n={insts[med]['n']}): warmstart, 3 COCG steps of one "
              f"shift, one Rayleigh-Ritz ({wall:.1f} s of CPU work); scaled by nnz to every "
              f"instance and to its GPU outer / COCG iteration counts x 2 shifts")
    return {"est": est, "sample": sample}


def _unit_laplacian(lap):
    """(values-free, off-diagonal count): whether the CSR is a unit-weight
    graph Laplacian (off-diagonal entries -1, diagonal = the row's number of
    off-diagonal entries), the matrices whose dot kernels gather on the
    pattern alone."""
    import numpy as np
    n = lap.n
    rp = lap.row_ptr.astype(np.int64)
    rows = np.repeat(np.arange(n), np.diff(rp))
    diag = rows == lap.col_idx
    off = ~diag
    deg = np.bincount(rows[off], minlength=n)
    vf = bool(np.all(lap.values[off] == -1.0) and np.all(lap.values[diag] == deg[rows[diag]]))
    return vf, int(off.sum())


def _fp64_dots_roofline(hbm, prof, lap, dev):
    """The FP64 product without fixed-point sums is bound by the FP64 pipe, not
    by HBM: every gathered entry costs one FP64 add (values-free) or FMA, 1.25
    TFLOP/s nominal on this part against 64x that for FP32. Its FP64 lane
    operations per launch: per active column, one per gathered entry and three
    per row (L u from the sum, the two dot products). The active columns come
    from the library's byte count of the same launches (A once plus, per
    column, u read and w written)."""
    import torch
    n = lap.n
    vf, nnz_off = _unit_laplacian(lap)
    abytes = (nnz_off * 4.0 if vf else lap.nnz * 12.0) + 4.0 * (n + 1)
    launches = max(prof["dots_launches"], 1.0)
    act_cols = (prof["dots_bytes"] - launches * abytes) / (2.0 * 8.0 * n)
    gathered = nnz_off if vf else lap.nnz
    ops = act_cols * (gathered + 3.0 * n)
    ms = prof["dots_ms"]
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    mhz = 2070.0
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            mhz = float(json.load(f).get("sm_max_mhz", mhz))
    peak = sms * FP64_OPS_PER_SM_CLK * mhz * 1e6 / 1e9
    achieved = ops / (ms * 1e-3) / 1e9
    out = {"bound": "alu", "kernel": hbm["kernel"], "achieved": achieved, "peak": peak,
           "peak_kind": (f"derived: {sms} SMs x {FP64_OPS_PER_SM_CLK:g} FP64 ops/clk x "
                         f"{mhz:g} MHz (nominal 1.25 TFLOP/s FP64)"),
           "unit": "G FP64 ops/s (an add or an FMA = 1)", "frac": achieved / peak,
           "traffic": None, "fp64_ops_per_launch": ops / launches,
           "ms_per_launch": hbm["ms_per_launch"], "launches": hbm["launches"],
           "shapes": hbm["shapes"], "other_kernel": hbm["other_kernel"],
           "share_of_step": hbm["share_of_step"],
           "hbm_view": {k: hbm[k] for k in ("achieved", "peak", "unit", "frac",
                                            "algorithmic_bytes_per_launch")}}
    return out


def _rgg_table(R, h, torch, stream, g, cfg, evals):
    """Table 1 of the paper on this GPU: standard FEAST (N_c = 8, random start,
    tight solves, to convergence) and RA-FEAST at N_c = 8, 4, 2 with the
    iteration limits 2 and 4, in FP64 and with float32 shifted solves; time
    (warm, CUDA events), speedup, maximum absolute eigenvalue error against
    ARPACK, warmstart (Phase 1) time."""
    import numpy as np
    ref = np.array(g["evals"])
    rows = []

    flush = torch.empty(64 * 1024 * 1024, dtype=torch.float64, device=evals.device)

    def timed(fn):
        fn()  # warm
        flush.fill_(1.0)  # cold L2 for the timed run
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        out = fn()
        e1.record(stream)
        torch.cuda.synchronize()
        return e0.elapsed_time(e1), out

    def solve(nc, max_outer, warm, solve_tol, prec=R.RAFEAST_FP64, max_inner=cfg.max_inner):
        def fn():
            t_ws = 0.0
            if warm:
                w0 = torch.cuda.Event(enable_timing=True)
                w1 = torch.cuda.Event(enable_timing=True)
                w0.record(stream)
                R.rafeast_warmstart(h, g["lmin"], g["lmax"], cfg.m0, cfg.p, cfg.q, cfg.seed)
                w1.record(stream)
                torch.cuda.synchronize()
                t_ws = w0.elapsed_time(w1)
            start = R.RAFEAST_START_SUBSPACE if warm else R.RAFEAST_START_RANDOM
            prm = R.make_params(g["lmin"], g["lmax"], cfg.m0, nc, 1.0, solve_tol, cfg.outer_tol,
                                max_outer, max_inner, prec,
                                R.RAFEAST_FORM_CORRECTION, start, cfg.seed)
            try:
                st, mf, info = R.rafeast_solve(h, prm, evals, None, None)
            except R.RafeastError as exc:
                return exc.code, 0, None, None, t_ws
            ev = evals.cpu().numpy()[:mf]
            err = float(np.max(np.abs(np.sort(ev) - ref))) if mf == len(ref) else None
            return st, mf, info, err, t_ws
        return fn

    ms, (st, mf, info, err, _) = timed(solve(8, 40, False, 1e-10))
    base = ms
    rows.append({"method": "standard FEAST (N_c=8, random start, COCG to 1e-10)", "ms": ms,
                 "speedup": 1.0, "max_abs_err": err, "phase1_ms": None,
                 "outer_iters": info.outer_iters if info else None, "status": st})
    for nc in (8, 4, 2):
        for mo in (2, 4):
            ms, (st, mf, info, err, tws) = timed(solve(nc, mo, True, cfg.solve_tol))
            rows.append({"method": f"RA-FEAST (N_c={nc}, max_iter={mo})", "ms": ms,
                         "speedup": base / ms, "max_abs_err": err, "phase1_ms": tws,
                         "outer_iters": info.outer_iters if info else None, "status": st})
    # the same with float32 shifted solves (the outer loop stays FP64): FP64
    # runs at 1/64 of the FP32 rate on this part, and the gathers of a dense
    # RGG row are FP64-issue bound. Float32 COCG keeps the 100-step cap of the
    # other mixed workloads (past it the float recurrences lose their
    # bi-orthogonality and may break down).
    for nc in (8, 4, 2):
        for mo in (2, 4):
            ms, (st, mf, info, err, tws) = timed(solve(nc, mo, True, cfg.solve_tol,
                                                       R.RAFEAST_MIXED, 100))
            rows.append({"method": f"RA-FEAST mixed (N_c={nc}, max_iter={mo}, COCG <= 100 steps)",
                         "ms": ms, "speedup": base / ms, "max_abs_err": err, "phase1_ms": tws,
                         "outer_iters": info.outer_iters if info else None, "status": st})
    return rows


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="knn200k", choices=sorted(WORKLOADS))
    ap.add_argument("--no-fp64", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--no-loop", action="store_true")
    ap.add_argument("--plain", action="store_true",
                    help="also time plain FEAST in FP64 (random start, N_c = 8, COCG to 1e-10; "
                         "about five minutes on knn200k)")
    ap.add_argument("--trace", default="", help="sbm64: write the batched per-step trace here")
    ap.add_argument("--shard", default="columns", choices=["columns", "shifts", "replicas"],
                    help="N > 1, single-problem workloads: share one solve out by subspace "
                         "columns or quadrature nodes (one all-reduce per outer iteration), "
                         "or run a whole replica per rank")
    args = ap.parse_args()
    if args.impl == "reference":
        return run_reference(args)
    if args.workload == "sbm64":
        return run_batched(args)

    import numpy as np
    import torch
    from paper_2512_01257_gb300 import rafeast as R
    from workloads import configs as CF

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    key = WORKLOADS[args.workload]["key"]
    cfg = CF.CONFIGS[key]
    g = CF.load_golden()[key]
    lap = cfg.make()
    assert lap.checksum() == g["checksum"], "workload differs from the stored spectrum"
    lmin, lmax = g["lmin"], g["lmax"]
    prec = R.RAFEAST_MIXED if cfg.precision == "mixed" else R.RAFEAST_FP64
    dev = torch.device("cuda", local)
    rp = torch.from_numpy(lap.row_ptr).to(dev)
    ci = torch.from_numpy(lap.col_idx).to(dev)
    va = torch.from_numpy(lap.values).to(dev)
    h = R.rafeast_create(rp, ci, va, lap.shift)
    m0, n = cfg.m0, lap.n
    evals = torch.zeros(m0, dtype=torch.float64, device=dev)
    evecs = torch.zeros((m0, n), dtype=torch.float64, device=dev)
    resid = torch.zeros(m0, dtype=torch.float64, device=dev)

    def params(p):
        return R.make_params(lmin, lmax, m0, cfg.nc, cfg.e, cfg.solve_tol, cfg.outer_tol,
                             cfg.max_outer, cfg.max_inner, p, R.RAFEAST_FORM_CORRECTION,
                             R.RAFEAST_START_SUBSPACE)

    infos = []
    # N ranks: one solve shared out over the ranks (rafeast_solve_sharded:
    # columns of the subspace, or quadrature nodes), one all-reduce of the
    # filtered block per outer iteration; or whole replicas (--shard replicas)
    sharded = world > 1 and args.shard != "replicas"
    shard_mode = R.RAFEAST_SHARD_SHIFTS if args.shard == "shifts" else R.RAFEAST_SHARD_COLUMNS
    sum_fn = R.allreduce_sum() if sharded else None

    def solve(hh, prm, ev, vec, res):
        if sharded:
            return R.rafeast_solve_sharded(hh, prm, shard_mode, rank, world, sum_fn, ev, vec, res)
        return R.rafeast_solve(hh, prm, ev, vec, res)

    # the RGG workloads stop at the paper's iteration limit (status 2 is the
    # expected outcome there); the others must converge
    ok_status = (R.RAFEAST_OK, R.RAFEAST_NO_CONVERGENCE) if key.startswith("rgg") else (R.RAFEAST_OK,)

    ws_events = []

    def step(p=prec):
        w0 = torch.cuda.Event(enable_timing=True)
        w1 = torch.cuda.Event(enable_timing=True)
        w0.record(torch.cuda.current_stream())
        R.rafeast_warmstart(h, lmin, lmax, m0, cfg.p, cfg.q, cfg.seed)
        w1.record(torch.cuda.current_stream())
        ws_events.append((w0, w1))
        st, mf, info = solve(h, params(p), evals, evecs, resid)
        if st not in ok_status:
            raise RuntimeError(f"solve status {st}: {info.as_dict()}")
        infos.append((mf, info))
        return mf, info

    for _ in range(args.warmup):
        step()
    infos.clear()
    ws_events.clear()
    R.rafeast_set_option(h, R.RAFEAST_OPT_PROFILE, 1)
    R.rafeast_profile(h, reset=True)
    clocks = Clocks(local)
    stream = torch.cuda.current_stream()
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    clocks.start()
    # every timed step starts with a cold L2: a 512 MB write (more than the
    # 126 MB L2) before it, outside its CUDA-event pair
    flush = torch.empty(64 * 1024 * 1024, dtype=torch.float64, device=dev)
    ms = 0.0
    for _ in range(args.steps):
        flush.fill_(1.0)
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        step()
        e1.record(stream)
        torch.cuda.synchronize()
        ms += e0.elapsed_time(e1)
    if dist:
        dist.barrier()
    ck = clocks.stop()
    del flush
    prof = R.rafeast_profile(h, reset=True)
    R.rafeast_set_option(h, R.RAFEAST_OPT_PROFILE, 0)
    ms = max_over_ranks(ms, dist, dev)
    ms_step = ms / args.steps
    value = sharded_rate(args.steps, ms) if sharded else whole_job_rate(args.steps, world, ms)
    # parity of the last timed step against the stored ARPACK eigenvalues
    mf, info = infos[-1]
    ev = evals.cpu().numpy()[:mf]
    ref = np.array(g["evals"])
    relerr = float(np.max(np.abs(np.sort(ev) - ref) / np.abs(ref))) if mf == len(ref) else None
    launches = sum(i.kernel_launches for _, i in infos)
    # rafeast_warmstart (Phase 1) is its own call, timed here; the solve's
    # own phases come from its info record (its start phase is the
    # Rayleigh-Ritz of the warmstart subspace)
    phases = {"warmstart_ms": statistics.mean(a.elapsed_time(b) for a, b in ws_events)}
    for k, name in (("t_warmstart_ms", "solve_start_ms"), ("t_filter_ms", "filter_ms"),
                    ("t_orth_ms", "orth_ms"), ("t_rr_ms", "rr_ms"), ("t_total_ms", "solve_ms")):
        phases[name] = statistics.mean(getattr(i, k) for _, i in infos)

    # roofline of the dominant COCG kernel (live CUDA-event times in the replays)
    peak, peak_kind = _peaks()
    # real Lanczos form (default): the product k_lz_dots or k_lz_dots_tiled and
    # k_lz_update; names of the ncu summaries under profiles/
    names = {"update": "lz_update",
             "dots": "lz_dots_tiled" if prof.get("dots_shape", 0) >= 1000000 else "lz_dots"}
    pre = "update" if prof["update_ms"] >= prof["dots_ms"] else "dots"
    kern = names[pre]
    launches_k = max(prof[f"{pre}_launches"], 1.0)
    bytes_per = prof[f"{pre}_bytes"] / launches_k
    ms_per = prof[f"{pre}_ms"] / launches_k
    achieved = bytes_per / (ms_per * 1e-3) / 1e9
    other = "dots" if pre == "update" else "update"
    roofline = {"bound": "hbm", "kernel": kern, "achieved": achieved, "peak": peak,
                "peak_kind": peak_kind, "unit": "GB/s", "frac": achieved / peak,
                "traffic": _traffic_per_launch(kern, key),
                "algorithmic_bytes_per_launch": bytes_per, "ms_per_launch": ms_per,
                "launches": int(launches_k),
                "shapes": {"dots": prof.get("dots_shape"), "update": prof.get("update_shape")},
                "other_kernel": {"kernel": names[other],
                                 "achieved": (prof[f"{other}_bytes"] / max(prof[f"{other}_ms"], 1e-9))
                                 / 1e6,
                                 "ms_per_launch": prof[f"{other}_ms"] / max(prof[f"{other}_launches"], 1)},
                "share_of_step": (prof["update_ms"] + prof["dots_ms"]) / ms}

    # (neighbour sums in 64-bit integers: the FP64 pipe does not bind them)
    if prec == R.RAFEAST_FP64 and pre == "dots" and not prof["fixed_sums"]:
        roofline = _fp64_dots_roofline(roofline, prof, lap, dev)
    # the sparse product the metric names: w = L u over the CSR pattern (tiled:
    # the gathered rows staged in shared memory) with the step's dot products
    spmm_kern = names["dots"]
    d_launch = max(prof["dots_launches"], 1.0)
    d_bytes = prof["dots_bytes"] / d_launch
    d_ms = prof["dots_ms"] / d_launch
    d_ach = d_bytes / (d_ms * 1e-3) / 1e9
    roofline_spmm = {"bound": "hbm", "kernel": spmm_kern, "achieved": d_ach, "peak": peak,
                     "peak_kind": peak_kind, "unit": "GB/s", "frac": d_ach / peak,
                     "traffic": _traffic_per_launch(spmm_kern, key),
                     "algorithmic_bytes_per_launch": d_bytes, "ms_per_launch": d_ms,
                     "launches": int(d_launch), "shape": prof.get("dots_shape"),
                     "algorithmic_bytes": "pattern once (4 B per index, 4 B per row pointer, "
                                          "values if read) + u read + w written"}

    line = {"metric": METRIC, "value": value, "unit": "solves/s", "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_step,
            "time_to_solution_s": ms_step / 1e3, "higher_is_better": True,
            "scaling": "weak" if args.shard == "replicas" else "strong",
            "vs_baseline": None, "dtype": "f32" if prec == R.RAFEAST_MIXED else "f64",
            "precision": ("mixed: f32 shifted solves and SpMM; f64 Gram, Cholesky-QR, "
                          "Rayleigh-Ritz, residuals") if prec == R.RAFEAST_MIXED else "f64",
            "data": "synthetic (seeded generator, no dataset)",
            "config": dict(_config(key), parallelism=(
                f"one solve sharded over {world} ranks by {args.shard} (one all-reduce of the "
                "n x m0 filtered block per outer iteration)" if sharded else
                f"{world} replicas" if world > 1 else "one GPU")),
            "parity": {"max_eig_relerr_vs_arpack": relerr, "m_found": mf, "count": g["count"],
                       "gate": 1e-8 if prec == R.RAFEAST_MIXED else 1e-10},
            "outer_iters": info.outer_iters, "cocg_iters_total": info.cocg_iters_total,
            "phases_ms": phases, "roofline": roofline, "roofline_spmm": roofline_spmm,
            "gpu_launches": int(launches), "clocks": ck}

    # a step's working set: u_{k-1}, u_k, u_{k+1}, w
    sv = 4 if prec == R.RAFEAST_MIXED else 8
    ws_bytes = n * ((m0 + 3) // 4 * 4) * sv * 4
    if ws_bytes < 126e6:
        line["roofline"]["note"] = (f"a step's working set {ws_bytes / 1e6:.0f} MB fits the 126 MB L2 "
                                    "after the first step: the HBM roofline does not bind")
    if key == "rgg16k":
        # the paper's Table 1 row for this workload: RA-FEAST, N_c = 2,
        # n = 16,000, 72.4 s per solve on one CPU thread with sparse direct
        # solves (another machine: context, not a target)
        line["vs_baseline"] = value * 72.4
        line["vs_baseline_source"] = ("paper Table 1, RA-FEAST (N_c=2) at n=16,000: 72.4 s per "
                                      "solve, single-threaded CPU, FEAST v4 direct solves")
    # the eigenspace of the last timed solve: Davis-Kahan in the spectral norm,
    # ||sin Theta||_2 <= ||A V - V diag(lam)||_2 / delta, delta the distance of
    # the returned values to the nearest eigenvalue outside the interval (the
    # stored spectrum); host FP64, outside the timed region
    if mf == len(ref) and g.get("neighbours"):
        vec = evecs[:mf].cpu().numpy().T
        a_sp = lap.scipy()
        res_blk = a_sp @ vec - vec * ev
        r2 = float(np.sqrt(max(np.linalg.eigvalsh(res_blk.T @ res_blk).max(), 0.0)))
        delta = float(min(abs(o - ev).min() for o in g["neighbours"][:1]))
        line["parity"]["sin_theta_bound"] = r2 / delta
        line["parity"]["sin_theta_gate"] = 1e-6 if prec == R.RAFEAST_MIXED else 1e-8
        line["parity"]["sin_theta_how"] = ("Davis-Kahan: ||A V - V diag(lam)||_2 / gap to the "
                                           "nearest eigenvalue outside the interval")
    if key.startswith("rgg"):
        line["parity"]["max_abs_err_vs_arpack"] = (float(np.max(np.abs(np.sort(ev) - ref)))
                                                   if mf == len(ref) else None)
        line["table"] = _rgg_table(R, h, torch, stream, g, cfg, evals)

    # FP64 comparison (same workload, same stream; one untimed-warm step)
    if not args.no_fp64 and prec == R.RAFEAST_MIXED:
        step(R.RAFEAST_FP64)
        f0 = torch.cuda.Event(enable_timing=True)
        f1 = torch.cuda.Event(enable_timing=True)
        f0.record(stream)
        mf64, info64 = step(R.RAFEAST_FP64)
        f1.record(stream)
        torch.cuda.synchronize()
        ev64 = evals.cpu().numpy()[:mf64]
        line["fp64"] = {"ms_per_step": f0.elapsed_time(f1), "outer_iters": info64.outer_iters,
                        "cocg_iters_total": info64.cocg_iters_total,
                        "max_eig_relerr_vs_arpack":
                            float(np.max(np.abs(np.sort(ev64) - ref) / np.abs(ref)))
                            if mf64 == len(ref) else None}
    # plain FEAST in FP64 (Algorithm 1: random start, N_c = 8, COCG to 1e-10,
    # to outer convergence), the standard-FEAST row of the paper's Table 1 on
    # this workload, one timed run. Its N_c = 8 half-contour ends close to the
    # spectrum; the multi-shift recurrence breaks down there on the kNN
    # graph, so it runs one COCG per shift (minutes: opt-in).
    if args.plain and prec == R.RAFEAST_MIXED:
        pprm = R.make_params(lmin, lmax, m0, 8, 1.0, 1e-10, cfg.outer_tol, cfg.max_outer, 20000,
                             R.RAFEAST_FP64, R.RAFEAST_FORM_CORRECTION, R.RAFEAST_START_RANDOM,
                             cfg.seed)
        R.rafeast_set_option(h, R.RAFEAST_OPT_SOLVER, 0)
        p0 = torch.cuda.Event(enable_timing=True)
        p1 = torch.cuda.Event(enable_timing=True)
        p0.record(stream)
        stp, mfp, infop = R.rafeast_solve(h, pprm, evals, None, None)
        p1.record(stream)
        torch.cuda.synchronize()
        evp = evals.cpu().numpy()[:mfp]
        line["fp64_plain"] = {
            "method": "plain FEAST FP64: random start, N_c=8, one COCG per shift to 1e-10",
            "ms_per_step": p0.elapsed_time(p1), "status": stp, "outer_iters": infop.outer_iters,
            "cocg_iters_total": infop.cocg_iters_total,
            "max_eig_relerr_vs_arpack": float(np.max(np.abs(np.sort(evp) - ref) / np.abs(ref)))
            if mfp == len(ref) else None,
            "mixed_speedup": p0.elapsed_time(p1) / ms_step}
    R.rafeast_destroy(h)

    # end to end through the C ABI with host buffers (pinned), copies inside
    if not args.no_e2e:
        hrp = torch.from_numpy(lap.row_ptr).pin_memory()
        hci = torch.from_numpy(lap.col_idx).pin_memory()
        hva = torch.from_numpy(lap.values).pin_memory()
        oev = np.zeros(m0)
        ove = np.zeros((m0, n))
        ore = np.zeros(m0)
        bi = hrp.numel() * 4 + hci.numel() * 4 + hva.numel() * 8
        bo = oev.nbytes + ove.nbytes + ore.nbytes
        ek = max(1, min(args.steps, 2))

        def e2e_step():
            hh = R.rafeast_create(hrp.numpy(), hci.numpy(), hva.numpy(), lap.shift)
            try:
                R.rafeast_warmstart(hh, lmin, lmax, m0, cfg.p, cfg.q, cfg.seed)
                st, _, _ = solve(hh, params(prec), oev, ove, ore)
                assert st == R.RAFEAST_OK
            finally:
                R.rafeast_destroy(hh)

        e2e_step()
        torch.cuda.synchronize()
        if dist:
            dist.barrier()
        t0 = time.perf_counter()
        for _ in range(ek):
            e2e_step()
        torch.cuda.synchronize()
        el = time.perf_counter() - t0
        el = max_over_ranks(el, dist, dev)
        line["e2e"] = {"value": ek / el if sharded else ek * world / el, "unit": "solves/s",
                       "h2d_bytes_per_step": bi,
                       "d2h_bytes_per_step": bo, "steps": ek,
                       "includes": "rafeast_create from pinned host CSR (row reorder on the "
                                   "host), warmstart, solve, copy of eigenpairs to host"}

    if not args.no_cpu and rank == 0 and world == 1:
        counts = dict(outer=info.outer_iters, cocg_total=info.cocg_iters_total)
        d = _cpu_sample(key, counts)
        if "est" in d:
            line["cpu_baseline"] = {
                "value": 1.0 / d["est"], "unit": "solves/s", "cores": 1, "kind": "oracle",
                "sample": (f"oracle warmstart + {d['steps']} COCG steps of one shift on the full "
                           f"matrix ({d['t_step']:.3f} s/step) + one Rayleigh-Ritz "
                           f"({d['t_rr']:.2f} s), extrapolated to this run's "
                           f"{counts['outer']} outer and {counts['cocg_total']} COCG iterations "
                           f"x {cfg.nc} shifts; {d['wall_s']:.1f} s of CPU work"),
                "est_seconds_per_solve": d["est"]}
        else:
            line["cpu_baseline"] = {"error": d.get("error")}
        # the same oracle with every host core as BLAS threads (its sparse
        # products and vector updates stay single-threaded)
        cores = os.cpu_count() or 1
        d = _cpu_sample(key, counts, threads=cores)
        if "est" in d:
            line["cpu_baseline_all_cores"] = {
                "value": 1.0 / d["est"], "unit": "solves/s", "cores": cores, "kind": "oracle",
                "sample": f"as cpu_baseline with {cores} BLAS threads; {d['wall_s']:.1f} s of CPU work",
                "est_seconds_per_solve": d["est"]}
    if rank == 0:
        print(json.dumps(line))
    if dist:
        dist.destroy_process_group()
    return 0


if __name__ == "__main__":
    sys.exit(main())
