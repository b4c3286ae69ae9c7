#!/usr/bin/env python
"""Trace-ratio throughput of the Krylov local-trace engine on one or more GB300s.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

Workload (five-orbital model, Sec. IV-V parameters): n=5, U=4, J=1, U'=U-2J,
crystal field Uniform[-0.05, 0.05], mu = 4.5U - 10J, beta = 50, Krylov
tolerance 1e-12; 4,096 walkers with per-flavor orders Poisson(6) (capped at
40); one proposed insert/remove move per walker per step (rounds of moves with
seeds 1000 + r; the walkers' configurations are not advanced). A step is one
trace-ratio evaluation of every walker's move: validation and move editing,
structural pruning, the trace of every surviving (walker, kept state) pair in
the block eigenbasis and the reduction to sign and log-ratio, one kernel. Inputs are resident in HBM; L2
is flushed (256 MiB write) before every timed step. Each rank runs its own
4,096 walkers (weak scaling); there is no data-path collective.

Prints one JSON line (rank 0). The FP32 path (KT_FP32_KRYLOV) is the headline; the plain
FP64 GPU path is timed on the same rounds (key "fp64_gpu"). Key "sweep": full
CT-HYB sweeps of the same model (semicircular bath, 1,024 chains, beta 50 by
default) through kt_sweep, FP32 and FP64 traces; --details FILE has all of its figures.
"""
from __future__ import annotations

import argparse
import hashlib
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

METRIC = "5-orbital trace-ratio evals/s (batched FP32) vs plain FP64 GPU; rel err ≤1e-5"
METRIC_7 = "7-orbital trace-ratio evals/s (batched FP32) vs plain FP64 GPU; rel err ≤1e-5"
UNIT = "evals/s"
N_WALKERS = 4096
N_ROUNDS = 200
SM_COUNT_GB300 = 152
FP32_LANES_PER_SM = 128
FP64_FMA_PER_SM_CLK = 2  # 1.25 TFLOP/s nominal / (152 SMs x 2.07 GHz x 2 flops)
MEASURED_FP32_TFLOPS = 66.9  # FP32 FMA-chain microbenchmark on this GPU type (every lane of a full grid)


def args_():
    p = argparse.ArgumentParser()
    p.add_argument("--gpus", type=int, default=1)
    p.add_argument("--steps", type=int, default=400)
    p.add_argument("--warmup", type=int, default=5)
    p.add_argument("--impl", choices=["ours", "reference"], default="ours")
    p.add_argument("--fp64-steps", type=int, default=0, help="steps for the FP64 comparator (default min(K, 100))")
    p.add_argument("--no-cpu-baseline", action="store_true")
    p.add_argument("--cpu-seconds", type=float, default=10.0, help="target CPU time of the oracle sample")
    p.add_argument("--sweep-steps", type=int, default=3000,
                   help="timed Metropolis steps of the CT-HYB sweep line (0 skips it)")
    p.add_argument("--sweep-beta", type=float, default=50.0)
    p.add_argument("--da-tries", type=int, default=DA_TRIES,
                   help="proposals per chain and call step of the multi-try delayed-acceptance sweep lines")
    p.add_argument("--sweep-other-steps", type=int, default=500,
                   help="timed steps of the lighter sweep lines at beta 10 and 100")
    p.add_argument("--no-other-betas", action="store_true", help="skip the beta 10 and 100 sweep lines")
    p.add_argument("--no-seven", action="store_true", help="skip the seven-orbital sub-dict of the default run")
    p.add_argument("--workload", choices=["five_orbital", "seven_orbital"], default="five_orbital",
                   help="five_orbital (4,096 walkers, the headline) or seven_orbital (256 walkers)")
    p.add_argument("--details", default=None, help="file for every figure of the run (JSON; the line has a summary of the sweeps)")
    p.add_argument("--trunc-eps", type=float, default=None,
                   help="truncation threshold of the outer trace (default: the workload's, 1e-10)")
    return p.parse_args()


def dist_env():
    return int(os.environ.get("RANK", 0)), int(os.environ.get("LOCAL_RANK", 0)), int(os.environ.get("WORLD_SIZE", 1))


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled every 200 ms during the timed region."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.f = tempfile.NamedTemporaryFile("w+", suffix=".csv", delete=False)
        self.p = None

    def start(self):
        try:
            self.p = subprocess.Popen(["nvidia-smi", f"--id={self.gpu}", f"--query-gpu={self.Q}", "--format=csv,noheader,nounits",
                                       "-lms", "200"], stdout=self.f, stderr=subprocess.DEVNULL)
        except OSError:
            self.p = None
        self.t0 = time.time()

    def stop(self):
        self.t1 = time.time()
        if self.p is not None:
            self.p.terminate()
            try:
                self.p.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.p.kill()
        self.f.flush()
        rows = []
        with open(self.f.name) as fh:
            for line in fh:
                parts = [x.strip() for x in line.split(",")]
                if len(parts) >= 9:
                    rows.append(parts)
        os.unlink(self.f.name)
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"], "samples": 0}
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4) if r[5 + i].lower().startswith("active")})
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(rows)}


ROOFLINE_DEFINITION = ("one dense product of two blocks per propagated interval (kt_stats.intervals of a counted call "
                       "times 2 d^2, the mean over the blocks) / time")
ITEMS_SOURCES = ("kt_internal.h", "kt_device.cuh", "kt_eig.cuh", "kt_eig_f32.cu")


def trim_hist(h):
    """Krylov-dimension histogram {p: propagations} without the empty bins (the last bin
    counts every p at or above it)."""
    return {str(p) if p < len(h) - 1 else f">={p}": c for p, c in enumerate(h) if c}


def source_sha() -> str:
    """Hash of the sources the FP32 kernel of a ratio call is compiled from (ties the committed
    ncu traffic record of that kernel to its code)."""
    h = hashlib.sha256()
    d = os.path.join(ROOT, "paper_0908_0681_gb300", "csrc")
    for f in ITEMS_SOURCES:
        h.update(f.encode())
        h.update(open(os.path.join(d, f), "rb").read())
    return h.hexdigest()[:16]


def mean_block_square(n_orb: int) -> float:
    """Mean squared size of the invariant blocks (n_up, n_dn, singly occupied orbitals)."""
    import numpy as np

    x = np.arange(4 ** n_orb)
    up, dn = [(x >> 2 * a) & 1 for a in range(n_orb)], [(x >> 2 * a + 1) & 1 for a in range(n_orb)]
    mask = sum((up[a] ^ dn[a]) << a for a in range(n_orb))
    d = np.unique((sum(up) * (n_orb + 1) + sum(dn)) * 2 ** n_orb + mask, return_counts=True)[1]
    return float((d * d).sum()) / len(d)


def measured_traffic(sha: str):
    """dram read+write bytes per launch of that kernel from a committed ncu summary, if it
    was taken on the current kernel source; else None."""
    p = os.path.join(ROOT, "profiles", "items_kernel_traffic.json")
    try:
        d = json.load(open(p))
    except (OSError, ValueError):
        return None
    return d.get("dram_bytes_per_launch") if d.get("source_sha") == sha else None


WALKERS = {"five_orbital": 4096, "seven_orbital": 256}


def rank_seeds(rank: int, rounds: int):
    """Per-rank seeds: each rank (replica) draws its own walkers and moves."""
    return 1 + 7919 * rank, [1000 + r + 100000 * rank for r in range(rounds)]


def aggregate(times_ms, n_per_rank: int, steps: int, world: int, reduce_max=None):
    """Whole-job throughput of weak-scaled replicas: units of all ranks / max time over ranks.

    times_ms: this rank's [timed total, ...] in ms; reduce_max: callable doing an element-wise
    max over ranks (None for one rank). Returns (value, max_times)."""
    t = list(times_ms)
    if world > 1 and reduce_max is not None:
        t = reduce_max(t)
    return world * n_per_rank * steps / (t[0] / 1000.0), t


def make_workload(rank: int, rounds: int, name: str = "five_orbital", trunc_eps: float | None = None):
    from paper_0908_0681_gb300 import workloads
    w = workloads.WORKLOADS[name]() if trunc_eps is None else workloads.WORKLOADS[name](trunc_eps=trunc_eps)
    seq_seed, move_seeds = rank_seeds(rank, rounds)
    seqs = workloads.generate_sequences(w, WALKERS[name], seed=seq_seed)
    moves = [workloads.generate_moves(w, seqs, seed=sd) for sd in move_seeds]
    return w, seqs, moves


def cpu_baseline(w, seqs, moves_list, gpu_ratio_round0, seconds: float):
    """Time the oracle (as it stands) on a bounded sample of the same workload on the host cores.
    gpu_ratio_round0: {name: (sign, logratio, current sign, current log|T|)} of GPU paths on the
    first timed round, each ratio formed against that path's own current traces. Reported: the
    largest relative error of those ratios against the oracle's ratios, and of every trace, current
    and proposed, against the oracle's."""
    import numpy as np
    from oracle.oracle import Model, Params, SeqBatch, classify, ratio

    spec = w.model
    P = Params(spec.n_orb, spec.U, spec.J, Up=spec.up, mu=spec.mu, delta=spec.delta, beta=spec.beta,
               trunc_eps=spec.trunc_eps, deg_tol=spec.deg_tol)
    o = Model(P)
    sb = SeqBatch(seqs.offsets, seqs.tau, seqs.flavor, seqs.dagger)
    cs, cl, _ = o.trace(sb)
    done, t_used, evals = 0, 0.0, 0
    errs = []
    r = 0
    while t_used < seconds and r < len(moves_list):
        mv = moves_list[r].as_dict()
        t0 = time.perf_counter()
        sgn, lr, ns, nl = ratio(o, sb, cs, cl, mv)
        t_used += time.perf_counter() - t0
        evals += seqs.n
        if r == 0 and gpu_ratio_round0:
            ok = (sgn != 0) & np.isfinite(lr)
            okc = cs != 0
            errs = {name: float(np.abs(np.expm1(v[1][ok] - lr[ok])).max()) for name, v in gpu_ratio_round0.items()}
            sign_ok = {name: bool((v[0] == sgn).all() and (v[2] == cs).all()) for name, v in gpu_ratio_round0.items()}
            terrs = {name: float(max(np.abs(np.expm1(v[3][okc] - cl[okc])).max(),
                                     np.abs(np.expm1((v[3] + v[1])[ok] - (cl + lr)[ok])).max()))
                     for name, v in gpu_ratio_round0.items()}
        r += 1
    out = {"value": evals / t_used, "unit": UNIT, "cores": int(o.threads_used), "kind": "oracle",
           "sample": f"{r} round(s) x {seqs.n} walkers of the same workload (FP64 dense-block oracle, OpenMP)"}
    if errs:
        out["max_rel_err_fp32_vs_oracle"] = errs.get("fp32")
        out["max_rel_err_vs_oracle"] = errs
        out["signs_equal"] = sign_ok
        out["max_rel_err_traces_vs_oracle"] = terrs
        out["error_definition"] = ("round 0, all walkers: |T_new/T_cur - 1| relative to the oracle ratio, the GPU ratio "
                                   "formed against the GPU path's own current traces (two evaluations, bound 2e-5 for "
                                   "FP32); traces: every current and proposed trace against the oracle's (bound 1e-5)")
    return out


def reference_arm(a):
    """Oracle timed on the host cores, on bounded samples of the same workload."""
    rank, _, world = dist_env()
    if rank != 0:
        return
    import numpy as np
    from oracle.oracle import Model, Params, SeqBatch, ratio

    w, seqs, moves = make_workload(0, min(N_ROUNDS, a.warmup + a.steps), a.workload, a.trunc_eps)
    spec = w.model
    P = Params(spec.n_orb, spec.U, spec.J, Up=spec.up, mu=spec.mu, delta=spec.delta, beta=spec.beta,
               trunc_eps=spec.trunc_eps, deg_tol=spec.deg_tol)
    o = Model(P)
    sample = min(256, seqs.n)
    sub = seqs.subset(range(sample))
    sb = SeqBatch(sub.offsets, sub.tau, sub.flavor, sub.dagger)
    cs, cl, _ = o.trace(sb)

    def mv_sub(m):
        return {k: v[:sample] for k, v in m.as_dict().items()}

    for i in range(a.warmup):
        ratio(o, sb, cs, cl, mv_sub(moves[i % len(moves)]))
    t0 = time.perf_counter()
    for i in range(a.steps):
        ratio(o, sb, cs, cl, mv_sub(moves[(a.warmup + i) % len(moves)]))
    dt = time.perf_counter() - t0
    v = sample * a.steps / dt
    line = {"impl": "reference", "metric": METRIC if a.workload == "five_orbital" else METRIC_7, "value": v, "unit": UNIT, "n_gpus": a.gpus, "steps": a.steps,
            "warmup": a.warmup, "ms_per_step": 1000 * dt / a.steps, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": f"{a.workload}_{seqs.n}_walkers", "n_orb": spec.n_orb, "walkers": seqs.n,
                       "beta": spec.beta, "sample_walkers_per_step": sample},
            "cpu_baseline": {"value": v, "unit": UNIT, "cores": int(o.threads_used), "kind": "oracle",
                             "sample": f"{sample} of {seqs.n} walkers per step, FP64 dense-block oracle, OpenMP"},
            "e2e": {"value": v, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


CACHE_OPS = 512   # partial-state cache length of the cached sweeps (operators per walker)
DA_TRIES = 8      # proposals per chain and call step of the multi-try delayed-acceptance sweeps (--da-tries)
# multi-try delayed-acceptance call steps (with the partial-state cache) at the end of the
# sweeps' thermalisation: about 8 10^4 Metropolis steps per chain, where the expansion order
# has stopped drifting (shorter starts left it several standard errors above its equilibrium)
THERM_DA_CALL_STEPS = 20000
LONG_PLAIN_STEPS = 12000    # Metropolis steps per chain of the longer cached comparison


def chain_estimates(acc, n_orb: int, beta: float, n_bins: int):
    """Per-chain estimates from sweep accumulators: double occupancy (mean over orbitals),
    expansion order (sum over flavors), n_f [chains][flavors] (flavor f = 2a + s), the orbital
    occupations n_a = n_{a up} + n_{a dn} [chains][orbitals] and G(tau) [chains][bins] (mean over
    flavors), each divided by the chain's sign sum."""
    ssum = acc["sign_sum"]
    obs = acc["obs_sum"] / ssum[:, None]
    nf = obs[:, :2 * n_orb]
    return {"docc": obs[:, 2 * n_orb: 3 * n_orb].mean(1), "order": acc["order_sum"].sum(1) / ssum,
            "n_f": nf, "n_orbital": nf[:, 0::2] + nf[:, 1::2],
            "G_tau": acc["g_tau"].mean(1) * (n_bins / beta ** 2) / ssum[:, None]}


def efficiencies(est, secs: float):
    """Statistical efficiency 1 / (variance across independent chains x wall time) of every
    observable (n_f per flavor, n_a per orbital, G(tau) per bin), and of G(tau) pooled over its
    bins (1 / (sum of the bins' variances x wall time))."""
    var = {k: v.var(axis=0, ddof=1) for k, v in est.items()}
    out = {k: (1.0 / (v * secs)) for k, v in var.items()}
    out["G_tau_pooled"] = 1.0 / (float(var["G_tau"].sum()) * secs)
    return out


def speedups(ea, eb):
    """Speedups at equal statistical error of path a over path b: ratios of efficiencies; for
    n_f, n_a and G(tau) the smallest over flavors, orbitals and bins, the median over bins and
    the ratio pooled over bins. A smallest ratio over many noisy ratios sits below their common
    value (each ratio of two variances over 1,024 chains carries about 6% noise)."""
    import numpy as np
    out = {"docc": float(ea["docc"] / eb["docc"]), "order": float(ea["order"] / eb["order"])}
    rf = np.asarray(ea["n_f"] / eb["n_f"])
    ro = np.asarray(ea["n_orbital"] / eb["n_orbital"])
    rg = np.asarray(ea["G_tau"] / eb["G_tau"])
    out["n_f_min_over_flavors"] = float(rf.min())
    out["n_orbital_min_over_orbitals"] = float(ro.min())
    out["G_tau_min_over_bins"] = float(rg.min())
    out["G_tau_median_over_bins"] = float(np.median(rg))
    out["G_tau_pooled"] = float(ea["G_tau_pooled"] / eb["G_tau_pooled"])
    return out


def sweep_beta_light(dev, beta: float, steps: int, seed: int):
    """CT-HYB sweeps of the five-orbital model at another beta (1,024 chains, semicircular bath):
    chains from Poisson(6) starts thermalise untimed with FP32 traces; from the same state
    `steps` steps are timed for FP32, FP32 with the partial-state cache and FP64 traces, measuring
    every 50 steps. Efficiencies at equal error cover double occupancy, the order, every n_f and
    G(tau) on every bin. The step's roofline fraction counts the products of its trace ratios
    (ROOFLINE_DEFINITION, intervals of 50 untimed steps) against the FP32 peak."""
    import numpy as np
    import torch

    from paper_0908_0681_gb300 import engine, kt, workloads

    nw, therm, meas, n_bins = 1024, 1500, 50, 200
    w = workloads.five_orbital()
    spec = workloads.five_orbital_sweep(beta).model
    gen = workloads.Workload(w.name, spec, start=w.start, order=w.order, lam=w.lam, cap=w.cap,
                             pattern_singles=w.pattern_singles)
    cand = workloads.generate_sequences(gen, 2 * nw, seed=seed)
    table = workloads.semicircular_hybridization(beta, 2 * spec.n_orb, n_tau=2000)
    g = torch.Generator(device=dev).manual_seed(seed)
    models = {"fp32": engine.model_from_spec(spec, precision=kt.KT_FP32_KRYLOV),
              "fp64": engine.model_from_spec(spec, precision=kt.KT_FP64)}
    sg, _, _ = engine.trace(models["fp32"], engine.DeviceSeqs.from_host(cand, dev))
    ok = np.nonzero(sg.cpu().numpy() != 0)[0][:nw]
    base = engine.Sweep(models["fp32"], table, beta, nw, k_cap=128, n_bins=n_bins, measure_obs=True)
    base.set_configs(cand.subset(ok))
    for _ in range(0, therm, 500):
        base.run(torch.rand((500, nw, 6), dtype=torch.float64, device=dev, generator=g))
    st = {k: v.cpu().numpy() for k, v in base.state().items()}
    lens = st["lens"]
    thermal = workloads.Sequences(np.concatenate([[0], np.cumsum(lens)]).astype(np.int32),
                                  np.concatenate([st["tau"][i, :lens[i]] for i in range(nw)]),
                                  np.concatenate([st["flavor"][i, :lens[i]] for i in range(nw)]),
                                  np.concatenate([st["dagger"][i, :lens[i]] for i in range(nw)]))
    del base
    steps = max(meas, steps - steps % meas)
    u = torch.rand((steps, nw, 6), dtype=torch.float64, device=dev, generator=g)
    mhz = 2070.0
    peak32 = SM_COUNT_GB300 * FP32_LANES_PER_SM * 2 * mhz * 1e6 / 1e12
    out, eff = {}, {}
    for name, model, cache in (("fp32", models["fp32"], 0), ("fp32_cached", models["fp32"], CACHE_OPS),
                               ("fp64", models["fp64"], 0)):
        sw = engine.Sweep(model, table, beta, nw, k_cap=128, n_bins=n_bins, measure_obs=True, cache_ops=cache)
        sw.set_configs(thermal)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        sw.run(u, meas_every=meas)
        e1.record()
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1)
        cnt = sw.counters()
        acc = {k: v.cpu().numpy() for k, v in sw.accumulators().items()}
        est = chain_estimates(acc, spec.n_orb, beta, n_bins)
        eff[name] = efficiencies(est, ms / 1000.0)
        stt = sw.state()
        K = stt["lens"].double().mean().item()
        wst = engine.new_stats(dev)
        sw.set_stats(wst)
        sw.run(u[:50])
        sw.set_stats(None)
        wk = kt.stats_from_tensor(wst)
        flops_step = wk["intervals"] / 50 * 2 * mean_block_square(spec.n_orb)
        props = nw * steps / (ms / 1000.0)
        out[name] = {"proposals_per_s": props, "ms_per_step": ms / steps, "sweeps_per_s": props / K,
                     "mean_ops_per_chain": K, "mean_order_per_flavor": stt["order"].double().mean().item(),
                     "acceptance": (cnt["insert_accepted"] + cnt["remove_accepted"]) / (nw * steps),
                     "mean_sign": float(acc["sign_sum"].sum() / (nw * cnt["measurements"])) if cnt["measurements"] else None,
                     "trace_errors": cnt["trace_errors"], "docc": float(est["docc"].mean()),
                     "n_f": float(est["n_f"].mean()), "order": float(est["order"].mean()),
                     "krylov_intervals_per_proposal": wk["intervals"] / (50 * nw),
                     "roofline": {"bound": "alu", "achieved": flops_step / (ms / steps / 1000.0) / 1e12,
                                  "peak": peak32, "unit": "TFLOP/s",
                                  "frac": flops_step / (ms / steps / 1000.0) / 1e12 / peak32,
                                  "definition": ROOFLINE_DEFINITION}}
        del sw
    sp = {f"{a_}_over_{b_}": speedups(eff[a_], eff[b_]) for a_, b_ in (("fp32", "fp64"), ("fp32_cached", "fp64"),
                                                                        ("fp32_cached", "fp32"))}
    return {"workload": f"five_orbital_sweep_beta{beta:g}_1024_chains", "beta": beta, "thermalisation_steps": therm,
            "measure_every": meas, "steps": steps, **out, "speedup_at_equal_error": sp}


def seven_bench(dev, K: int):
    """The seven-orbital batch (256 walkers, N_tr = 63, beta 40): FP32 and FP64
    trace-ratio evaluations per second (L2 flushed before every step) and the largest relative
    error of each path's ratios, formed against its own current traces, against the oracle's
    ratios on the first round."""
    import numpy as np
    import torch

    from oracle.oracle import Model, Params, SeqBatch, ratio
    from paper_0908_0681_gb300 import engine, kt

    w, seqs, moves = make_workload(0, K + 3, "seven_orbital")
    spec = w.model
    n = seqs.n
    d = engine.DeviceSeqs.from_host(seqs, dev)
    dm = [engine.DeviceMoves.from_host(m, dev) for m in moves]
    flush = torch.empty(64 * 1024 * 1024, dtype=torch.int32, device=dev)
    stream = torch.cuda.current_stream()
    res, round0 = {}, {}
    for name, prec in (("fp32", kt.KT_FP32_KRYLOV), ("fp64", kt.KT_FP64)):
        m = engine.model_from_spec(spec, precision=prec)
        ws = engine.workspace(m, n, dev)
        cs, cl, _ = engine.trace(m, d, ws=ws)
        o = (torch.empty(n, dtype=torch.int8, device=dev), torch.empty(n, dtype=torch.float64, device=dev),
             torch.empty(n, dtype=torch.int32, device=dev))
        kt.kt_trace_ratio(m, d.batch(), cs, cl, dm[0].batch(), *o, None, ws, stream)
        torch.cuda.synchronize()
        round0[name] = (o[0].cpu().numpy(), o[1].cpu().numpy(), cs.cpu().numpy(), cl.cpu().numpy())
        for k in range(3):
            kt.kt_trace_ratio(m, d.batch(), cs, cl, dm[k % len(dm)].batch(), *o, None, ws, stream)
        tot = 0.0
        for k in range(K):
            flush.zero_()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            kt.kt_trace_ratio(m, d.batch(), cs, cl, dm[(3 + k) % len(dm)].batch(), *o, None, ws, stream)
            e1.record(stream)
            torch.cuda.synchronize()
            tot += e0.elapsed_time(e1)
        res[name] = {"value": n * K / (tot / 1000.0), "unit": UNIT, "ms_per_step": tot / K}
    P = Params(spec.n_orb, spec.U, spec.J, Up=spec.up, mu=spec.mu, delta=spec.delta, beta=spec.beta,
               trunc_eps=spec.trunc_eps, deg_tol=spec.deg_tol)
    om = Model(P)
    sb = SeqBatch(seqs.offsets, seqs.tau, seqs.flavor, seqs.dagger)
    ocs, ocl, _ = om.trace(sb)
    osg, olr, _, _ = ratio(om, sb, ocs, ocl, moves[0].as_dict())
    okr = (osg != 0) & np.isfinite(olr)
    okc = ocs != 0
    for name, (gs, gl, gcs, gcl) in round0.items():
        er = np.abs(np.expm1(gl[okr] - olr[okr]))
        res[name]["max_rel_err_vs_oracle"] = float(er.max())
        res[name]["signs_equal"] = bool((gs == osg).all() and (gcs == ocs).all())
        res[name]["walkers_above_1e-5"] = int((er > 1e-5).sum())
        # each trace on its own (the 1e-5 bar of one FP32 evaluation): current and proposed
        ec = np.abs(np.expm1(gcl[okc] - ocl[okc]))
        en = np.abs(np.expm1((gcl + gl)[okr] - (ocl + olr)[okr]))
        res[name]["max_rel_err_traces_vs_oracle"] = float(max(ec.max(), en.max()))
        res[name]["traces_above_1e-5"] = int((ec > 1e-5).sum() + (en > 1e-5).sum())
    return {"workload": f"seven_orbital_{n}_walkers", "metric": METRIC_7, "steps": K, "n_kept": om.nkept,
            "error_definition": "round 0, all walkers: ratios against the path's own current traces vs the FP64 oracle "
                                "(two FP32 evaluations, bound 2e-5); traces, current and proposed, each vs the oracle "
                                "(bound 1e-5)",
            **res, "speedup_fp32_over_fp64": res["fp32"]["value"] / res["fp64"]["value"]}


def sweep_bench(dev, steps: int, beta: float, seed: int):
    """Full CT-HYB sweeps of the five-orbital model (semicircular bath, 2,000 tau points,
    1,024 chains). Chains start from Poisson(6) configurations and thermalise untimed
    (FP32 traces). The surrogate is trained on the chains' own ratios
    (kt_sweep_collect, then Adam on the tensor cores). From the same thermalised state,
    `steps` Metropolis steps are then timed with CUDA events for plain FP32
    sweeps, delayed-acceptance FP32 sweeps and plain FP64 sweeps,
    measuring G(tau), the orders and the beta/2 observables every 50 steps.

    Statistical efficiency at equal error: for an observable O the per-chain estimates
    have a variance s2 across the 1,024 independent chains after wall time t; the time
    needed for a given error scales as s2 * t, so eff = 1 / (s2 t) and the ratios of eff
    between paths are the speedups at equal statistical error."""
    import numpy as np
    import torch

    from paper_0908_0681_gb300 import engine, kt, workloads

    nw, therm, meas, ncollect = 1024, 2000, 50, 1000
    w = workloads.five_orbital()
    spec = workloads.five_orbital_sweep(beta).model
    gen = workloads.Workload(w.name, spec, start=w.start, order=w.order, lam=w.lam, cap=w.cap,
                             pattern_singles=w.pattern_singles)
    cand = workloads.generate_sequences(gen, 2 * nw, seed=seed)
    table = workloads.semicircular_hybridization(beta, 2 * spec.n_orb, n_tau=2000)
    g = torch.Generator(device=dev).manual_seed(seed)

    def uni(n, k):
        return torch.rand((n, nw, k), dtype=torch.float64, device=dev, generator=g)

    models = {name: engine.model_from_spec(spec, precision=prec)
              for name, prec in (("fp32", kt.KT_FP32_KRYLOV), ("fp64", kt.KT_FP64))}
    sg, _, _ = engine.trace(models["fp32"], engine.DeviceSeqs.from_host(cand, dev))
    ok = np.nonzero(sg.cpu().numpy() != 0)[0][:nw]
    # thermalisation (untimed), with the partial-state cache: plain steps, the surrogate's
    # training steps, then multi-try delayed-acceptance steps, the fastest route to many
    # Metropolis steps per chain
    base = engine.Sweep(models["fp32"], table, beta, nw, k_cap=128, n_bins=200, measure_obs=True, cache_ops=CACHE_OPS)
    base.set_configs(cand.subset(ok))
    for _ in range(0, therm, 500):
        base.run(uni(500, 6))
    # the surrogate: training data from the chains themselves, then Adam on the tensor cores
    torch.cuda.synchronize()
    t0 = time.time()
    X, t = base.collect(uni(ncollect, 6), capacity=nw * ncollect)
    torch.cuda.synchronize()
    t_collect = time.time() - t0
    # targets clipped to where the acceptance test can go either way (the chain stays exact
    # for any surrogate; accuracy only matters near log ratio 0)
    t = t.clamp(-25.0, 10.0)
    net = engine.Surrogate(base.n_features, max_batch=max(8192, DA_TRIES * nw), seed=seed)
    t0 = time.time()
    hist = net.train(X, t, epochs=10, batch=4096, lr=3e-3, seed=seed)
    hist += net.train(X, t, epochs=10, batch=4096, lr=1e-3, seed=seed + 1)
    torch.cuda.synchronize()
    t_train = time.time() - t0
    pred = net.predict(X[:65536]).double()
    resid = float(torch.sqrt(torch.mean((pred - t[:65536].double()) ** 2)).item())
    spread = float(torch.std(t[:65536].double()).item())
    n_train = int(X.shape[0])
    del X, t
    base.set_surrogate(net)
    for _ in range(0, THERM_DA_CALL_STEPS, 500):
        base.run_da_multi(torch.rand((500, nw, DA_TRIES, 7), dtype=torch.float64, device=dev, generator=g))
    cth = base.counters()
    therm_mh = cth["insert_proposed"] + cth["remove_proposed"]
    st = {k: v.cpu().numpy() for k, v in base.state().items()}
    lens = st["lens"]
    thermal = workloads.Sequences(np.concatenate([[0], np.cumsum(lens)]).astype(np.int32),
                                  np.concatenate([st["tau"][i, :lens[i]] for i in range(nw)]),
                                  np.concatenate([st["flavor"][i, :lens[i]] for i in range(nw)]),
                                  np.concatenate([st["dagger"][i, :lens[i]] for i in range(nw)]))
    del base

    out = {}
    per_chain = {}
    effs = {}
    mhz = 2070.0
    peak32 = SM_COUNT_GB300 * FP32_LANES_PER_SM * 2 * mhz * 1e6 / 1e12
    steps = max(meas, steps - steps % meas)   # whole measurement blocks
    n_blocks = steps // meas
    u_plain = uni(steps, 6)      # the FP32 and FP64 plain runs share their uniforms
    u_da = uni(steps, 7)         # and so do the delayed-acceptance runs
    u_multi = None
    for name, model, mode, n_t, cache in (("fp32", models["fp32"], "plain", steps, 0),
                                          ("fp32_da", models["fp32"], "da", steps, 0),
                                          ("fp32_da_multi", models["fp32"], "multi", steps, 0),
                                          ("fp64", models["fp64"], "plain", steps, 0),
                                          ("fp32_cached", models["fp32"], "plain", steps, CACHE_OPS),
                                          ("fp32_da_cached", models["fp32"], "da", steps, CACHE_OPS),
                                          ("fp32_da_multi_cached", models["fp32"], "multi", steps, CACHE_OPS),
                                          ("fp64_cached", models["fp64"], "plain", steps, CACHE_OPS)):
        sw = engine.Sweep(model, table, beta, nw, k_cap=128, n_bins=200, measure_obs=True, cache_ops=cache)
        sw.set_configs(thermal)
        if mode != "plain":
            sw.set_surrogate(net)
        meas_m = meas
        if mode == "multi":
            # measure at the Metropolis-step spacing of the other lines: a call step is E[n]
            # Metropolis steps, from the stage-1 pass rate p of the one-try line
            pp = out["fp32_da"]["trace_evaluations_per_proposal"]
            en = (1.0 - (1.0 - pp) ** DA_TRIES) / pp
            meas_m = max(1, int(round(meas / en)))
            n_t = n_blocks * 3 * meas_m
            if u_multi is None or u_multi.shape[0] < n_t:
                u_multi = torch.rand((n_t, nw, DA_TRIES, 7), dtype=torch.float64, device=dev, generator=g)
        u = {"plain": u_plain, "da": u_da, "multi": u_multi[:n_t] if mode == "multi" else None}[mode]
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        blocks = sw.run_blocks(u, meas_m, n_blocks, delayed=(mode != "plain"))
        e1.record()
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1)
        cnt = sw.counters()
        # error bars: binning analysis over the measurement blocks of every chain
        series = {"docc": [], "order": [], "G_beta_half": []}
        for blk in blocks:
            bs = blk["sign_sum"].cpu().numpy()
            series["docc"].append((blk["obs_sum"].cpu().numpy()[:, 2 * spec.n_orb: 3 * spec.n_orb].mean(1)) / bs)
            series["order"].append(blk["order_sum"].cpu().numpy().sum(1) / bs)
            series["G_beta_half"].append((blk["g_tau"].cpu().numpy()[:, :, 95:105].mean(2) * (200 / beta ** 2)).mean(1) / bs)
        binning = {}
        for k, v in series.items():
            b = engine.binning_analysis(np.stack(v, axis=1))
            binning[k] = {"mean": float(np.mean(v)), "error": b["error"], "tau_int_measurements": b["tau_int"],
                          "plateau": b["plateau"],
                          "errors_by_bin_size": {str(sz): e for sz, e in b["errors"].items()}}
        del blocks
        stt = sw.state()
        acc = {k: v.cpu().numpy() for k, v in sw.accumulators().items()}
        ssum = acc["sign_sum"]
        obs = acc["obs_sum"] / ssum[:, None]
        docc = obs[:, 2 * spec.n_orb: 3 * spec.n_orb].mean(1)
        order = acc["order_sum"].sum(1) / ssum
        gmid = (acc["g_tau"][:, :, 95:105].mean(2) * (200 / beta ** 2) / ssum[:, None]).mean(1)
        K = stt["lens"].double().mean().item()
        effs[name] = efficiencies(chain_estimates(acc, spec.n_orb, beta, 200), ms / 1000.0)
        # intervals of the step's trace ratios (50 untimed, counted steps)
        wst = engine.new_stats(dev)
        sw.set_stats(wst)
        if mode == "multi":
            sw.run_da_multi(u[:50])
        elif mode == "da":
            sw.run_da(u[:50])
        else:
            sw.run(u[:50])
        sw.set_stats(None)
        flops_step = kt.stats_from_tensor(wst)["intervals"] / 50 * 2 * mean_block_square(spec.n_orb)
        del sw
        per_chain[name] = {"docc": docc, "order": order, "G_beta_half": gmid,
                           "n_f": obs[:, :2 * spec.n_orb].mean(1), "S2": obs[:, 3 * spec.n_orb],
                           "lens": stt["lens"].cpu().numpy(), "tau": stt["tau"].cpu().numpy()}
        # Metropolis steps taken (a multi-try call step is 1 to DA_TRIES of them per chain)
        n_mh = cnt["insert_proposed"] + cnt["remove_proposed"]
        props = n_mh / (ms / 1000.0)
        secs = ms / 1000.0
        out[name] = {"proposals_per_s": props, "ms_per_step": ms / n_t, "steps": n_t, "measure_every": meas_m,
                     "metropolis_steps_per_call_step": n_mh / (nw * n_t),
                     "sweeps_per_s": props / K, "mean_ops_per_chain": K,
                     "mean_order_per_flavor": stt["order"].double().mean().item(),
                     "acceptance": (cnt["insert_accepted"] + cnt["remove_accepted"]) / n_mh,
                     "trace_evaluations_per_proposal": cnt["trace_evaluations"] / n_mh,
                     "stage1_rejected_per_proposal": cnt["stage1_rejected"] / n_mh,
                     # multi-try sums carry the tries as weights, so their sign sum is no count
                     "mean_sign": (float(ssum.sum() / (nw * cnt["measurements"]))
                                   if cnt["measurements"] and mode != "multi" else None),
                     "trace_errors": cnt["trace_errors"], "refused_at_k_cap": cnt["refused_at_k_cap"],
                     "docc": float(docc.mean()), "G_beta_half": float(gmid.mean()),
                     "n_f": float(obs[:, :2 * spec.n_orb].mean()), "S2": float(obs[:, 3 * spec.n_orb].mean()),
                     "eff": {"docc": 1.0 / (docc.var(ddof=1) * secs), "order": 1.0 / (order.var(ddof=1) * secs),
                             "G_beta_half": 1.0 / (gmid.var(ddof=1) * secs)},
                     "error_bars_binning": binning,
                     "roofline": {"bound": "alu", "achieved": flops_step / (ms / n_t / 1000.0) / 1e12, "peak": peak32,
                                  "unit": "TFLOP/s", "frac": flops_step / (ms / n_t / 1000.0) / 1e12 / peak32,
                                  "flops_per_step": flops_step,
                                  "definition": ROOFLINE_DEFINITION}}
    # FP32 against FP64 on the same uniforms: chains whose final configurations agree took
    # the same decisions all along, so their accumulators differ only by the trace arithmetic
    a32, a64 = per_chain["fp32"], per_chain["fp64"]
    same = np.array([a32["lens"][i] == a64["lens"][i] and
                     np.array_equal(a32["tau"][i, :a32["lens"][i]], a64["tau"][i, :a64["lens"][i]]) for i in range(nw)])
    err32 = {"chains_on_identical_paths": int(same.sum()), "chains": nw}
    for k in ("docc", "order", "G_beta_half", "n_f", "S2"):
        d = np.abs(a32[k][same] - a64[k][same])
        err32[f"max_abs_diff_{k}"] = float(d.max()) if d.size else None

    def identical(p, q):
        a, b = per_chain[p], per_chain[q]
        return int(sum(a["lens"][i] == b["lens"][i] and np.array_equal(a["tau"][i, :a["lens"][i]], b["tau"][i, :b["lens"][i]])
                       for i in range(nw)))
    cache_same = {f"{c}_vs_{p}": identical(c, p) for c, p in (("fp32_cached", "fp32"), ("fp32_da_cached", "fp32_da"),
                                                            ("fp32_da_multi_cached", "fp32_da_multi"),
                                                            ("fp64_cached", "fp64"))}
    speed = {f"{a}_over_{b}": {k: out[a]["eff"][k] / out[b]["eff"][k] for k in out[a]["eff"]}
             for a, b in (("fp32", "fp64"), ("fp32_da", "fp64"), ("fp32_da", "fp32"), ("fp32_cached", "fp64"),
                          ("fp32_da_cached", "fp64"), ("fp32_cached", "fp32"), ("fp64_cached", "fp64"),
                          ("fp32_da_multi", "fp64"), ("fp32_da_multi", "fp32"), ("fp32_da_multi_cached", "fp64"),
                          ("fp32_da_multi_cached", "fp32_cached"))}
    # longer runs for the slow observables: with the cache, plain and multi-try delayed
    # acceptance from the same equilibrium state over about 12,000 Metropolis steps per chain
    # each, measured every ~50 Metropolis steps (the spin of the high-spin ground multiplet
    # turns over slowly, so n_f needs runs of many thousand steps to resolve its variance)
    long_run = {}
    effs_long = {}
    for name, mode in (("fp32_cached", "plain"), ("fp32_da_multi_cached", "multi")):
        sw = engine.Sweep(models["fp32"], table, beta, nw, k_cap=128, n_bins=200, measure_obs=True, cache_ops=CACHE_OPS)
        sw.set_configs(thermal)
        meas_l = meas if mode == "plain" else out["fp32_da_multi"]["measure_every"]
        chunk = (500 // meas_l) * meas_l
        n_chunks = LONG_PLAIN_STEPS // chunk if mode == "plain" else -(-LONG_PLAIN_STEPS // (4 * chunk))
        if mode == "multi":
            sw.set_surrogate(net)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(n_chunks):
            if mode == "plain":
                sw.run(uni(chunk, 6), meas_every=meas_l)
            else:
                sw.run_da_multi(torch.rand((chunk, nw, DA_TRIES, 7), dtype=torch.float64, device=dev, generator=g),
                                meas_every=meas_l)
        e1.record()
        torch.cuda.synchronize()
        secs = e0.elapsed_time(e1) / 1000.0
        cnt = sw.counters()
        acc = {k: v.cpu().numpy() for k, v in sw.accumulators().items()}
        effs_long[name] = efficiencies(chain_estimates(acc, spec.n_orb, beta, 200), secs)
        est = chain_estimates(acc, spec.n_orb, beta, 200)
        long_run[name] = {"call_steps": n_chunks * chunk, "measure_every": meas_l, "seconds": secs,
                          "metropolis_steps_per_chain": (cnt["insert_proposed"] + cnt["remove_proposed"]) / nw,
                          "order": float(est["order"].mean()),
                          "order_stderr": float(est["order"].std(ddof=1) / np.sqrt(nw)),
                          "docc": float(est["docc"].mean()), "docc_stderr": float(est["docc"].std(ddof=1) / np.sqrt(nw))}
        del sw
    long_run["speedup_at_equal_error"] = speedups(effs_long["fp32_da_multi_cached"], effs_long["fp32_cached"])
    # throughput-bound batch: 8,192 chains (the 1,024-chain batch is bound by its longest chains)
    nbig, nsteps_big = 8192, max(steps // 4, 100)

    def unib(n, k):
        return torch.rand((n, nbig, k), dtype=torch.float64, device=dev, generator=g)

    # the same network, with room for DA_TRIES proposals of every chain
    net_big = engine.Surrogate(net.n_in, max_batch=DA_TRIES * nbig, params=net.params())
    # start: the 1,024 thermalised configurations, each repeated nbig / nw times, decorrelated
    # by 2,000 multi-try call steps (about 7,600 Metropolis steps, many autocorrelation times)
    big = engine.Sweep(models["fp32"], table, beta, nbig, k_cap=128, n_bins=200, measure_obs=True, cache_ops=CACHE_OPS)
    big.set_configs(thermal.subset(np.tile(np.arange(nw), nbig // nw)))
    big.set_surrogate(net_big)
    for _ in range(0, 2000, 250):
        big.run_da_multi(torch.rand((250, nbig, DA_TRIES, 7), dtype=torch.float64, device=dev, generator=g))
    stb = {k: v.cpu().numpy() for k, v in big.state().items()}
    lb = stb["lens"]
    thermal_big = workloads.Sequences(np.concatenate([[0], np.cumsum(lb)]).astype(np.int32),
                                      np.concatenate([stb["tau"][i, :lb[i]] for i in range(nbig)]),
                                      np.concatenate([stb["flavor"][i, :lb[i]] for i in range(nbig)]),
                                      np.concatenate([stb["dagger"][i, :lb[i]] for i in range(nbig)]))
    del big
    thr = {}
    ub = {6: unib(nsteps_big, 6), 7: unib(nsteps_big, 7)}
    meas_big_m = out["fp32_da_multi"]["measure_every"]
    # the multi-try lines take as many Metropolis steps as the others (fewer call steps)
    nsteps_big_m = max(50, int(round(nsteps_big / out["fp32_da_multi"]["metropolis_steps_per_call_step"])))
    ub[(DA_TRIES, 7)] = torch.rand((nsteps_big_m, nbig, DA_TRIES, 7), dtype=torch.float64, device=dev, generator=g)
    for mode in ("plain", "da", "da_multi", "plain_cached", "da_cached", "da_multi_cached"):
        big = engine.Sweep(models["fp32"], table, beta, nbig, k_cap=128, n_bins=200, measure_obs=True,
                           cache_ops=CACHE_OPS if mode.endswith("cached") else 0)
        big.set_configs(thermal_big)
        multi = mode.startswith("da_multi")
        if mode.startswith("da"):
            big.set_surrogate(net_big if multi else net)
        u = ub[(DA_TRIES, 7)] if multi else ub[7 if mode.startswith("da") else 6]
        run = big.run_da_multi if multi else (big.run_da if mode.startswith("da") else big.run)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        run(u, meas_every=meas_big_m if multi else meas)
        e1.record()
        torch.cuda.synchronize()
        c1 = big.counters()
        ms = e0.elapsed_time(e1)
        n_mh = c1["insert_proposed"] + c1["remove_proposed"]
        # trace-pipeline work of 50 more (untimed) call steps
        wst = engine.new_stats(dev)
        big.set_stats(wst)
        run(u[:50])
        big.set_stats(None)
        c2 = big.counters()
        n_mh50 = c2["insert_proposed"] + c2["remove_proposed"] - n_mh
        wk = kt.stats_from_tensor(wst)
        ab = {k: v.cpu().numpy() for k, v in big.accumulators().items()}
        docc_b = (ab["obs_sum"] / ab["sign_sum"][:, None])[:, 2 * spec.n_orb: 3 * spec.n_orb].mean(1)
        order_b = ab["order_sum"].sum(1) / ab["sign_sum"]
        n_call = nsteps_big_m if multi else nsteps_big
        thr[mode] = {"proposals_per_s": n_mh / (ms / 1000.0), "ms_per_step": ms / n_call, "call_steps": n_call,
                     "metropolis_steps_per_call_step": n_mh / (nbig * n_call),
                     "work_per_proposal": {"intervals": wk["intervals"] / n_mh50,
                                           "ops_applied": wk["ops_applied"] / n_mh50,
                                           "krylov_iters": wk["krylov_iters"] / n_mh50,
                                           "items_alive": wk["items_alive"] / n_mh50},
                     "trace_evaluations_per_proposal": c1["trace_evaluations"] / n_mh,
                     "acceptance": (c1["insert_accepted"] + c1["remove_accepted"]) / n_mh,
                     "eff": {"docc": 1.0 / (docc_b.var(ddof=1) * ms / 1000.0),
                             "order": 1.0 / (order_b.var(ddof=1) * ms / 1000.0)}}
        del big
    thr.update(chains=nbig, steps=nsteps_big, cache_ops=CACHE_OPS,
               start=(f"the {nw} thermalised configurations, each repeated {nbig // nw} times, then 2,000 "
                      f"multi-try delayed-acceptance call steps"),
               speedup_da_over_plain=thr["da"]["proposals_per_s"] / thr["plain"]["proposals_per_s"],
               speedup_cached_over_plain=thr["plain_cached"]["proposals_per_s"] / thr["plain"]["proposals_per_s"],
               speedup_da_cached_over_plain=thr["da_cached"]["proposals_per_s"] / thr["plain"]["proposals_per_s"],
               speedup_da_multi_over_plain=thr["da_multi"]["proposals_per_s"] / thr["plain"]["proposals_per_s"],
               speedup_da_multi_cached_over_plain=(thr["da_multi_cached"]["proposals_per_s"]
                                                  / thr["plain"]["proposals_per_s"]),
               speedup_at_equal_error_over_plain={m: {k: thr[m]["eff"][k] / thr["plain"]["eff"][k]
                                                         for k in ("docc", "order")}
                                                      for m in ("da", "da_multi", "plain_cached", "da_cached",
                                                                "da_multi_cached")})
    return {"workload": f"five_orbital_sweep_beta{beta:g}_1024_chains", "metric": "Metropolis proposals/s (all chains)",
            "sweep_definition": "one sweep = as many proposals per chain as the chain holds operators on average",
            "bath": "semicircular DOS, bandwidth 4, 2000 tau points", "thermalisation_steps": therm,
            "thermalisation": {"plain_steps": therm, "surrogate_training_steps": ncollect,
                               "da_multi_call_steps": THERM_DA_CALL_STEPS,
                               "metropolis_steps_per_chain": therm_mh / nw},
            "measure_every": meas, **out,
            "speedup_fp32_over_fp64": out["fp32"]["proposals_per_s"] / out["fp64"]["proposals_per_s"],
            "speedup_at_equal_error": speed,
            "speedup_at_equal_error_all_observables": {
                f"{a_}_over_{b_}": speedups(effs[a_], effs[b_])
                for a_, b_ in (("fp32", "fp64"), ("fp32_da", "fp64"), ("fp32_da", "fp32"), ("fp32_cached", "fp64"),
                               ("fp32_da_cached", "fp64"), ("fp32_cached", "fp32"), ("fp64_cached", "fp64"),
                               ("fp32_da_multi", "fp64"), ("fp32_da_multi", "fp32"), ("fp32_da_multi_cached", "fp64"),
                               ("fp32_da_multi_cached", "fp32_cached"))},
            "da_tries": DA_TRIES,
            "throughput_8192_chains": thr, "fp32_vs_fp64_same_uniforms": err32,
            "long_run_1024_chains": long_run,
            "cached_vs_uncached_identical_paths": cache_same, "cache_ops": CACHE_OPS,
            "surrogate": {"training_samples": n_train, "collect_s": t_collect, "train_s": t_train,
                          "epochs": len(hist), "loss_per_epoch": hist, "rms_residual_log_ratio": resid,
                          "target_std": spread, "network": "n_in-256-256-1 ReLU, BF16 tcgen05, FP32 accumulate"}}


def brief(x, digits: int = 6):
    """x with its floats rounded to `digits` significant digits."""
    if isinstance(x, float):
        return float(f"{x:.{digits}g}") if math.isfinite(x) else x
    if isinstance(x, dict):
        return {k: brief(v, digits) for k, v in x.items()}
    return [brief(v, digits) for v in x] if isinstance(x, list) else x


def brief_sweep(s):
    """The sweep's rates and speedups: sweep_bench's own dict is about 37,000 characters."""
    if s is None:
        return None

    def rates(d):
        return {m: {k: v[k] for k in ("proposals_per_s", "ms_per_step", "acceptance") if k in v}
                for m, v in d.items() if isinstance(v, dict) and "proposals_per_s" in v}

    out = {k: s[k] for k in ("workload", "metric", "measure_every", "speedup_fp32_over_fp64") if k in s}
    out.update(rates(s))
    out["speedup_at_equal_error_docc"] = {k: v["docc"] for k, v in s.get("speedup_at_equal_error", {}).items()}
    if "throughput_8192_chains" in s:
        out["throughput_8192_chains"] = {m: v["proposals_per_s"] for m, v in rates(s["throughput_8192_chains"]).items()}
    for b, v in s.get("other_betas", {}).items():
        out[b] = {m: r["proposals_per_s"] for m, r in rates(v).items()}
    return out


def printed_line(line):
    """The line printed: the contract's numbers in full, the others to six digits, the sweep as its rates. It
    stays below 8,192 characters, so that a reader of the last few kilobytes of the output gets it whole."""
    full = ("value", "ms_per_step", "e2e", "clocks")
    out = {k: v if k in full else brief(v) for k, v in line.items()}
    out["sweep"] = brief(brief_sweep(line.get("sweep")))
    return out


def main():
    global DA_TRIES
    a = args_()
    DA_TRIES = a.da_tries
    if a.impl == "reference":
        reference_arm(a)
        return
    import numpy as np
    import torch

    from paper_0908_0681_gb300 import engine, kt

    rank, local, world = dist_env()
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)

    def barrier():
        if world > 1:
            torch.distributed.barrier()

    n_rounds = min(N_ROUNDS, a.warmup + a.steps)
    w, seqs, moves = make_workload(rank, n_rounds, a.workload, a.trunc_eps)
    dseq = engine.DeviceSeqs.from_host(seqs, dev)
    dmoves = [engine.DeviceMoves.from_host(m, dev) for m in moves]
    m32 = engine.model_from_spec(w.model, precision=kt.KT_FP32_KRYLOV)
    m64 = engine.model_from_spec(w.model, precision=kt.KT_FP64)
    info = kt.kt_model_query(m32)
    ws = engine.workspace(m32, seqs.n, dev)
    stream = torch.cuda.current_stream()
    n = seqs.n
    out_s = torch.empty(n, dtype=torch.int8, device=dev)
    out_l = torch.empty(n, dtype=torch.float64, device=dev)
    out_st = torch.empty(n, dtype=torch.int32, device=dev)
    flush = torch.empty(64 * 1024 * 1024, dtype=torch.int32, device=dev)  # 256 MiB > 129 MB L2

    def current(model):
        s, l, st = engine.trace(model, dseq, ws=ws)
        return s, l

    # tiling: the autotuner times every compiled lane-group size on this batch
    tuned = {}
    for name, model in (("fp32", m32), ("fp64", m64)):
        tuned[name] = kt.kt_autotune(model, dseq.batch(), out_s, out_l, out_st, ws)
    cur32 = current(m32)
    cur64 = current(m64)
    torch.cuda.synchronize()

    def step(model, cur, r, stats=None):
        kt.kt_trace_ratio(model, dseq.batch(), cur[0], cur[1], dmoves[r % n_rounds].batch(), out_s, out_l, out_st,
                          stats, ws, stream)

    def timed_loop(model, cur, K, start_round):
        evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(K)]
        kt.kt_timing_begin(model, K)
        barrier()
        torch.cuda.synchronize()
        for k in range(K):
            flush.zero_()
            evs[k][0].record(stream)
            step(model, cur, start_round + k)
            evs[k][1].record(stream)
        torch.cuda.synchronize()
        barrier()
        stage_ms, nl = kt.kt_timing_end(model)
        ms = [e0.elapsed_time(e1) for e0, e1 in evs]
        return ms, stage_ms, nl

    # warm-up
    for k in range(a.warmup):
        step(m32, cur32, k)
        step(m64, cur64, k)
    torch.cuda.synchronize()

    sampler = ClockSampler(local)
    sampler.start()
    ms32, stage32, nl32 = timed_loop(m32, cur32, a.steps, a.warmup)
    clocks = sampler.stop()
    if st_bad := int((out_st != 0).sum().item()):
        vals, cnts = torch.unique(out_st, return_counts=True)
        hist = {kt.status_name(int(v)): int(c) for v, c in zip(vals.tolist(), cnts.tolist())}
        print(f"warning: {st_bad} walkers with non-OK status in the last step: {hist}", file=sys.stderr)

    K64 = a.fp64_steps if a.fp64_steps > 0 else min(a.steps, 100)
    ms64, stage64, _ = timed_loop(m64, cur64, K64, a.warmup)

    # the same with KT_FP32_TRIDIAG64, which changes Krylov propagations only
    m32t = engine.model_from_spec(w.model, precision=kt.KT_FP32_KRYLOV, flags=kt.KT_FP32_TRIDIAG64)
    tuned["fp32_tridiag64"] = kt.kt_autotune(m32t, dseq.batch(), out_s, out_l, out_st, ws)
    cur32t = current(m32t)
    for k in range(a.warmup):
        step(m32t, cur32t, k)
    Kt = min(a.steps, 100)
    ms32t, _, _ = timed_loop(m32t, cur32t, Kt, a.warmup)

    # Latency floor: the walkers with the longest edited sequences of the last timed round,
    # each evaluated alone (a batch of one: no other work on the GPU). The batch cannot finish
    # before its longest unit, so single_ms bounds items_ms from below.
    r_last = (a.warmup + a.steps - 1) % n_rounds
    lens = np.diff(seqs.offsets) + np.where(moves[r_last].kind == 0, 2, -2)
    longest = np.argsort(-lens, kind="stable")[:4]
    single = []
    for i in longest:
        s1 = engine.DeviceSeqs.from_host(seqs.subset([int(i)]), dev)
        m1 = engine.DeviceMoves.from_host(moves[r_last].subset([int(i)]), dev)
        c1 = (cur32[0][int(i):int(i) + 1].contiguous(), cur32[1][int(i):int(i) + 1].contiguous())
        o1 = (torch.empty(1, dtype=torch.int8, device=dev), torch.empty(1, dtype=torch.float64, device=dev),
              torch.empty(1, dtype=torch.int32, device=dev))
        w1 = engine.workspace(m32, 1, dev)
        ts = []
        for k in range(12):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            kt.kt_trace_ratio(m32, s1.batch(), c1[0], c1[1], m1.batch(), *o1, None, w1, stream)
            e1.record(stream)
            torch.cuda.synchronize()
            if k >= 2:
                ts.append(e0.elapsed_time(e1))
        single.append(float(np.median(ts)))
    latency_floor = {"longest_edited_lengths": [int(lens[i]) for i in longest], "single_walker_ms": single,
                     "items_ms_per_launch": stage32["items"] / max(nl32, 1),
                     "step_ms": sum(ms32) / a.steps,
                     "step_over_longest_single": (sum(ms32) / a.steps) / max(single)}

    # Ratios from cached partial states of the same fixed configurations (kt_ratio_cache):
    # the build stores every forward and backward state once (timed apart); each step
    # then propagates only the window that its update edits.
    cache = engine.RatioCache(m32, n, max_ops=CACHE_OPS)
    torch.cuda.synchronize()
    eb0, eb1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    eb0.record(stream)
    cache.build(dseq)
    eb1.record(stream)
    torch.cuda.synchronize()
    build_ms = eb0.elapsed_time(eb1)
    out_c = (torch.empty_like(out_s), torch.empty_like(out_l), torch.empty_like(out_st))
    for k in range(a.warmup):
        cache.ratio(dseq, cur32[0], cur32[1], dmoves[k % n_rounds], out=out_c)
    torch.cuda.synchronize()
    evc = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(a.steps)]
    barrier()
    torch.cuda.synchronize()
    for k in range(a.steps):
        flush.zero_()
        evc[k][0].record(stream)
        cache.ratio(dseq, cur32[0], cur32[1], dmoves[(a.warmup + k) % n_rounds], out=out_c)
        evc[k][1].record(stream)
    torch.cuda.synchronize()
    barrier()
    ms_c = [e0.elapsed_time(e1) for e0, e1 in evc]
    # agreement with the full evaluation on the last round
    step(m32, cur32, a.warmup + a.steps - 1)
    torch.cuda.synchronize()
    okc = (out_st == 0) & (out_c[2] == 0) & (out_s != 0)
    cached_ratio = {
        "value": n * a.steps / (sum(ms_c) / 1000.0), "unit": UNIT, "ms_per_step": sum(ms_c) / a.steps,
        "build_ms": build_ms, "cache_ops": CACHE_OPS,
        "speedup_over_full_evaluation": sum(ms32) / sum(ms_c),
        "signs_equal_to_full_evaluation": bool((out_s == out_c[0]).all().item()),
        "max_abs_log_diff_vs_full_evaluation": float((out_l - out_c[1]).abs()[okc].max().item()) if bool(okc.any()) else 0.0,
        "note": "same fixed configurations and rounds as the headline; the cache of those configurations is built once "
                "(build_ms, outside the timed steps, as the current traces are)"}
    del cache

    # algorithmic work of the timed FP32 steps (untimed stats pass over the same rounds)
    stats = engine.new_stats(dev)
    nonzero = torch.zeros((), dtype=torch.int64, device=dev)
    for k in range(a.steps):
        step(m32, cur32, a.warmup + k, stats)
        nonzero += (out_s != 0).sum()
    torch.cuda.synchronize()
    st = kt.stats_from_tensor(stats)
    nonzero_frac = float(nonzero.item()) / (n * a.steps)
    stats64 = engine.new_stats(dev)
    for k in range(K64):
        step(m64, cur64, a.warmup + k, stats64)
    torch.cuda.synchronize()
    st64 = kt.stats_from_tensor(stats64)

    # end to end through the C ABI from pinned host buffers
    host = {k: torch.from_numpy(np.ascontiguousarray(v)).pin_memory() for k, v in
            dict(off=seqs.offsets, tau=seqs.tau, fl=seqs.flavor, dg=seqs.dagger).items()}
    cs_h, cl_h = cur32[0].cpu().pin_memory(), cur32[1].cpu().pin_memory()
    mv_h = [{k: torch.from_numpy(np.ascontiguousarray(v)).pin_memory() for k, v in m.as_dict().items()}
            for m in moves]
    res_h = (torch.empty(n, dtype=torch.int8).pin_memory(), torch.empty(n, dtype=torch.float64).pin_memory(),
             torch.empty(n, dtype=torch.int32).pin_memory())
    d_cs, d_cl = torch.empty_like(cur32[0]), torch.empty_like(cur32[1])
    d_mv = engine.DeviceMoves.from_host(moves[0], dev)
    h2d = sum(t.numel() * t.element_size() for t in host.values()) + n * 9 + d_mv.nbytes()
    d2h = n * (1 + 8 + 4)
    K_e2e = min(a.steps, 200)
    barrier()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for k in range(K_e2e):
        r = (a.warmup + k) % n_rounds
        dseq.offsets.copy_(host["off"], non_blocking=True)
        dseq.tau.copy_(host["tau"], non_blocking=True)
        dseq.flavor.copy_(host["fl"], non_blocking=True)
        dseq.dagger.copy_(host["dg"], non_blocking=True)
        d_cs.copy_(cs_h, non_blocking=True)
        d_cl.copy_(cl_h, non_blocking=True)
        for name in ("kind", "flavor", "t_dag", "t_ann", "rem_idx"):
            getattr(d_mv, name).copy_(mv_h[r][name], non_blocking=True)
        kt.kt_trace_ratio(m32, dseq.batch(), d_cs, d_cl, d_mv.batch(), out_s, out_l, out_st, None, ws, stream)
        res_h[0].copy_(out_s, non_blocking=True)
        res_h[1].copy_(out_l, non_blocking=True)
        res_h[2].copy_(out_st, non_blocking=True)
        stream.synchronize()
    e1.record(stream)
    torch.cuda.synchronize()
    e2e_ms = e0.elapsed_time(e1) / K_e2e
    barrier()

    # aggregate over ranks: max time
    def reduce_max(vals):
        t = torch.tensor(vals, dtype=torch.float64, device=dev)
        torch.distributed.all_reduce(t, op=torch.distributed.ReduceOp.MAX)
        return t.tolist()

    value, (tot32, tot64, e2e_ms) = aggregate([sum(ms32), sum(ms64), e2e_ms], n, a.steps, world, reduce_max)
    value64 = world * n * K64 / (tot64 / 1000.0)
    value32t = n * Kt / (sum(ms32t) / 1000.0)
    tridiag = {"value": value32t, "unit": UNIT, "ms_per_step": sum(ms32t) / Kt, "steps": Kt,
               "speedup_over_fp64": value32t / value64, "flag": "KT_FP32_TRIDIAG64",
               "precision": "as the default: the flag changes Krylov propagations only, and this model's blocks "
                            "(at most 36 rows) are not propagated that way"}
    e2e_value = world * n / (e2e_ms / 1000.0)

    # roofline of the kernel of a ratio call (block eigenbasis)
    items_ms = stage32["items"] / max(nl32, 1)
    sha = source_sha()
    mhz = clocks.get("sm_max_mhz") or 2070.0
    peak32 = SM_COUNT_GB300 * FP32_LANES_PER_SM * 2 * mhz * 1e6 / 1e12
    peak64 = SM_COUNT_GB300 * FP64_FMA_PER_SM_CLK * 2 * mhz * 1e6 / 1e12
    f32_per_launch = st["intervals"] / a.steps * 2 * mean_block_square(w.model.n_orb)
    ach32 = f32_per_launch / (items_ms / 1000.0) / 1e12
    # The algorithmic work of the path is one dense block-to-block product per interval on the FP32
    # pipe; its serial per-walker dependency chain (not a pipe) is what bounds the kernel.
    roofline = {"bound": "alu", "achieved": ach32, "peak": peak32, "unit": "TFLOP/s", "frac": ach32 / peak32,
                "traffic": measured_traffic(sha), "kernel": "eig_kernel", "pipe": "fp32",
                "flops_per_launch": f32_per_launch,
                "flops_definition": ROOFLINE_DEFINITION,
                "items_ms_per_launch": items_ms,
                "stage_ms_per_step": {k: v / max(nl32, 1) for k, v in stage32.items()},
                "peak_source": "derived: 152 SMs x 128 FP32 lanes x 2 flops x max SM clock (sampled)",
                "frac_of_measured_fp32_peak": ach32 / MEASURED_FP32_TFLOPS,
                "measured_fp32_peak_tflops": MEASURED_FP32_TFLOPS,
                "fp64_peak_tflops": peak64,
                # the kernel is bound by its longest serial chain, not by a pipe: the step time
                # of its longest walker evaluated alone is the floor (bench key latency_floor)
                "latency_floor_ms": max(latency_floor["single_walker_ms"]),
                "frac_of_latency_floor": max(latency_floor["single_walker_ms"]) / (tot32 / a.steps)}

    sweep = sweep_bench(dev, a.sweep_steps, a.sweep_beta, seed=100 + rank) if a.sweep_steps > 0 else None
    if sweep is not None and rank == 0 and not a.no_other_betas:
        sweep["other_betas"] = {f"beta_{b:g}": sweep_beta_light(dev, b, a.sweep_other_steps, seed=300 + int(b))
                                for b in (10.0, 100.0)}
    seven = seven_bench(dev, min(a.steps, 40)) if (rank == 0 and a.workload == "five_orbital" and not a.no_seven) else None

    cpu = None
    if rank == 0 and world == 1 and not a.no_cpu_baseline:
        # GPU ratios of the first timed round, for the sampled error statement
        g = {}
        for name, model, cur in (("fp32", m32, cur32), ("fp32_tridiag64", m32t, cur32t), ("fp64", m64, cur64)):
            step(model, cur, a.warmup)
            torch.cuda.synchronize()
            g[name] = (out_s.cpu().numpy(), out_l.cpu().numpy(), cur[0].cpu().numpy(), cur[1].cpu().numpy())
        cpu = cpu_baseline(w, seqs, moves[a.warmup % n_rounds:] + moves[:a.warmup % n_rounds], g, a.cpu_seconds)
        if "fp32_tridiag64" in cpu.get("max_rel_err_vs_oracle", {}):
            tridiag["max_rel_err_vs_oracle"] = cpu["max_rel_err_vs_oracle"]["fp32_tridiag64"]

    if rank == 0:
        line = {
            "metric": METRIC if a.workload == "five_orbital" else METRIC_7, "value": value, "unit": UNIT, "n_gpus": world, "steps": a.steps, "warmup": a.warmup,
            "ms_per_step": tot32 / a.steps, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f32", "data": "synthetic",
            "config": {"workload": f"{a.workload}_{n}_walkers" + ("" if a.trunc_eps is None else f"_trunc{a.trunc_eps:g}"), "n_orb": w.model.n_orb, "U": w.model.U,
                       "J": w.model.J, "beta": w.model.beta,
                       "walkers_per_gpu": n, "mean_ops_per_walker": float(seqs.offsets[-1]) / n,
                       "krylov_tol": w.model.krylov_tol, "trunc_eps": w.model.trunc_eps, "precision": "fp32 pairs in the block eigenbasis (exact leading products, fp64 log-weights)",
                       "blocks": "(n_up, n_dn, singly-occupied mask)", "n_blocks": info["n_blocks"],
                       "d_max": info["d_max"], "n_kept": info["n_kept"], "group_lanes": tuned, "l2": "flushed (256 MiB write) before every timed step",
                       "parallelism": f"replicas x{world}"},
            "fp64_gpu": {"value": value64, "unit": UNIT, "ms_per_step": tot64 / K64, "steps": K64,
                         "stage_ms_per_step": {k: v / max(K64, 1) for k, v in stage64.items()},
                         "speedup_fp32_over_fp64": value / value64},
            "work": {"items_alive_per_step": st["items_alive"] / a.steps, "intervals_per_step": st["intervals"] / a.steps,
                     "mean_krylov_dim": st["krylov_iters"] / max(st["intervals"], 1), "p_max": st["p_max"],
                     "noconv": st["noconv"], "counted_by": "an untimed call with kt_stats (the Krylov route on the same inputs)",
                     "flops_per_step": f32_per_launch,
                     "nonzero_fraction": nonzero_frac,
                     "value_over_nonzero_proposals": value * nonzero_frac,
                     "p_hist_fp32": trim_hist(st["p_hist"]), "p_hist_fp64": trim_hist(st64["p_hist"]),
                     "mean_krylov_dim_fp64": st64["krylov_iters"] / max(st64["intervals"], 1)},
            "roofline": roofline,
            "fp32_tridiag64": tridiag,
            "seven_orbital": seven,
            "cached_ratio": cached_ratio,
            "latency_floor": latency_floor,
            "cpu_baseline": cpu,
            "e2e": {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h},
            "sweep": sweep,
            "clocks": clocks,
            # one kernel per ratio call (traces in the block eigenbasis)
            "gpu_launches": a.steps,
            "kernel_source_sha": sha,
        }
        if a.details:
            with open(a.details, "w") as f:
                json.dump(line, f)
        print(json.dumps(printed_line(line)), flush=True)
    if world > 1:
        torch.distributed.destroy_process_group()


if __name__ == "__main__":
    main()
