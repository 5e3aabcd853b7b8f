"""Benchmark: PSE Brownian samples per second on one GB300 (replicas on N GPUs).

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]

One step = one full PSE sample (cell list, neighbour list, device-side
Lanczos loop, k-space noise, inverse FFT, interpolation, combination) of the
headline workload: N = 1e6 random hard spheres (a = 1, RSA seed 1) at volume
fraction 0.1, tol 1e-3 -- the paper's Table 1 setting at N ~ 1e6 -- with the
splitting xi and FFT grid chosen before the timed region by pse_tune_xi (the
eq. xistar model calibrated at xi a = 0.5, then a timed scan of the grids
around it, each at the largest xi it admits).
L2 is flushed (a 256 MB write) before every timed step; each step is timed
with CUDA events on the launching stream.  Prints one JSON line.

The path has no data-parallel split: N > 1 GPUs run independent replicas
(their own seeds), value = all ranks' particle-samples / max rank time.
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "particle-samples/s at tol 1e-3 (N=1e6), learned+batched vs plain PSE"
UNIT = "particle-samples/s"
N_PART, PHI, XI, TOL, SEED_POS = 1_000_000, 0.1, 0.5, 1e-3, 1
# the splitting the timed scan picks for the headline workload on a GB300
# (grid 256^3, the largest xi that grid admits); the oracle arm, which has no
# GPU to run the scan, samples at it
XI_TUNED, M_TUNED = 0.5178442916, 256
CPU_SAMPLE_N = 100_000  # bounded CPU sample: same density and parameters, smaller box
REF_BUDGET_S = 150.0    # the oracle arm's warm-up + timed steps together
# wall time of one oracle sample per particle on the GPU machine's host (16 Arm
# cores): 6.5 s for N = 2.5e5
REF_S_PER_PARTICLE = 2.6e-5


def ref_sample_size(steps, warmup):
    """Particles per oracle-arm step: a function of the step count only."""
    n = int(REF_BUDGET_S / (max(steps + warmup, 1) * REF_S_PER_PARTICLE)) // 1000 * 1000
    return max(4000, min(CPU_SAMPLE_N, n))


def workload_config(plan=None, tuning=None, xi=XI_TUNED):
    cfg = {"workload": "random hard spheres, N=1e6, phi=0.1, a=1, tol=1e-3 (RSA seed 1), xi from the timed scan "
                       "started at xi*a=0.5, one PSE sample per step",
           "N": N_PART, "phi": PHI, "xi": xi, "tol": TOL, "precision": "fp32 grid/FFT/matvec, fp64 Lanczos scalars",
           "l2": "flushed (256 MB write) before every timed step"}
    if plan:
        cfg.update({"xi": plan["xi"], "L": round(plan["L"], 4), "M": plan["M"], "P": plan["P"],
                    "r_cut": round(plan["r_cut"], 4), "ncell": plan["ncell"]})
    if tuning:
        cfg["xi_tuning"] = {"xi_start": tuning["xi_start"], "xi_model": round(tuning["xi_model"], 4),
                            "xi_best": tuning["xi_best"], "M_best": tuning["M_best"],
                            "ms_start": round(tuning["ms_start"], 4), "ms_best": round(tuning["ms_best"], 4),
                            "grids_timed": tuning["n_grids"], "samples_timed": len(tuning["trials"])}
    return cfg


def replica_plan(xi, M, dev):
    """Every replica samples rank 0's splitting and grid (one broadcast)."""
    import torch
    import torch.distributed as dist
    t = torch.tensor([xi, float(M)], dtype=torch.float64, device=dev)
    dist.broadcast(t, 0)
    return float(t[0]), int(t[1])


def replica_time(total_ms, dev):
    """The slowest replica's timed region (max over ranks), in ms."""
    import torch
    import torch.distributed as dist
    t = torch.tensor([total_ms], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def replica_value(ws, n_part, steps, total_ms):
    """Whole-job particle-samples/s: every replica's samples over the slowest time."""
    return ws * n_part * steps / (total_ms / 1e3)


def replica_seed(rank):
    """Independent noise per replica."""
    return 1000 + rank


def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def clocks_start(rank=0, log_path=None):
    keep = rank == 0 and log_path  # one raw log, from rank 0, when asked for
    f = open(log_path if keep else os.devnull, "w")
    try:
        p = subprocess.Popen(["nvidia-smi", "--query-gpu=index,clocks.sm,clocks.max.sm,power.draw,"
                              "clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
                              "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
                              "clocks_event_reasons.sw_power_cap", "--format=csv,noheader,nounits", "-lms", "100"],
                             stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
    except OSError:
        p = None
    return p, f


def clocks_stop(p, f, device_index=0):
    if p is None:
        return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
    p.terminate()
    try:
        out, _ = p.communicate(timeout=5)
    except subprocess.TimeoutExpired:
        p.kill()
        out, _ = p.communicate()
    f.write(out)
    f.close()
    sm, smax, reasons = [], None, set()
    names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
    for line in out.strip().splitlines():
        cols = [c.strip() for c in line.split(",")]
        if len(cols) < 9 or cols[0] != str(device_index):
            continue
        try:
            sm.append(float(cols[1]))
            smax = float(cols[2])
        except ValueError:
            continue
        for n, v in zip(names, cols[5:9]):
            if v.lower().startswith("active"):
                reasons.add(n)
    return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": smax, "reasons": sorted(reasons),
            "samples": len(sm)}


# DRAM bytes (read + write) of one launch, from an ncu capture of the kernel
# at the workload (xi, M) recorded with it, valid only while the kernel's
# sources hash to the value recorded with it (profiles/ holds the summaries).
TRAFFIC = {
    "k_lz_matvec": (121_507_840 + 5_579_008, ("csrc/kernels_real.cu",),
                    "576669cd7df13d1201931b9a8718877e44acb9594b693f9939bca6acf4ff4efe", (0.5178442916, 256)),
    "k_interp4": (289_427_968 + 12_569_088, ("csrc/kernels_wave.cu",),
                  "0f86116b8713891908c3ea43879a6994b93437abe81f695edf53a8832dd6de20", (0.5178442916, 256)),
}


def captured_traffic(kernel, xi, M):
    import hashlib
    if kernel not in TRAFFIC:
        return None
    nbytes, files, digest, (xi_c, M_c) = TRAFFIC[kernel]
    if abs(xi - xi_c) > 1e-6 * xi_c or M != M_c:
        return None
    pkg = os.path.join(os.path.dirname(os.path.abspath(__file__)), "paper_1611_09322_gb300")
    h = hashlib.sha256()
    for f in files:
        with open(os.path.join(pkg, f), "rb") as fh:
            h.update(fh.read())
    return nbytes if h.hexdigest() == digest else None


def measured_peak():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return float(json.load(f)["hbm_gbs"]), "measured"
    except (OSError, KeyError, ValueError):
        return 6800.0, "fallback"


def _oracle_sample_times(n, xi, reps, seed0=0, keep=None):
    """Wall and CPU seconds of `reps` FP64 oracle PSE samples (real Lanczos
    part + gridded wave part) of an n-particle box at the headline's density
    and parameters; the configuration is generated outside the timing.  With
    a dict `keep`, the first sample, its configuration and seeds go there."""
    import resource
    import numpy as np
    from oracle import ewald, pse
    from paper_1611_09322_gb300 import workloads
    pos, L, _ = workloads.hard_spheres(n, PHI, SEED_POS)
    p = pos.astype(np.float64)
    walls, cpus, js = [], [], []
    for r in range(reps):
        r0 = resource.getrusage(resource.RUSAGE_SELF)
        t0 = time.perf_counter()
        plan = ewald.plan(L, 1.0, xi, TOL)
        ur, j, _ = pse.real_sample(p, plan, 7, seed0 + r)
        uw = pse.wave_sample_grid(p, plan, 7, seed0 + r)
        walls.append(time.perf_counter() - t0)
        r1 = resource.getrusage(resource.RUSAGE_SELF)
        cpus.append(r1.ru_utime - r0.ru_utime + r1.ru_stime - r0.ru_stime)
        js.append(j)
        if keep is not None and r == 0:
            keep.update(pos=pos, L=L, u=ur + uw, J=j, M=plan.M, seed=7, sample=seed0)
    return walls, cpus, js, plan.M


def _one_thread_env():
    env = dict(os.environ)
    for k in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS", "NUMEXPR_NUM_THREADS"):
        env[k] = "1"
    return env


def _quartiles(x):
    q = statistics.quantiles(x, n=4, method="inclusive") if len(x) > 1 else [x[0]] * 3
    return q[0], statistics.median(x), q[2]


def accuracy(first, xi):
    """Measured errors of the CUDA path, computed in the oracle leg: (1) the
    FP32 GPU sample of the first timed oracle sample's configuration, seeds
    and Lanczos count against that FP64 oracle sample, element by element;
    (2) what tol buys: the GPU sample (stop rule at tol) of N = 64 hard
    spheres at phi = 0.1 against the exact split sample -- M_r^{1/2} z1 by
    dense eigendecomposition of the all-image near-field mobility at the same
    r_cut, plus the wave part summed directly over modes with the same noise
    -- relative 2-norms (the wave part's error is the quadrature error of the
    paper's parameter rule, several times tol)."""
    import numpy as np
    import torch
    from oracle import ewald, pse
    from paper_1611_09322_gb300 import Sampler, workloads
    out = {}
    if first:
        s = Sampler(first["L"], 1.0, xi=xi, tol=TOL, grid_M=first["M"], fixed_iter=first["J"])
        u = s.sample(torch.from_numpy(first["pos"]).cuda(), first["seed"], first["sample"]).cpu().numpy()
        s.close()
        ref = first["u"]
        out["gpu_fp32_vs_fp64_oracle"] = {
            "N": int(first["pos"].shape[0]), "J": int(first["J"]), "M": int(first["M"]),
            "rel": float(np.linalg.norm(u - ref) / np.linalg.norm(ref)),
            "maxrel": float(np.abs(u - ref).max() / np.abs(ref).max())}
    N, phi, xi64, seed, sample = 64, 0.1, 0.5, 13579, 5
    pos, L, _ = workloads.hard_spheres(N, phi, 17)
    p64 = pos.astype(np.float64)
    plan = ewald.plan(L, 1.0, xi64, TOL)
    s = Sampler(L, 1.0, xi=xi64, tol=TOL)
    _, r, w = s.sample(torch.from_numpy(pos).cuda(), seed, sample, parts=True)
    J = s.stats()["lanczos_iters"]
    s.close()
    r, w = r.cpu().numpy().astype(np.float64), w.cpu().numpy().astype(np.float64)
    lam, Q = np.linalg.eigh(ewald.mobility_real_dense(p64, L, 1.0, xi64, plan.r_cut))
    z1 = pse.real_noise(N, seed, sample).ravel()
    ur = (Q @ (np.sqrt(np.maximum(lam, 0.0)) * (Q.T @ z1))).reshape(N, 3)
    uw = pse.wave_sample_direct(p64, plan, seed, sample)
    rel = lambda a, b: float(np.linalg.norm(a - b) / np.linalg.norm(b))  # noqa: E731
    out["method_vs_exact_split_sample"] = {"N": N, "phi": phi, "xi": xi64, "tol": TOL, "J": int(J),
                                            "rel": rel(r + w, ur + uw), "rel_real": rel(r, ur),
                                            "rel_wave": rel(w, uw)}
    return out


def cpu_baseline(xi=XI_TUNED, n=CPU_SAMPLE_N, reps=3, one_thread=True, with_accuracy=False):
    """The FP64 oracle as it stands, on a bounded sample of the headline
    workload: `reps` samples of an n-particle box at the same density, xi and
    tol (median and interquartile range of particle-samples/s), on the host's
    cores as the oracle uses them (`cores` = CPU time / wall time, the
    threads it actually kept busy), plus one sample in a subprocess limited
    to one thread."""
    first = {} if with_accuracy else None
    walls, cpus, js, M = _oracle_sample_times(n, xi, reps, keep=first)
    rates = [n / w for w in walls]
    q1, med, q3 = _quartiles(rates)
    busy = sum(cpus) / sum(walls)
    out = {"value": med, "unit": UNIT, "cores": max(1, round(busy)), "cpu_time_per_wall": round(busy, 2),
           "host_cores": os.cpu_count(), "cpu_model": _cpu_model(), "kind": "oracle",
           "iqr": [q1, q3], "samples": len(rates),
           "sample": f"{reps} FP64 oracle PSE samples of N={n} hard spheres at phi={PHI}, tol={TOL}, xi={xi:.4f} "
                     f"(M={M}, Lanczos j={js}); numpy/scipy; median {statistics.median(walls):.2f} s per sample"}
    if one_thread:
        code = ("import json,sys; sys.path.insert(0, %r); import bench; w, c, j, M = "
                "bench._oracle_sample_times(%d, %r, 1, 100); print(json.dumps([w[0], c[0]]))" % (ROOT, n, xi))
        try:
            p = subprocess.run([sys.executable, "-c", code], env=_one_thread_env(), capture_output=True, text=True,
                               timeout=600)
            w1, c1 = json.loads(p.stdout.strip().splitlines()[-1])
            out["one_thread"] = {"value": n / w1, "unit": UNIT, "wall_s": round(w1, 3),
                                 "cpu_time_per_wall": round(c1 / w1, 2)}
        except (subprocess.SubprocessError, ValueError, IndexError) as e:
            out["one_thread"] = {"unavailable": str(e)[:200]}
    if with_accuracy:
        # the oracle samples of this leg also measure the CUDA path's errors
        try:
            out["accuracy"] = accuracy(first, xi)
        except Exception as e:  # the throughput line stands without it
            out["accuracy"] = {"unavailable": str(e)[:200]}
    return out


def _cpu_model():
    try:
        with open("/proc/cpuinfo") as f:
            for line in f:
                k = line.split(":")[0].strip().lower()
                if k in ("model name", "cpu model", "processor name"):
                    return line.split(":", 1)[1].strip()
        out = subprocess.run(["lscpu"], capture_output=True, text=True).stdout
        for line in out.splitlines():
            if line.lower().startswith("model name"):
                return line.split(":", 1)[1].strip()
    except OSError:
        pass
    return "unknown"


def run_cpu_full(args):
    """The CPU protocol at the headline size: N = 1e6, `--steps` FP64 oracle
    samples (at least 3) on the host's cores as the oracle uses them, median
    and interquartile range, and one sample limited to one thread."""
    reps = max(3, min(args.steps, 10))
    line = cpu_baseline(XI_TUNED, n=N_PART, reps=reps, one_thread=True)
    line = {"impl": "oracle-cpu", "metric": METRIC,
            "config": dict(workload_config(), precision="fp64 throughout (the CPU oracle)"), **line}
    print(json.dumps(line), flush=True)
    return 0


def run_reference(args):
    ws, rank, _ = dist_env()
    if rank != 0:
        return 0
    import numpy as np
    from oracle import ewald, pse
    from paper_1611_09322_gb300 import workloads

    def setup(n):
        pos, L, _ = workloads.hard_spheres(n, PHI, SEED_POS)
        p = pos.astype(np.float64)
        plan = ewald.plan(L, 1.0, XI_TUNED, TOL)
        return p, plan, pse.RealOperator(p, plan)

    # each step is a bounded sample: the box (same density and parameters)
    # holds N_ref particles, fixed by the step count alone (no timing), so
    # that warm-up and timed steps take about REF_BUDGET_S together at the
    # oracle's measured cost of REF_S_PER_PARTICLE seconds per particle
    n_ref = ref_sample_size(args.steps, args.warmup)
    p, plan, op = setup(n_ref)

    def step(i):
        ur, j, _ = pse.real_sample(p, plan, 7, i, op=op)
        uw = pse.wave_sample_grid(p, plan, 7, i)
        return j

    import resource
    for i in range(args.warmup):
        step(i)
    r0 = resource.getrusage(resource.RUSAGE_SELF)
    t0 = time.perf_counter()
    for i in range(args.steps):
        step(1000 + i)
    dt = time.perf_counter() - t0
    r1 = resource.getrusage(resource.RUSAGE_SELF)
    busy = (r1.ru_utime - r0.ru_utime + r1.ru_stime - r0.ru_stime) / dt
    value = n_ref * args.steps / dt
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": dt / args.steps * 1e3,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": dict(workload_config(), precision="fp64 throughout (the CPU oracle)", M=plan.M),
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": max(1, round(busy)),
                             "cpu_time_per_wall": round(busy, 2), "host_cores": os.cpu_count(), "kind": "oracle",
                             "sample": f"each step: one FP64 oracle PSE sample of N={n_ref} at phi={PHI} "
                                       f"(same density, tol and xi={XI_TUNED:.4f} as the N=1e6 workload; N "
                                       f"fixed by --steps/--warmup for ~{REF_BUDGET_S:.0f} s over all steps; "
                                       f"neighbour pairs built once outside the timed steps)"},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


def timed_steps(run, steps, flush, stream):
    """Per-step CUDA-event times (ms) of `run(i)`, L2 flushed before each step."""
    import torch
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(steps)]
    for i in range(steps):
        flush.fill_(float(i))
        evs[i][0].record(stream)
        run(i)
        evs[i][1].record(stream)
    torch.cuda.synchronize()
    return [a.elapsed_time(b) for a, b in evs]


def matvec_bytes(N, n_pairs):
    """Algorithmic bytes of one near-field matvec (the minimum the method must
    move): positions 16N + input vector 12N + output 12N + the neighbour list
    4 bytes per directed pair."""
    return 16 * N + 12 * N + 12 * N + 4 * n_pairs


def kernel_roofline(stages, N, M, n_pairs, peak, interp_kernel="k_interp4"):
    """Per-kernel achieved GB/s (algorithmic bytes per launch / live per-launch
    time from pse_profile_stages) and its fraction of the measured peak."""
    interp_bytes = 16 * N + (16 if interp_kernel == "k_interp4" else 12) * M ** 3 + 16 * N
    per_kernel = {
        "matvec": ("k_lz_matvec", matvec_bytes(N, n_pairs)),
        "neighbours": ("k_nbr", 16 * N + 4 * n_pairs + 4 * N),
        "lanczos_update": ("k_lz_update", 80 * N),
        "interp": (interp_kernel, interp_bytes),
        "grid_copy": ("k_grid_aos", 28 * M ** 3),
        "wave_noise": ("k_wave_noise", 24 * M * M * (M // 2 + 1)),
    }
    if "fft" in stages and stages["fft"][0] == 0:  # the library's own transforms: noise + x and y (in place), then z to the node records
        half = 24 * M * M * ((M + 1) // 2)
        per_kernel["wave_noise"] = ("k_fft_x, k_fft_y", 3 * half // 2)
        per_kernel["grid_copy"] = ("k_fft_z_inv", half + 16 * M ** 3)
    out = {}
    for stage, (kname, nbytes) in per_kernel.items():
        ms, n = stages[stage]
        if n == 0 or ms <= 0:
            continue
        # (the search's launch of float64 decisions at r_cut, from 7e4 particles on, counts with it)
        per = ms if stage == "neighbours" else ms / n
        gbs = nbytes / (per / 1e3) / 1e9
        out[kname] = {"ms_per_launch": round(per, 5), "algorithmic_bytes": int(nbytes), "achieved_gbs": round(gbs, 1),
                      "frac": round(gbs / peak, 4)}
    return out


def variants_configs(dev, flush, stream, steps, peak):
    """The other workloads at full size: N = 1e6 hard spheres at phi = 0.3
    (tol 1e-3), N = 4e6 at phi = 0.3 (tol 1e-3 and 1e-5) and the 2.5e5 fractal gels (phi = 0.05, 0.1), each at the
    xi and grid of its own timed scan, plain vs learned preconditioner (network
    trained on the GPU at that xi and tol): throughput, Lanczos counts and the
    per-kernel roofline."""
    import torch
    from paper_1611_09322_gb300 import Sampler, precond_train, pse_tune_xi, workloads
    out = {}
    cases = [("hs_1e6_phi0.3", "hs", 1_000_000, 0.3, 5, 3.0, 1e-3)]  # the headline N at config 5's density
    cases += [("hs_4e6_phi0.3", "hs", 4_000_000, 0.3, 4, 3.0, tol) for tol in (1e-3, 1e-5)]
    cases += [(f"gel_2.5e5_phi{phi:g}", "gel", 250_000, phi, 3, 2.0, 1e-3) for phi in (0.05, 0.1)]
    cache = {}
    for name, kind, N, phi, seed, d_f, tol in cases:
        if (kind, N, phi) not in cache:
            cache.clear()
            cache[(kind, N, phi)] = workloads.make(kind, N, phi, seed)
        pos, L, _ = cache[(kind, N, phi)]
        d = torch.from_numpy(pos).to(dev)
        o = torch.empty_like(d)
        tun = pse_tune_xi(L, d, xi=XI, tol=tol, d_f=d_f, reps=3, autotune=1)
        xi, M = tun["xi_best"], tun["M_best"]
        theta, info = precond_train.train(xi=xi, tol=tol, steps=1500, lr=3e-3)
        for variant, th in (("plain", None), ("learned", theta)):
            s = Sampler(L, 1.0, xi=xi, tol=tol, grid_M=M)
            if th is not None:
                s.precond_set_weights(th)
            for i in range(2):
                s.sample(d, 1, i, out=o)
            per = timed_steps(lambda i: s.sample(d, 1, 500 + i, out=o), steps, flush, stream)
            st = s.stats()
            stages = s.profile_stages(d, 1, 9000, out=o)
            P = s.plan["P"]
            out[f"{name}_tol{tol:g}_{variant}"] = {
                "value": N * steps / (sum(per) / 1e3), "ms_per_step": sum(per) / steps, "unit": UNIT,
                "lanczos_iters": st["lanczos_iters"], "converged": st["converged"], "xi": round(xi, 5), "M": M,
                "P": P, "n_pairs": st["n_pairs"], "xi_start_ms": round(tun["ms_start"], 4),
                "kernels": kernel_roofline(stages, N, M, st["n_pairs"], peak,
                                           "k_interp4" if 3 <= P <= 10 else "k_interp")}
            s.close()
        del d, o
        torch.cuda.empty_cache()
    return out


def variants_full_lanczos(dev, flush, stream, steps, xi, M):
    """The paper's comparison method on the same GPU (Sec. IV, Fig. timing,
    Fig. RelLanc): Lanczos on the whole mobility, every iteration one M q
    product (spreading, FFT pair, interpolation, near-field matvec), against
    the PSE sample of the same configuration and parameters; N = 1e5 at
    xi a = 0.5 (planned grid) and the headline N = 1e6 at its tuned xi and
    grid.  The iteration count grows with N for the whole mobility, not for
    the real-space part (the paper's conditioning argument)."""
    import torch
    from paper_1611_09322_gb300 import Sampler, workloads
    out = {}
    for name, N, xi_n, M_n in (("full_lanczos_N1e5", 100_000, XI, 0), ("full_lanczos_N1e6", N_PART, xi, M)):
        pos, L, _ = workloads.hard_spheres(N, PHI, SEED_POS)
        d = torch.from_numpy(pos).to(dev)
        o = torch.empty_like(d)
        s = Sampler(L, 1.0, xi=xi_n, tol=TOL, grid_M=M_n)
        for i in range(2):
            s.sample_full_lanczos(d, 1, i, out=o)
        per = timed_steps(lambda i: s.sample_full_lanczos(d, 1, 800 + i, out=o), steps, flush, stream)
        st = s.stats()
        for i in range(3):
            s.sample(d, 1, i, out=o)
        per_pse = timed_steps(lambda i: s.sample(d, 1, 900 + i, out=o), max(steps, 10), flush, stream)
        j_pse = s.stats()["lanczos_iters"]
        ms, ms_pse = sum(per) / len(per), sum(per_pse) / len(per_pse)
        out[name] = {"value": N / (ms / 1e3), "ms_per_step": ms, "unit": UNIT, "lanczos_iters": st["lanczos_iters"],
                     "converged": st["converged"], "xi": s.plan["xi"], "M": s.plan["M"],
                     "pse_ms_per_step": ms_pse, "pse_lanczos_iters": j_pse, "pse_speedup": ms / ms_pse}
        s.close()
        del d, o
        torch.cuda.empty_cache()
    return out


def variants_poly(dev, flush, stream, steps):
    """Polydisperse suspension (Sec. V's size-dependent shape factor): N = 1e6
    random non-overlapping spheres of radii 1 and 0.5 (half each) at total
    volume fraction 0.1, xi a_max = 0.5, tol 1e-3, FFT size tuned; one
    spectrum and grid per species."""
    import numpy as np
    import torch
    from paper_1611_09322_gb300 import PolySampler, workloads
    pos, species, L, info = workloads.polydisperse(N_PART, PHI, SEED_POS, (1.0, 0.5))
    d = torch.from_numpy(pos).to(dev)
    sp = torch.from_numpy(species.astype(np.int32)).to(dev)
    o = torch.empty_like(d)
    s = PolySampler(L, (1.0, 0.5), xi=XI, tol=TOL, autotune=1)
    for i in range(3):
        s.sample(d, sp, 1, i, out=o)
    per = timed_steps(lambda i: s.sample(d, sp, 1, 700 + i, out=o), steps, flush, stream)
    st = s.stats()
    out = {"poly_bidisperse_N1e6": {"value": N_PART * steps / (sum(per) / 1e3), "ms_per_step": sum(per) / steps,
                                    "unit": UNIT, "lanczos_iters": st["lanczos_iters"], "converged": st["converged"],
                                    "n_pairs": st["n_pairs"], "xi": s.plan["xi"], "M": s.plan["M"], "L": L,
                                    "workload": "N=1e6 spheres of radii 1 and 0.5 (half each), phi=0.1, tol 1e-3"}}
    s.close()
    return out


def variants_learned_batched(dev, flush, stream, steps, xi, M):
    """The metric's comparison: learned preconditioner and batching vs plain."""
    import numpy as np
    import torch
    from paper_1611_09322_gb300 import BatchSampler, Sampler, precond_train, tune_batch_grid_step, workloads
    out = {}
    # the network is kept only if it cuts the held-out mean Lanczos count by
    # one iteration; otherwise the learned form falls back to P = I
    theta, info = precond_train.train_or_fallback(xi=xi, tol=TOL, steps=1500, lr=3e-3)
    theta_raw = info.pop("theta")
    out["learned_training"] = {k: v for k, v in info.items() if k != "loss_hist"}
    pos, L, _ = workloads.hard_spheres(N_PART, PHI, SEED_POS)
    d = torch.from_numpy(pos).to(dev)
    o = torch.empty_like(d)
    # list_free_N1e6: the plain sample with the list-free matvec (no
    # neighbour list; every product walks the 27 stencil cells)
    for name, th in (("plain_N1e6", None), ("learned_N1e6", theta), ("learned_no_fallback_N1e6", theta_raw),
                     ("list_free_N1e6", None)):
        s = Sampler(L, 1.0, xi=xi, tol=TOL, grid_M=M, matvec_shape=12 if name == "list_free_N1e6" else 0)
        if th is not None:
            s.precond_set_weights(th)
        for i in range(3):
            s.sample(d, 1, i, out=o)
        per = timed_steps(lambda i: s.sample(d, 1, 200 + i, out=o), steps, flush, stream)
        st = s.stats()
        out[name] = {"value": N_PART * steps / (sum(per) / 1e3), "ms_per_step": sum(per) / steps,
                     "lanczos_iters": st["lanczos_iters"], "converged": st["converged"],
                     "preconditioner": "none" if th is None and "learned" not in name else
                     ("network" if th is not None else "fallback P = I (no held-out iteration gain)")}
        s.close()
    # the forces path at the same workload: deterministic M F alone (the
    # paper's deterministic benchmark), one fused Euler-Maruyama displacement
    # dt M F + sqrt(2 dt) M^{1/2} z (kT = 1, dt = 1e-3), and the plain sample
    # with the wave noise drawn on the grid
    F = torch.randn(d.shape, device=dev, generator=torch.Generator(device=dev).manual_seed(3))
    s = Sampler(L, 1.0, xi=xi, tol=TOL, grid_M=M, autotune=2)
    runs = (("mobility_apply_N1e6", lambda i: s.sample_with_forces(d, F, 1, 400 + i, 1.0, 0.0, out=o)),
            ("euler_maruyama_N1e6", lambda i: s.sample_with_forces(d, F, 1, 500 + i, 1e-3, math.sqrt(2e-3), out=o)))
    for name, fn in runs:
        for i in range(3):
            fn(i)
        per = timed_steps(fn, steps, flush, stream)
        out[name] = {"value": N_PART * steps / (sum(per) / 1e3), "ms_per_step": sum(per) / steps}
    out["euler_maruyama_N1e6"]["lanczos_iters"] = s.stats()["lanczos_iters"]
    # a whole Brownian dynamics step: neighbour list, overlap repulsion
    # (k_rep = 100), the fused displacement and the position update, in place
    x = d.clone()
    bd = lambda i: s.bd_step(x, 1, 700 + i, 1e-3, 1.0, 100.0)  # noqa: E731
    for i in range(3):
        bd(i)
    per = timed_steps(bd, steps, flush, stream)
    out["bd_step_N1e6"] = {"value": N_PART * steps / (sum(per) / 1e3), "ms_per_step": sum(per) / steps,
                           "lanczos_iters": s.stats()["lanczos_iters"]}
    s.close()
    s = Sampler(L, 1.0, xi=xi, tol=TOL, grid_M=M, wave_noise=1)
    for i in range(3):
        s.sample(d, 1, i, out=o)
    per = timed_steps(lambda i: s.sample(d, 1, 600 + i, out=o), steps, flush, stream)
    out["grid_noise_sample_N1e6"] = {"value": N_PART * steps / (sum(per) / 1e3), "ms_per_step": sum(per) / steps,
                                     "lanczos_iters": s.stats()["lanczos_iters"]}
    s.close()
    spec = workloads.batch_spec()
    pos_list, Ls = [], []
    for sp in spec:
        p, Lk, _ = workloads.make(sp["kind"], sp["N"], sp["phi"], sp["seed"])
        pos_list.append(p)
        Ls.append(Lk)
    offsets = np.cumsum([0] + [p.shape[0] for p in pos_list])
    pa = torch.from_numpy(np.concatenate(pos_list)).to(dev)
    po = torch.empty_like(pa)
    # the systems' grids: their planned size classes or one or two classes
    # finer (each then at the largest xi its grid admits), by a timed choice
    # before the timed region, like the xi scan of the single system
    gtune = tune_batch_grid_step(Ls, pa, offsets, xi=XI, tol=TOL, autotune=9)
    for name, th in (("batched_64sys_plain", None), ("batched_64sys_learned", theta)):
        b = BatchSampler(Ls, 1.0, params=gtune["params"])
        if th is not None:
            for k in range(len(spec)):
                b.set_precond(k, th)
        for i in range(3):
            b.sample(pa, offsets, 1, i, out=po)
        per = timed_steps(lambda i: b.sample(pa, offsets, 1, 300 + i, out=po), steps, flush, stream)
        its = [b.stats(k)["lanczos_iters"] for k in range(len(spec))]
        out[name] = {"value": int(offsets[-1]) * steps / (sum(per) / 1e3), "ms_per_step": sum(per) / steps,
                     "n_systems": len(spec), "n_particles": int(offsets[-1]), "lanczos_iters_mean": float(np.mean(its)),
                     "grid_step": gtune["step"], "grid_step_ms": {str(k): round(v, 4) for k, v in gtune["ms"].items()},
                     "preconditioner": "none" if th is None and name.endswith("plain") else
                     ("network" if th is not None else "fallback P = I (no held-out iteration gain)")}
        grids = [b.plan(k)["M"] for k in range(len(spec))]
        xis = [b.plan(k)["xi"] for k in range(len(spec))]
        b.close()
    # the same 64 systems without batching: one lone sampler per system (its
    # own xi, grid and CUDA graph, the settings the batch gave it), sampled
    # one after another on one stream, timed with the same protocol
    lone = [Sampler(Lk, 1.0, xi=xis[k], tol=TOL, grid_M=grids[k], system=k) for k, Lk in enumerate(Ls)]
    views = [pa[offsets[k]:offsets[k + 1]] for k in range(len(spec))]
    outs = [po[offsets[k]:offsets[k + 1]] for k in range(len(spec))]

    def lone_step(i):
        for k, sk in enumerate(lone):
            sk.sample(views[k], 1, 300 + i, out=outs[k])
    for i in range(3):
        lone_step(i)
    per = timed_steps(lone_step, steps, flush, stream)
    its = [sk.stats()["lanczos_iters"] for sk in lone]
    out["batched_64sys_lone"] = {"value": int(offsets[-1]) * steps / (sum(per) / 1e3), "ms_per_step": sum(per) / steps,
                                 "n_systems": len(spec), "n_particles": int(offsets[-1]),
                                 "lanczos_iters_mean": float(np.mean(its)),
                                 "what": "the 64 systems through 64 lone samplers (one CUDA graph each, same xi and "
                                         "grid as in the batch), one after another on one stream"}
    for sk in lone:
        sk.close()
    out["workload_batched"] = ("64 periodic systems, N log-uniform in [1e3, 5e4], phi uniform in [0.05, 0.4], "
                               "half fractal gels (phi <= 0.2), each with its own box, FFT grid (the planned grid "
                               "raised to a size class, then 0-2 classes finer by one timed choice for the batch) "
                               "and xi (the largest its grid admits, from xi a = 0.5), tol 1e-3; one CUDA graph "
                               "launch per step")
    out["variants_xi"] = {"xi": xi, "M": M, "note": "the N=1e6 variants run at the headline's tuned xi and grid"}
    return out


def run_only(args):
    """One secondary workload alone (for profiling its kernels): the
    deterministic product M F at N = 1e6 ("forces") or the 64-system batch
    ("batch"); --no-graph launches the same kernels without a CUDA graph so
    that a profiler sees every kernel.  Prints one JSON line."""
    import numpy as np
    import torch
    from paper_1611_09322_gb300 import BatchSampler, Sampler, tune_batch_grid_step, workloads
    dev = torch.device("cuda", 0)
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
    stream = torch.cuda.current_stream()
    graph = not args.no_graph
    if args.only == "forces":
        pos, L, _ = workloads.hard_spheres(N_PART, PHI, SEED_POS)
        d = torch.from_numpy(pos).to(dev)
        F = torch.randn(d.shape, device=dev, generator=torch.Generator(device=dev).manual_seed(3))
        o = torch.empty_like(d)
        s = Sampler(L, 1.0, xi=XI, tol=TOL, use_graph=graph, spread_tile=4)
        for i in range(args.warmup):
            s.mobility_apply(d, F, out=o)
        per = timed_steps(lambda i: s.mobility_apply(d, F, out=o), args.steps, flush, stream)
        n, variant = N_PART, "deterministic M F, N=1e6 hard spheres, phi=0.1, tiles of 4^3 cells"
        s.close()
    else:
        spec = workloads.batch_spec()
        pos_list, Ls = [], []
        for sp in spec:
            p, Lk, _ = workloads.make(sp["kind"], sp["N"], sp["phi"], sp["seed"])
            pos_list.append(p)
            Ls.append(Lk)
        offsets = np.cumsum([0] + [p.shape[0] for p in pos_list])
        pa = torch.from_numpy(np.concatenate(pos_list)).to(dev)
        po = torch.empty_like(pa)
        gtune = tune_batch_grid_step(Ls, pa, offsets, xi=XI, tol=TOL, autotune=9)
        b = BatchSampler(Ls, 1.0, params=[dict(pk, use_graph=graph) for pk in gtune["params"]])
        for i in range(args.warmup):
            b.sample(pa, offsets, 1, i, out=po)
        per = timed_steps(lambda i: b.sample(pa, offsets, 1, 100 + i, out=po), args.steps, flush, stream)
        n = int(offsets[-1])
        variant = (f"64-system batch (N log-uniform in [1e3, 5e4], phi in [0.05, 0.4], half gels), grids "
                   f"{gtune['step']} size classes finer than planned (timed choice)")
        b.close()
    print(json.dumps({"only": args.only, "variant": variant, "graph": graph, "steps": args.steps,
                      "ms_per_step": sum(per) / args.steps, "value": n * args.steps / (sum(per) / 1e3),
                      "unit": UNIT}), flush=True)
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="native", choices=["native", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--cpu-full", action="store_true",
                    help="only the CPU protocol at N = 1e6: the FP64 oracle, max(3, min(--steps, 10)) samples, "
                         "median and IQR, and one sample on one thread")
    ap.add_argument("--no-variants", action="store_true")
    ap.add_argument("--only", choices=["forces", "batch"], default=None,
                    help="run one secondary workload alone (profiling aid)")
    ap.add_argument("--no-graph", action="store_true", help="with --only: launch without CUDA graphs")
    ap.add_argument("--xi", type=float, default=None,
                    help="skip the xi scan and sample at this xi (with --grid; a profiling aid)")
    ap.add_argument("--grid", type=int, default=0, help="with --xi: the FFT grid per side")
    ap.add_argument("--clock-log", default=None,
                    help="also write the raw nvidia-smi samples of the timed region to this file")
    ap.add_argument("--interp-form", type=int, default=0, choices=[0, 1],
                    help="interpolation form of the headline sampler (1: planar grids; a profiling aid)")
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    if args.impl == "reference":
        return run_reference(args)
    if args.cpu_full:
        return run_cpu_full(args)
    if args.only:
        return run_only(args)

    import torch
    import torch.distributed as dist
    from paper_1611_09322_gb300 import Sampler, pse_tune_xi, workloads

    ws, rank, local = dist_env()
    if ws > 1:
        torch.cuda.set_device(local)
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    dev = torch.device("cuda", local if ws > 1 else 0)
    torch.cuda.set_device(dev)

    pos, L, _ = workloads.hard_spheres(N_PART, PHI, SEED_POS)
    d_pos = torch.from_numpy(pos).to(dev)
    # the splitting and grid: the timed scan around the model's xi* (untimed
    # setup, like the cuFFT plans); replicas take rank 0's choice
    if args.xi is not None:
        tuning = None
        xi, M_grid = args.xi, args.grid
    else:
        tuning = pse_tune_xi(L, d_pos, xi=XI, tol=TOL, reps=10, autotune=1)
        xi, M_grid = tuning["xi_best"], tuning["M_best"]
    if ws > 1:
        xi, M_grid = replica_plan(xi, M_grid, dev)
    s = Sampler(L, 1.0, xi=xi, tol=TOL, grid_M=M_grid, interp_form=args.interp_form)
    out = torch.empty_like(d_pos)
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
    stream = torch.cuda.current_stream()
    seed = replica_seed(rank)

    clk, clkf = clocks_start(rank, args.clock_log)
    for i in range(args.warmup):
        s.sample(d_pos, seed, i, out=out)
    torch.cuda.synchronize()
    if ws > 1:
        dist.barrier()
    torch.cuda.synchronize()
    per = timed_steps(lambda i: s.sample(d_pos, seed, 100 + i, out=out), args.steps, flush, stream)
    if ws > 1:
        dist.barrier()
    clocks = clocks_stop(clk, clkf, dev.index)
    total_ms = sum(per)
    st = s.stats()
    J = st["lanczos_iters"]
    if ws > 1:
        total_ms = replica_time(total_ms, dev)
    value = replica_value(ws, N_PART, args.steps, total_ms)

    # live per-stage timing (CUDA events on the launching stream) for the roofline
    stages = None
    for i in range(3):
        stages = s.profile_stages(d_pos, seed, 10_000 + i, out=out)
    n_pairs = s.stats()["n_pairs"]
    plan = s.plan
    M = plan["M"]
    dom = max(stages, key=lambda k: stages[k][0])
    # algorithmic bytes per launch: matvec_bytes (positions, input, output,
    # 4 B of list per pair); the grid copy reads the three planar grids and
    # writes the 16-byte node records; interpolation reads positions and the
    # node records once, writes u_w; the FFT stage, where there is one, is cuFFT's.
    bytes_mv = matvec_bytes(N_PART, n_pairs)
    bytes_in = 16 * N_PART + 16 * M ** 3 + 16 * N_PART
    bytes_cp = 12 * M ** 3 + 16 * M ** 3
    kernel_bytes = {"matvec": ("k_lz_matvec", bytes_mv), "interp": ("k_interp4", bytes_in),
                    "grid_copy": ("k_grid_aos", bytes_cp)}
    if stages["fft"][0] == 0:  # the library's own transforms: their z pass writes the node records
        kernel_bytes["grid_copy"] = ("k_fft_z_inv", 24 * M * M * ((M + 1) // 2) + 16 * M ** 3)
    key = max(kernel_bytes, key=lambda k: stages[k][0])
    kname, kb = kernel_bytes[key]
    kms = stages[key][0] / max(stages[key][1], 1)
    peak, peak_kind = measured_peak()
    achieved = kb / (kms / 1e3) / 1e9
    roofline = {"bound": "hbm", "kernel": kname, "achieved": round(achieved, 1), "peak": peak, "unit": "GB/s",
                "frac": round(achieved / peak, 4), "traffic": captured_traffic(kname, plan["xi"], M), "peak_kind": f"{peak_kind} hbm_gbs (copy), burst",
                "algorithmic_bytes_per_launch": kb, "ms_per_launch": round(kms, 5), "dominant_stage": dom,
                "kernels": kernel_roofline(stages, N_PART, M, n_pairs, peak),
                "stages_ms": {k: round(v[0], 4) for k, v in stages.items()},
                "stages_launches": {k: v[1] for k, v in stages.items()}}

    # end to end through the C ABI with host buffers (pinned), copies inside
    # the timed region: every step copies its positions in and its result
    # out (pse_sample_host_async: the copies of one step overlap the
    # sampling of its neighbours), all results on the host at the end
    hp = torch.from_numpy(pos).pin_memory()
    ho = [torch.empty_like(hp).pin_memory() for _ in range(2)]
    for i in range(2):
        s.sample_host_async_ptr(N_PART, hp.data_ptr(), ho[i % 2].data_ptr(), seed, 50_000 + i)
    s.host_sync()
    K2 = max(3, min(args.steps, 50))
    t0 = time.perf_counter()
    for i in range(K2):
        s.sample_host_async_ptr(N_PART, hp.data_ptr(), ho[i % 2].data_ptr(), seed, 60_000 + i)
    s.host_sync()
    e2e_s = (time.perf_counter() - t0) / K2
    e2e = {"value": ws * N_PART / e2e_s, "unit": UNIT, "h2d_bytes_per_step": 12 * N_PART,
           "d2h_bytes_per_step": 12 * N_PART}
    s.close()

    if rank == 0:
        line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps,
                "warmup": args.warmup, "ms_per_step": total_ms / args.steps,
                "ms_per_step_median": statistics.median(per),
                "ms_per_step_iqr": [round(q, 5) for q in _quartiles(per)[0::2]],
                "higher_is_better": True, "scaling": "weak",
                "vs_baseline": None, "dtype": "f32", "data": "synthetic",
                "config": workload_config(plan, tuning), "lanczos_iters": J, "n_pairs": n_pairs,
                "variant": "plain PSE, one system, one CUDA graph per sample",
                "roofline": roofline, "e2e": e2e, "clocks": clocks,
                "gpu_launches": sum(n for _, n in stages.values()) * args.steps,
                "parallelism": "replicas" if ws > 1 else "single GPU"}
        if not args.no_variants and ws == 1:
            line["variants"] = variants_learned_batched(dev, flush, stream, max(20, args.steps // 4), xi, M_grid)
            # the metric's comparison at the top level: learned (with its
            # fallback) and batched against plain, and the batch against the
            # same systems sampled one by one
            for k in ("learned_N1e6", "batched_64sys_plain", "batched_64sys_learned", "batched_64sys_lone"):
                line[k] = line["variants"][k]
            line["variants"].update(variants_full_lanczos(dev, flush, stream, 5, xi, M_grid))
            line["variants"].update(variants_poly(dev, flush, stream, max(20, args.steps // 4)))
            line["variants"].update(variants_configs(dev, flush, stream, 10, peak))
        if not args.no_cpu_baseline and ws == 1:
            line["cpu_baseline"] = cpu_baseline(xi, with_accuracy=True)
            line["accuracy"] = line["cpu_baseline"].pop("accuracy")
        print(json.dumps(line), flush=True)
    if ws > 1:
        dist.destroy_process_group()
    return 0


if __name__ == "__main__":
    sys.exit(main())
