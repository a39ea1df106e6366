"""Benchmark: band-k H|psi> applications per second of the batched mixed-precision Davidson
solve, converged to 1e-8 Ry, on one GB300 (or N replicas), against the per-k FP64 form.

Workload (one step): the lowest 20 eigenpairs of H(k) for all 512 k-points of the 1-atom fcc
cell (a = 7.5 bohr, ecutwfc = 45 Ry, npw 528-548, FFT 24^3, 9 projectors, 8x8x8 MP grid) by
one pwk_davidson_batched call in the mixed mode (FP32 H applications, FP64 refinement and
FP64 reduced eigensolves inside the call), from the generator's random orthonormal trial
vectors, to |d eps| < 1e-10 Ry and ||H psi - eps psi|| < 1e-5 (eigenvalues checked against the
oracle's dense eigensolver to 1e-8 Ry).  value = the band-k H applications the solve performs
(FP32 and FP64 together) / its device time.  Inputs are resident in HBM; the L2 is flushed (a
512 MiB write) before every timed step.

Also reported: the same solve with every H application in FP64 (batched), the per-k FP64 form
(one plan and one call per k-point, on a sample of k-points, extrapolated), where the solve
spends its device time (H applications, reduced eigensolves, the rest), the end-to-end rate
through the C ABI with the trial vectors and results in host memory, the raw H|psi> kernel
rates and rooflines, the DFPT Sternheimer solve and induced density, the other cells, the
serving loop and the CPU oracle baseline.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference] [--quick]
  python bench.py --case hpsi|davidson|sternheimer --cfg C [--nk NK] [--precision P] [--reps R]

--case runs one operation of the library on one synthetic cell (the command the profiles
under profiles/ were captured with) and prints the CUDA-event time of each repetition; the
repetitions sit in an NVTX range "case", plan creation outside it.
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
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "band-k H|psi> applies/s, batched mixed-prec vs per-k FP64 at 1e-8 Ry; p99 latency"
UNIT = "band-k applies/s"
CFG = 2
WORKLOAD = ("batched Davidson to 1e-8 Ry (mixed FP32/FP64): fcc 1 atom a=7.5 ecut=45Ry FFT 24^3, "
            "512 k (8x8x8 MP), 20 bands, 9 projectors")
ETH, RES_TOL, MAX_ITER = 1e-10, 1e-5, 300     # Davidson stopping (|d eps| Ry, residual norm)
EIG_TOL = 1e-8                                  # Ry: the accuracy the metric is quoted at
FLUSH_BYTES = 512 * 1024 * 1024


def measured_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    d = {}
    if os.path.exists(path):
        with open(path) as f:
            d = json.load(f)
    return {"hbm_gbs": d.get("hbm_gbs", 6800.0),
            "hbm_source": "measured (MEASURED_PEAKS.json)" if "hbm_gbs" in d else "fallback",
            "sm_max_mhz": d.get("sm_max_mhz", 2070.0)}


def src_digest(*names) -> str:
    """Short digest of kernel sources: a DRAM traffic figure copied from an ncu capture is
    reported only while the sources it was captured at are unchanged."""
    h = hashlib.sha256()
    for n in names:
        with open(os.path.join(ROOT, "paper_2412_01695_gb300", "csrc", n), "rb") as f:
            h.update(f.read())
    return h.hexdigest()[:12]


# projector paths (pwk_plan_projector_choice)
PATH_NAMES = {1: "separate tensor-core kernels", 2: "separate CUDA-core kernels", 3: "fused in the local kernel"}

# dram__bytes_read.sum + dram__bytes_write.sum of one launch of a kernel, from ncu captures
# summarised under profiles/, with the digest of the sources they were captured at.
# rr_kernel: a full-batch launch of the 64-k solve (10.61 MB) scaled by k-points to the
# 512-k batch of the headline step.
# The H|psi> kernels of the 512-k cell in FP32: mean of three launches.
TRAFFIC = {
    "rr_kernel": {"bytes": 8 * (10562816 + 44288), "profile": "profiles/rr_kernel_davidson_fcc64k_20b.md",
                  "sources": ["rr.cu", "solvers.h"], "digest": "561669374c49"},
    "fused_window_kernel<float,float,24,6>": {
        "bytes": 48409941 + 4088405, "profile": "profiles/hpsi_step_kernels_fcc512k_20b_fp32.md",
        "sources": ["fused_window.cuh", "fft_line.cuh", "hpsi_f32.cu"], "digest": "dbb74c7b7ac9"},
    "nl_project_kernel<float,float,9>": {
        "bytes": 65060011 + 12288, "profile": "profiles/hpsi_step_kernels_fcc512k_20b_fp32.md",
        "sources": ["nonlocal.cu"], "digest": "67c9475f7eb9"},
    "nl_addback_kernel<float,float,9>": {
        "bytes": 66527147 + 159061, "profile": "profiles/hpsi_step_kernels_fcc512k_20b_fp32.md",
        "sources": ["nonlocal.cu"], "digest": "67c9475f7eb9"},
    "fused_window_kernel_nl<float,float,24,6>": {
        "bytes": 68629077 + 11927797, "profile": "profiles/fused_window_kernel_nl_hpsi_fcc512k_20b_fp32.md",
        "sources": ["fused_window.cuh", "fft_line.cuh", "nl_fused.cuh", "hpsi_f32_nl.cu"],
        "digest": "bdf361b8ae02"},
}


def traffic_for(kernel: str):
    t = TRAFFIC.get(kernel)
    if t is None or src_digest(*t["sources"]) != t["digest"]:
        return None, None
    return t["bytes"], t["profile"]


# --------------------------------------------------------------------------- clocks
class ClockSampler:
    """nvidia-smi sampling of SM clock and throttle reasons during a timed region."""
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except (OSError, FileNotFoundError):
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.thread.join(timeout=2)
        sm, smax, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax = float(parts[2])
            except ValueError:
                continue
            for n, v in zip(names, parts[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(n)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": smax,
                "reasons": sorted(reasons), "samples": len(sm)}


# --------------------------------------------------------------------------- work counts
def hit_planes(prob):
    """Per k-point: the z-sticks (distinct (m1, m2)) and the m1 planes its sphere hits."""
    ns, npl = [], []
    for ik in range(prob.nk):
        m = prob.miller[ik, :prob.npw[ik]]
        ns.append(len(set(map(tuple, m[:, :2].tolist()))))
        npl.append(len(np.unique(m[:, 0])))
    return np.array(ns, float), np.array(npl, float)


def local_flops_per_band(prob) -> float:
    """The local term of one H application (the algorithmic count of the pruned transform pair,
    5 n log2 n per 1D transform: z on the k-point's sticks, y on its hit m1 planes, x on every
    line, inverse and forward), 2 N_r for V(r) u(r) and 2 npw for the kinetic term, averaged
    over the k-points."""
    N = prob.N
    f1 = 5.0 * N * math.log2(N)
    ns, npl = hit_planes(prob)
    fft = f1 * 2.0 * (ns + npl * N + N * N)
    return float(np.mean(fft + 2.0 * N ** 3 + 2.0 * prob.npw))


def nonlocal_flops_per_band(prob) -> float:
    """Projection and add-back (Eqs. lambdah, finalnl): 8 flops per complex multiply-add, two
    contractions of nkb x npw."""
    return 16.0 * prob.nkb * float(np.mean(prob.npw))


def algorithmic_bytes_per_band(prob, elem_bytes: int) -> float:
    """read psi + write H psi + (beta + |k+G|^2 + index per k) / nb; V stays in L2."""
    npw = float(np.mean(prob.npw))
    per_k = prob.nkb * prob.npw_max * elem_bytes + prob.npw_max * (8 + 4)
    return 2.0 * npw * elem_bytes + per_k / prob.nb


# --------------------------------------------------------------------------- timing helpers
class Timer:
    def __init__(self, torch, dev, stream):
        self.torch, self.stream = torch, stream
        self.flush = torch.empty(FLUSH_BYTES // 4, dtype=torch.float32, device=dev)

    def run(self, fn, steps, warmup, prep=None, flush=True):
        """CUDA-event time of each of `steps` calls of fn after `warmup` untimed ones; prep()
        (untimed) and an L2 flush before every call.  self.launches: the library's kernel
        launches inside the timed calls (pwk_launch_count before and after each)."""
        from paper_2412_01695_gb300 import pwk
        torch = self.torch
        for _ in range(warmup):
            if prep:
                prep()
            fn()
        torch.cuda.synchronize()
        out = []
        self.launches = 0
        for _ in range(steps):
            if prep:
                prep()
            if flush:
                self.flush.fill_(1.0)
            a = torch.cuda.Event(enable_timing=True)
            b = torch.cuda.Event(enable_timing=True)
            c0 = pwk.launch_count()
            a.record(self.stream)
            r = fn()
            b.record(self.stream)
            self.launches += pwk.launch_count() - c0
            torch.cuda.synchronize()
            out.append((a.elapsed_time(b) / 1e3, r))
        return out


def fma_peaks(torch, dev, stream):
    """Measured FP32 / FP64 CUDA-core FMA throughput (pwk_measure_fma_peak), with the clocks
    seen during the measurement."""
    from paper_2412_01695_gb300 import pwk
    clk = ClockSampler(dev.index or 0)
    clk.start()
    f32, sms = pwk.measure_fma_peak(pwk.PWK_FP32, stream)
    f64, _ = pwk.measure_fma_peak(pwk.PWK_FP64, stream)
    c = clk.stop()
    return {"fp32_tflops": f32 / 1e12, "fp64_tflops": f64 / 1e12, "sm_count": sms,
            "source": "pwk_measure_fma_peak (independent FMA chains on every SM, best of 3, CUDA events)",
            "sm_mhz_during": c.get("sm_mhz")}


# --------------------------------------------------------------------------- the headline
def davidson_runner(torch, pwk, plan, prob, dev, mode, stream):
    psi0 = torch.from_numpy(prob.psi).to(dev)
    psi = torch.empty_like(psi0)
    eig = torch.zeros((prob.nk, prob.nb), dtype=torch.float64, device=dev)

    def prep():
        psi.copy_(psi0)

    def solve():
        rc, iters, notc, napply = pwk.davidson_batched(plan, mode, psi, eig, prob.nb, ETH, RES_TOL,
                                                       MAX_ITER, 0, stream)
        return {"rc": int(rc), "iters_max": int(iters.max()), "iters_p50": float(np.median(iters)),
                "applies_fp64": int(napply[0]), "applies_fp32": int(napply[1]),
                "stats": plan.solver_stats()}
    return prep, solve, psi, eig


def per_k_fp64(torch, pwk, synth, prob, dev, stream, nks):
    """The per-k FP64 form: one plan and one FP64 Davidson call per k-point (the same trial
    vectors), on a seeded sample of k-points; plan creation is outside the time."""
    ks = synth.sample_k(prob.nk, nks, seed=21)
    t_tot, applies = 0.0, 0
    for ik in ks:
        sub = synth.make_config(CFG, k_subset=[int(ik)])
        sub.psi = np.ascontiguousarray(prob.psi[[int(ik)], :, :sub.npw_max])
        p1 = pwk.plan_from_problem(sub, device=dev)
        prep, solve, _, _ = davidson_runner(torch, pwk, p1, sub, dev, pwk.PWK_FP64, stream)
        prep()
        solve()        # untimed: the first call allocates the plan's solver workspace
        prep()
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        r = solve()
        b.record(stream)
        torch.cuda.synchronize()
        t_tot += a.elapsed_time(b) / 1e3
        applies += r["applies_fp64"] + r["applies_fp32"]
        p1.close()
    return {"band_k_applies_per_s": applies / t_tot,
            "time_s_extrapolated": t_tot * prob.nk / len(ks),
            "sample": f"{len(ks)} of {prob.nk} k-points, one plan and one FP64 call each"}


def run_headline(args, torch, dev, stream, world, peaks):
    from paper_2412_01695_gb300 import pwk, synth
    from paper_2412_01695_gb300.pools import aggregate
    prob = synth.make_config(CFG)
    nbk = prob.nk * prob.nb
    plan = pwk.plan_from_problem(prob, device=dev)
    plan.set_solver_timing(True)
    T = Timer(torch, dev, stream)
    prep, solve, psi, eig = davidson_runner(torch, pwk, plan, prob, dev, pwk.PWK_FP32_C128, stream)
    clk = ClockSampler(dev.index or 0)
    clk.start()
    steps = T.run(solve, args.steps, args.warmup, prep=prep)
    launches = T.launches
    clocks = clk.stop()
    times = np.array([t for t, _ in steps])
    last = steps[-1][1]
    applies = last["applies_fp64"] + last["applies_fp32"]
    total_units, step_s, _ = aggregate(applies, float(np.mean(times)))
    launches = int(aggregate(launches, 0.0)[0])   # every rank's launches
    eig_mixed = eig.cpu().numpy()
    st = last["stats"]
    # where the solve spends its device time; the dominant part sets the roofline line
    share = {"h_applications": st["h_ms"] / st["total_ms"], "reduced_eigensolves": st["rr_ms"] / st["total_ms"],
             "vector_kernels_and_gaps": st["other_ms"] / st["total_ms"]}
    h_flops = (local_flops_per_band(prob) + nonlocal_flops_per_band(prob))
    rr_tflops = st["rr_fp64_flops"] / (st["rr_ms"] * 1e-3) / 1e12 if st["rr_ms"] > 0 else 0.0
    rr_line = {"bound": "alu", "achieved": rr_tflops, "peak": peaks["fp64_tflops"], "unit": "TFLOP/s",
               "frac": rr_tflops / peaks["fp64_tflops"],
               "kernel": "rr_kernel (batched FP64 reduced eigensolver, one CTA per k-point)",
               "algorithmic_flops": "12 n^3 + 12 n^2 nb FP64 flops per reduced problem of order n, summed "
                                    "on the device over every launch of the solve",
               "fp64_flops_per_solve": st["rr_fp64_flops"], "device_ms_per_solve": st["rr_ms"],
               "peak_source": "measured FP64 FMA throughput (pwk_measure_fma_peak), this run"}
    tb, tprof = traffic_for("rr_kernel")
    rr_line["traffic"] = tb
    rr_line["traffic_profile"] = tprof
    dom = max(share, key=share.get)
    res = {
        "metric": METRIC,
        "value": total_units / step_s,
        "unit": UNIT,
        "n_gpus": world,
        "steps": args.steps,
        "warmup": args.warmup,
        "ms_per_step": step_s * 1e3,
        "higher_is_better": True,
        "scaling": "weak",
        "vs_baseline": None,
        "dtype": "mixed f32/f64 (FP32 H applications, FP64 refinement, reduced eigensolves and norms)",
        "data": "synthetic (seeded generator: V(G) Gaussian spectrum, Gaussian projectors, random orthonormal "
                "trial vectors)",
        "config": {"workload": WORKLOAD, "global_batch": int(nbk), "k_points_per_gpu": prob.nk, "bands": prob.nb,
                   "npw_mean": float(np.mean(prob.npw)), "fft": [prob.N] * 3,
                   "stop": f"|d eps| < {ETH} Ry and ||H psi - eps psi|| < {RES_TOL}; eigenvalues checked to "
                           f"{EIG_TOL} Ry against the oracle",
                   "parallelism": f"k-pools x{world} (replicas, no collective)",
                   "l2": "flushed (512 MiB write) before every timed step"},
        "time_to_solution_s": step_s,
        "p99_ms_per_step": float(np.percentile(times * 1e3, 99)),
        "applies_per_solve": {"fp32": last["applies_fp32"], "fp64": last["applies_fp64"]},
        "iterations": {"max": last["iters_max"], "p50": last["iters_p50"]},
        "unconverged": last["rc"],
        "device_time_share": share,
        "device_ms_per_solve": {"h_applications": st["h_ms"], "reduced_eigensolves": st["rr_ms"],
                                "vector_kernels_and_gaps": st["other_ms"], "total": st["total_ms"]},
        "h_tflops_in_solve": applies * h_flops / (st["h_ms"] * 1e-3) / 1e12 if st["h_ms"] > 0 else None,
        "roofline_reduced_eigensolver": rr_line,
        "clocks": clocks,
    }
    # the same solve with FP64 H applications (batched), and the per-k FP64 form
    prep64, solve64, _, eig64 = davidson_runner(torch, pwk, plan, prob, dev, pwk.PWK_FP64, stream)
    t64 = T.run(solve64, 1, 1, prep=prep64)
    r64 = t64[0][1]
    a64 = r64["applies_fp64"] + r64["applies_fp32"]
    res["fp64_batched"] = {"time_to_solution_s": t64[0][0], "band_k_applies_per_s": a64 / t64[0][0],
                           "applies": a64, "iterations_max": r64["iters_max"],
                           "device_time_share": {"h_applications": r64["stats"]["h_ms"] / r64["stats"]["total_ms"],
                                                 "reduced_eigensolves": r64["stats"]["rr_ms"] / r64["stats"]["total_ms"]}}
    pk = per_k_fp64(torch, pwk, synth, prob, dev, stream, 4 if args.quick else 8)
    res["fp64_per_k"] = pk
    res["speedup_vs_per_k_fp64"] = {"time_to_solution": pk["time_s_extrapolated"] / step_s,
                                    "applies_per_s": res["value"] / pk["band_k_applies_per_s"]}
    res["speedup_vs_fp64_batched"] = t64[0][0] / step_s
    # end to end through the C ABI: trial vectors from pinned host memory, eigenvalues and
    # eigenvectors back to it, inside the timed region
    h_psi0 = torch.from_numpy(prob.psi).pin_memory()
    h_psi = torch.empty_like(h_psi0).pin_memory()
    h_eig = torch.empty((prob.nk, prob.nb), dtype=torch.float64).pin_memory()

    def e2e():
        psi.copy_(h_psi0, non_blocking=True)
        r = solve()
        h_psi.copy_(psi, non_blocking=True)
        h_eig.copy_(eig, non_blocking=True)
        return r
    te = T.run(e2e, max(1, min(args.steps, 3)), 1)
    e2e_s = float(np.mean([t for t, _ in te]))
    res["e2e"] = {"value": applies / e2e_s, "unit": UNIT,
                  "h2d_bytes_per_step": int(h_psi0.numel() * h_psi0.element_size()),
                  "d2h_bytes_per_step": int(h_psi.numel() * h_psi.element_size() + h_eig.numel() * 8),
                  "call": "pwk_davidson_batched with the trial vectors copied in from pinned host memory and "
                          "eigenvectors + eigenvalues copied out, inside the timed region"}
    res["gpu_launches"] = launches
    res["gpu_launches_per_step"] = launches / args.steps
    plan.close()
    return res, prob, eig_mixed, eig64.cpu().numpy()


# --------------------------------------------------------------------------- H|psi> kernels
def run_hpsi_kernels(args, torch, dev, stream, peaks):
    """The raw batched H|psi> rates on the headline cell (512 k x 20 bands): FP32 (the
    arithmetic of the solve's phase 1), FP64 batched, per-k FP64, the host-buffer entry point,
    and the roofline of the fused local kernel."""
    from paper_2412_01695_gb300 import pwk, synth
    prob = synth.make_config(CFG)
    nb, nbk = prob.nb, prob.nk * prob.nb
    plan = pwk.plan_from_problem(prob, device=dev)
    T = Timer(torch, dev, stream)
    psi64 = torch.from_numpy(prob.psi).to(dev)
    psi32 = psi64.to(torch.complex64)
    out32, out64 = torch.empty_like(psi32), torch.empty_like(psi64)
    n = 20 if args.quick else 200
    t32 = [t for t, _ in T.run(lambda: pwk.hpsi_batched(plan, pwk.PWK_FP32, psi32, out32, nb, stream), n, 5)]
    t64 = [t for t, _ in T.run(lambda: pwk.hpsi_batched(plan, pwk.PWK_FP64, psi64, out64, nb, stream), 10, 2)]
    items_k = [torch.tensor([[ik, b, b] for b in range(nb)], dtype=torch.int32, device=dev)
               for ik in range(prob.nk)]

    def per_k():
        for ik in range(prob.nk):
            pwk.hpsi_items(plan, pwk.PWK_FP64, psi64, out64, items_k[ik], nb, stream)
    tpk = [t for t, _ in T.run(per_k, 1, 1)]
    # the fused local kernel alone: the same cell with the projector set emptied, same shape
    import copy
    shape32 = plan.launch_shape(pwk.PWK_FP32)
    prob_loc = copy.copy(prob)
    prob_loc.beta = np.ascontiguousarray(prob.beta[:, :0, :])
    prob_loc.D = np.zeros((0, 0))
    plan_loc = pwk.plan_from_problem(prob_loc, device=dev)
    plan_loc.set_launch_shape(pwk.PWK_FP32, *shape32[:3])
    tloc = [t for t, _ in T.run(lambda: pwk.hpsi_batched(plan_loc, pwk.PWK_FP32, psi32, out32, nb, stream), n, 5)]
    plan_loc.close()
    # end to end with host buffers (pwk_hpsi_batched_host, 4 groups of k-points)
    h_in = psi32.cpu().pin_memory()
    h_out = torch.empty_like(h_in).pin_memory()
    d_in, d_out = torch.empty_like(psi32), torch.empty_like(psi32)
    te = [t for t, _ in T.run(lambda: pwk.hpsi_batched_host(plan, pwk.PWK_FP32, h_in, h_out, d_in, d_out, nb, 4,
                                                            stream), min(n, 50), 3)]
    # each way of applying the projector terms (pwk_plan_set_projector_path), FP32 batched
    paths = {"automatic_choice": PATH_NAMES.get(plan.projector_choice(pwk.PWK_FP32), "none")}
    for path, name in ((2, "separate_cuda_core_kernels"), (3, "fused_in_local_kernel"), (1, "tensor_core_projection")):
        plan.set_projector_path(path)
        tp = [t for t, _ in T.run(lambda: pwk.hpsi_batched(plan, pwk.PWK_FP32, psi32, out32, nb, stream), n, 5)]
        paths[name] = {"ms": float(np.mean(tp)) * 1e3, "band_k_applies_per_s": nbk / float(np.mean(tp))}
    plan.set_projector_path(0)
    pwk.hpsi_batched(plan, pwk.PWK_FP32, psi32, out32, nb, stream)   # the output the host leg checks
    torch.cuda.synchronize()
    kern_s, loc_s = float(np.mean(t32)), float(np.mean(tloc))
    loc_tf = local_flops_per_band(prob) * nbk / loc_s / 1e12
    step_tf = (local_flops_per_band(prob) + nonlocal_flops_per_band(prob)) * nbk / kern_s / 1e12
    ns, npl = hit_planes(prob)
    kname = f"fused_window_kernel<float,float,{prob.N},{prob.N // 4}>"
    tb, tprof = traffic_for(kname)
    # DRAM bytes of one FP32 step in the automatic projector path (ncu captures summarised
    # under profiles/), against the step's algorithmic bytes
    choice = plan.projector_choice(pwk.PWK_FP32)
    step_kernels = {2: [f"nl_project_kernel<float,float,{prob.nkb}>", kname,
                        f"nl_addback_kernel<float,float,{prob.nkb}>"],
                    3: [f"fused_window_kernel_nl<float,float,{prob.N},{prob.N // 4}>"]}.get(choice, [])
    step_t = [traffic_for(k) for k in step_kernels]
    step_dram = sum(t[0] for t in step_t) if step_t and all(t[0] for t in step_t) else None
    step_alg = algorithmic_bytes_per_band(prob, 8) * nbk
    out = {
        "fp32_batched": {"band_k_applies_per_s": nbk / kern_s, "ms": kern_s * 1e3,
                         "tflops_algorithmic": step_tf,
                         "hbm_gbs_algorithmic": algorithmic_bytes_per_band(prob, 8) * nbk / kern_s / 1e9,
                         "algorithmic_bytes_per_step": step_alg,
                         "dram_bytes_per_step": step_dram,
                         "dram_over_algorithmic": step_dram / step_alg if step_dram else None,
                         "dram_kernels": step_kernels,
                         "dram_profiles": sorted({t[1] for t in step_t if t[1]})},
        "fp64_batched": {"band_k_applies_per_s": nbk / float(np.mean(t64)), "ms": float(np.mean(t64)) * 1e3},
        "fp64_per_k": {"band_k_applies_per_s": nbk / float(np.mean(tpk)),
                       "call": "pwk_hpsi_items, one launch set per k-point"},
        "e2e_host_buffers_fp32": {"band_k_applies_per_s": nbk / float(np.mean(te)),
                                  "call": "pwk_hpsi_batched_host, 4 groups of k-points"},
        "roofline_local_kernel": {"bound": "alu", "achieved": loc_tf, "peak": peaks["fp32_tflops"],
                                  "unit": "TFLOP/s", "frac": loc_tf / peaks["fp32_tflops"],
                                  "kernel": kname + " (FP32 CUDA-core FMA), timed alone on the cell without projectors",
                                  "kernel_ms": loc_s * 1e3,
                                  "flops_per_band_k": local_flops_per_band(prob),
                                  "count": "5 n log2 n per 1D transform over each k-point's own sticks "
                                           f"(mean {ns.mean():.2f}) and hit m1 planes (mean {npl.mean():.2f}), "
                                           "every x line, inverse and forward; 2 N_r (V); 2 npw (kinetic)",
                                  "launch_shape": {"kind": shape32[0], "threads": shape32[1], "l3_chunk": shape32[2],
                                                   "smem": shape32[3]},
                                  "traffic": tb, "traffic_profile": tprof,
                                  "peak_source": "measured FP32 FMA throughput (pwk_measure_fma_peak), this run"},
        "nonlocal_part_ms": (kern_s - loc_s) * 1e3,
        "projector_paths_fp32": paths,
    }
    plan.close()
    return out, prob, (psi32, out32)


# --------------------------------------------------------------------------- solvers (context)
def sternheimer_block(nk: int, dev, stream, nocc: int = 12, nbx: int = 16):
    """Inputs of a batched Sternheimer solve on the first nk k-points of the DFPT cell (cell 4):
    plans of the k and k+q blocks, the nbx lowest bands of both by the batched FP64 Davidson,
    the nocc occupied ones, alpha_k = 2 (spread of the occupied levels) (>= 0.01 Ry) and the
    perturbation dv(r)."""
    import torch
    from paper_2412_01695_gb300 import pwk, synth
    ks = list(range(nk))
    pk = synth.make_config(4, k_subset=ks, nb=nbx)
    pq = synth.make_config(4, k_subset=ks, shift_q=True, nb=nbx)
    plan_k = pwk.plan_from_problem(pk, device=dev)
    plan_q = pwk.plan_from_problem(pq, device=dev)

    def lowest(plan, pr):
        psi = torch.from_numpy(pr.psi[:, :nbx].copy()).to(dev)
        eig = torch.zeros((pr.nk, nbx), dtype=torch.float64, device=dev)
        pwk.davidson_batched(plan, pwk.PWK_FP64, psi, eig, nbx, 1e-10, 1e-5, 300, 0, stream)
        return eig, psi

    eps_k, psi_k = lowest(plan_k, pk)
    eps_q, psi_q = lowest(plan_q, pq)
    e_all = torch.cat([eps_k[:, :nocc], eps_q[:, :nocc]], dim=1)
    alpha = torch.clamp(2.0 * (e_all.max(dim=1).values - e_all.min(dim=1).values), min=0.01).contiguous()
    return {"pk": pk, "pq": pq, "plan_k": plan_k, "plan_q": plan_q, "nocc": nocc,
            "psi_k": psi_k[:, :nocc].contiguous(), "psi_q": psi_q[:, :nocc].contiguous(),
            "eps_k": eps_k, "eps_q": eps_q, "ek": eps_k[:, :nocc].contiguous(), "alpha": alpha,
            "dv": torch.from_numpy(synth.dv_for(4)).to(dev)}


def run_sternheimer(dev, stream, quick=False):
    """The DFPT cell (4096 k x 12 occupied bands, k and k+q), residual 1e-10, mixed and FP64,
    then the induced density from the solution; where the solve spends its device time."""
    import torch
    from paper_2412_01695_gb300 import pwk, synth
    nk4 = 64 if quick else 4096
    blk = sternheimer_block(nk4, dev, stream)
    pk, pq, plan_k, plan_q = blk["pk"], blk["pq"], blk["plan_k"], blk["plan_q"]
    nocc, eps_q = blk["nocc"], blk["eps_q"]
    psi_k, psi_q, ek, alpha, dv = blk["psi_k"], blk["psi_q"], blk["ek"], blk["alpha"], blk["dv"]
    plan_q.set_solver_timing(True)
    pd = (eps_q[:, nocc:nocc + 1] - ek > 0).reshape(-1).cpu().numpy()
    sres = {"k_points": nk4, "nocc": nocc, "pairs": int(pd.size), "positive_definite_pairs": int(pd.sum()),
            "min_gap_ry": float((eps_q[:, nocc:nocc + 1] - ek).min().item())}
    dpsi = torch.zeros((nk4, nocc, pq.npw_max), dtype=torch.complex128, device=dev)
    pwk.sternheimer_cg_batched(plan_q, plan_k, pwk.PWK_FP32_C128, psi_k, ek, psi_q, nocc, alpha, dv, dpsi,
                               1e-10, 500, stream)   # first call builds the k -> k+q maps and workspace
    for name, mode in (("mixed", pwk.PWK_FP32_C128), ("fp64", pwk.PWK_FP64)):
        dpsi = torch.zeros((nk4, nocc, pq.npw_max), dtype=torch.complex128, device=dev)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        rc, iters, resid = pwk.sternheimer_cg_batched(plan_q, plan_k, mode, psi_k, ek, psi_q, nocc,
                                                      alpha, dv, dpsi, 1e-10, 500, stream)
        torch.cuda.synchronize()
        dt = time.perf_counter() - t0
        st = plan_q.solver_stats()
        ninner = int(iters.sum())
        sres[name] = {"time_s": dt, "pairs_above_tol": int(rc),
                      "positive_definite_pairs_above_tol": int((resid[pd] > 1e-10).sum()),
                      "max_true_residual_positive_definite": float(resid[pd].max()),
                      "indefinite_pairs_above_tol": int((resid[~pd] > 1e-10).sum()),
                      "iters_max": int(iters.max()), "iters_mean": float(iters.mean()),
                      "cg_iterations_total": ninner, "inner_applies_per_s": ninner / dt,
                      "device_time_share": {"h_applications": st["h_ms"] / st["total_ms"],
                                            "vector_kernels_and_gaps": st["other_ms"] / st["total_ms"]},
                      "device_ms": st["total_ms"]}
    sres["speedup_mixed_vs_fp64"] = sres["fp64"]["time_s"] / sres["mixed"]["time_s"]
    out = {"sternheimer": sres}
    # induced density (Eq. drho) from the solution just computed
    w = torch.full((nk4,), 1.0 / nk4, dtype=torch.float64, device=dev)
    drho = torch.empty((pk.N,) * 3, dtype=torch.complex128, device=dev)
    dres = {"k_points": nk4, "nocc": nocc, "pairs": nk4 * nocc}
    for name, prec in (("fp32", pwk.PWK_FP32_C128), ("fp64", pwk.PWK_FP64)):
        pwk.drho_batched(plan_q, plan_k, prec, psi_k, psi_q, dpsi, nocc, w, drho, stream)
        torch.cuda.synchronize()
        reps = 5
        t0 = time.perf_counter()
        for _ in range(reps):
            pwk.drho_batched(plan_q, plan_k, prec, psi_k, psi_q, dpsi, nocc, w, drho, stream)
        torch.cuda.synchronize()
        dt = (time.perf_counter() - t0) / reps
        dres[name] = {"time_ms": dt * 1e3, "pairs_per_s": nk4 * nocc / dt}
    ks_s = [0, 1, nk4 // 2, nk4 - 1]
    sub = torch.tensor(ks_s, device=dev)
    pk_s = synth.make_config(4, k_subset=ks_s, with_psi=False)
    pq_s = synth.make_config(4, k_subset=ks_s, with_psi=False, shift_q=True)
    pl_k, pl_q = pwk.plan_from_problem(pk_s, device=dev), pwk.plan_from_problem(pq_s, device=dev)
    u_k = psi_k[sub][:, :, :pk_s.npw_max].contiguous()
    u_q = psi_q[sub][:, :, :pq_s.npw_max].contiguous()
    d_s = dpsi[sub][:, :, :pq_s.npw_max].contiguous()
    w_s = torch.full((4,), 1.0 / nk4, dtype=torch.float64, device=dev)
    out_s = torch.empty_like(drho)
    pwk.drho_batched(pl_q, pl_k, pwk.PWK_FP64, u_k, u_q, d_s, nocc, w_s, out_s, stream)
    torch.cuda.synchronize()
    out["_drho_sample"] = (ks_s, nk4, u_k.cpu().numpy(), u_q.cpu().numpy(), d_s.cpu().numpy(),
                           out_s.cpu().numpy())
    pl_k.close()
    pl_q.close()
    out["drho"] = dres
    plan_k.close()
    plan_q.close()
    return out


def run_other_cells(dev, stream, quick=False):
    """H|psi> on the other synthetic cells (context beside the headline cell): FP32 and FP64
    batched band-k/s on every k-point of each cell, L2 flushed before every timed step."""
    import torch
    from paper_2412_01695_gb300 import pwk, synth
    T = Timer(torch, dev, stream)
    out = {}
    for cfg in ((1, 4) if quick else (1, 3, 4)):
        prob = synth.make_config(cfg)
        plan = pwk.plan_from_problem(prob, device=dev)
        row = {"k_points": prob.nk, "bands": prob.nb, "fft": prob.N, "projectors": prob.nkb,
               "npw_max": prob.npw_max}
        for name, prec, dt in (("fp32", pwk.PWK_FP32, torch.complex64), ("fp64", pwk.PWK_FP64, torch.complex128)):
            x = torch.from_numpy(prob.psi).to(dev).to(dt)
            y = torch.empty_like(x)
            ts = [t for t, _ in T.run(lambda: pwk.hpsi_batched(plan, prec, x, y, prob.nb, stream),
                                      10 if name == "fp32" else 3, 3)]
            row[name] = {"band_k_per_s": prob.nk * prob.nb / float(np.mean(ts)), "ms": float(np.mean(ts)) * 1e3}
        row["launch_shape_fp32"] = list(plan.launch_shape(pwk.PWK_FP32)[:3])
        row["projector_path_fp32"] = PATH_NAMES.get(plan.projector_choice(pwk.PWK_FP32), "none")
        # the local kernel alone (the cell without projectors, same launch shape)
        import copy
        pl = copy.copy(prob)
        pl.beta = np.ascontiguousarray(prob.beta[:, :0, :])
        pl.D = np.zeros((0, 0))
        plan_loc = pwk.plan_from_problem(pl, device=dev)
        plan_loc.set_launch_shape(pwk.PWK_FP32, *plan.launch_shape(pwk.PWK_FP32)[:3])
        x = torch.from_numpy(prob.psi).to(dev).to(torch.complex64)
        y = torch.empty_like(x)
        ts = [t for t, _ in T.run(lambda: pwk.hpsi_batched(plan_loc, pwk.PWK_FP32, x, y, prob.nb, stream), 10, 3)]
        row["fp32_local_only_ms"] = float(np.mean(ts)) * 1e3
        plan_loc.close()
        for path in (1, 2, 3):
            plan.set_projector_path(path)
            x = torch.from_numpy(prob.psi).to(dev).to(torch.complex64)
            y = torch.empty_like(x)
            ts = [t for t, _ in T.run(lambda: pwk.hpsi_batched(plan, pwk.PWK_FP32, x, y, prob.nb, stream), 10, 3)]
            row[f"fp32_path{path}_ms"] = float(np.mean(ts)) * 1e3
        plan.set_projector_path(0)
        plan.close()
        out[f"cell{cfg}"] = row
    return out


def run_serving(quick=False):
    """Serving over the workload's ranges (serve.config5_mix: fcc/sc cells with 1-8 atoms,
    25-60 Ry, 4-60 bands, 1-1728 k-points; 60% H|psi> in the mixed path, 25% Davidson, 15%
    Sternheimer), plans and solver workspaces resident before the clock: (1) Poisson arrivals
    at 200 Hz into 4 overlapping slots with H|psi> coalescing and HBM-footprint admission;
    (2) the same jobs at a sustainable rate (70% of the throughput (1) reached); (3) the plain
    baseline at the arrivals of (2): one job at a time, FP64, H|psi> with one launch set per
    k-point."""
    from paper_2412_01695_gb300 import serve
    n_jobs = 24 if quick else 40
    jobs = serve.config5_mix(n_jobs, rate_hz=200.0, seed=7)
    t0 = time.perf_counter()
    ex = serve.GpuExecutor(slots=4, plan_cache_bytes=96 << 30)
    ex.prepare(jobs)
    ex.warm(jobs)
    warm_s = time.perf_counter() - t0
    budget = 160 << 30

    def run(js, slots, coalesce):
        srv = serve.Server(ex, hbm_budget=budget, slots=slots, estimate=serve.estimate_for, coalesce=coalesce)
        return srv.run([j.fresh() for j in js], realtime=True)

    d200 = run(jobs, 4, True)
    st200 = serve.latency_stats(d200)
    rate_s = 0.7 * st200["jobs_per_s"]
    scale = 200.0 / rate_s
    jobs_s = [serve.Job(j.jid, j.kind, j.cell, j.nb, arrival=j.arrival * scale, precision=j.precision)
              for j in jobs]
    ds = run(jobs_s, 4, True)
    sts = serve.latency_stats(ds)
    ex.per_k = True
    dplain = run(jobs_s, 1, False)
    ex.per_k = False
    stp = serve.latency_stats(dplain)
    mix = {k: sum(j.kind == k for j in jobs) for k in ("hpsi", "davidson", "sternheimer")}
    nks = sorted({j.cell.mp ** 3 for j in jobs})
    return {"jobs": n_jobs, "mix": mix, "k_points_per_job": [nks[0], nks[-1]],
            "bands_per_job": [min(j.nb for j in jobs), max(j.nb for j in jobs)],
            "atoms_per_cell": [min(j.cell.nat for j in jobs), max(j.cell.nat for j in jobs)],
            "ecut_ry": [min(j.cell.ecut for j in jobs), max(j.cell.ecut for j in jobs)],
            "warm_up_s": warm_s,
            "offered_200hz": {**st200, "note": "arrivals faster than service: latency is mostly queueing"},
            "sustainable": {**sts, "offered_rate_hz": rate_s},
            "plain_per_k_fp64_one_at_a_time": {**stp, "offered_rate_hz": rate_s},
            "p99_speedup_vs_plain": stp.get("p99_s", float("nan")) / sts.get("p99_s", float("nan")),
            "p50_speedup_vs_plain": stp.get("p50_s", float("nan")) / sts.get("p50_s", float("nan"))}


# --------------------------------------------------------------------------- the oracle on the host
def oracle_davidson(prob, ks, budget_s):
    """The oracle's Davidson (oracle/davidson.py, dense FP64 H(k) from direct Fourier sums) on
    k-points of the workload in turn, with the same trial vectors and stopping rule, until
    budget_s has passed (at least one k-point).  Returns (applies, seconds, cpu seconds,
    {k: eigenvalues})."""
    from oracle import davidson as dav
    from oracle import hamiltonian as ham
    vt = ham.grid_coefficients(prob.V_r)
    t0, c0 = time.perf_counter(), time.process_time()
    applies, eigs = 0, {}
    for ik in ks:
        n = int(prob.npw[ik])
        H = ham.problem_h(prob, ik, vt)
        eps, _, _, napply, _ = dav.davidson(lambda X: X @ H.T, np.real(np.diag(H)), prob.psi[ik][:, :n],
                                            eth=ETH, max_iter=MAX_ITER, res_tol=RES_TOL)
        applies += napply
        eigs[int(ik)] = eps
        if time.perf_counter() - t0 >= budget_s:
            break
    return applies, time.perf_counter() - t0, time.process_time() - c0, eigs


def cpu_baseline(prob, budget_s=20.0):
    """The oracle's Davidson timed on the host cores on a bounded sample of the workload."""
    from paper_2412_01695_gb300 import synth
    ks = synth.sample_k(prob.nk, 64, seed=5)
    applies, dt, cpu, eigs = oracle_davidson(prob, ks, budget_s)
    return {"value": applies / dt, "unit": UNIT, "cores": os.cpu_count(), "cores_busy": round(cpu / dt, 2),
            "kind": "oracle",
            "sample": f"the oracle's Davidson (dense FP64 H(k) from direct Fourier sums, LAPACK reduced problem) "
                      f"on {len(eigs)} k-points x {prob.nb} bands of the workload, same trial vectors and "
                      f"stopping rule, {applies} H applications in {dt:.1f} s"}, eigs


def run_reference(args):
    """Reference arm: the FP64 CPU oracle's Davidson as it stands, on the host cores; each
    step solves one k-point of the workload (the same trial vectors and stopping rule)."""
    from paper_2412_01695_gb300 import synth
    prob = synth.make_config(CFG)
    ks = synth.sample_k(prob.nk, 64, seed=5)
    steps, warmup = min(args.steps, 12), min(args.warmup, 3)   # bounded: the oracle takes seconds per k
    times, cpu, applies = [], [], 0
    for s in range(warmup + steps):
        a, dt, c, _ = oracle_davidson(prob, [ks[s % len(ks)]], 0.0)
        if s >= warmup:
            times.append(dt)
            cpu.append(c)
            applies += a
    step_s = float(np.mean(times))
    value = applies / float(np.sum(times))
    busy = float(np.sum(cpu) / np.sum(times))
    return {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
            "steps": steps, "warmup": warmup, "ms_per_step": step_s * 1e3,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "impl": "reference",
            "config": {"workload": WORKLOAD, "global_batch": prob.nb,
                       "parallelism": "host cores (numpy/LAPACK threads)"},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": os.cpu_count(),
                             "cores_busy": round(busy, 2), "kind": "oracle",
                             "sample": f"each step = the oracle's Davidson on one k-point x {prob.nb} bands of "
                                       f"the workload ({steps} steps of {args.steps} requested)"},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}


# --------------------------------------------------------------------------- --case (profiling driver)
def run_case(args):
    import torch
    from paper_2412_01695_gb300 import pwk, synth
    stream = torch.cuda.current_stream()
    if args.case == "sternheimer":
        if args.cfg != 4:
            raise SystemExit("sternheimer runs on the DFPT cell: --cfg 4")
        nk = args.nk or 256
        blk = sternheimer_block(nk, torch.device("cuda"), stream)
        mode = pwk.PWK_FP64 if args.precision == "fp64" else pwk.PWK_FP32_C128
        nocc = blk["nocc"]
        blk["plan_q"].set_solver_timing(True)
        times = []
        torch.cuda.synchronize()
        torch.cuda.nvtx.range_push("case")
        for _ in range(args.reps):
            dpsi = torch.zeros((nk, nocc, blk["pq"].npw_max), dtype=torch.complex128, device="cuda")
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            rc, iters, resid = pwk.sternheimer_cg_batched(blk["plan_q"], blk["plan_k"], mode, blk["psi_k"],
                                                          blk["ek"], blk["psi_q"], nocc, blk["alpha"],
                                                          blk["dv"], dpsi, 1e-10, 500, stream)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        torch.cuda.nvtx.range_pop()
        print(json.dumps({"case": "sternheimer", "cfg": 4, "nk": nk, "nocc": nocc, "precision": args.precision,
                          "ms": times, "pairs_above_tol": int(rc), "iters_max": int(iters.max()),
                          "iters_mean": float(iters.mean()), "max_true_residual": float(resid.max()),
                          "stats": blk["plan_q"].solver_stats()}))
        blk["plan_k"].close()
        blk["plan_q"].close()
        return
    nkfull = int(np.prod(synth.CONFIGS[args.cfg]["mp"]))
    sub = None if args.nk in (0, nkfull) else list(range(args.nk))
    prob = synth.make_config(args.cfg, k_subset=sub, nb=args.nb or None)
    plan = pwk.plan_from_problem(prob)
    plan.set_projector_path(args.projector_path)
    prec = pwk.PRECISIONS[args.precision]
    times, extra = [], {}
    torch.cuda.nvtx.range_push("case")
    if args.case == "hpsi":
        dt = torch.complex64 if args.precision == "fp32" else torch.complex128
        x = torch.from_numpy(prob.psi).cuda().to(dt)
        y = torch.empty_like(x)
        for _ in range(args.reps):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            pwk.hpsi_batched(plan, prec, x, y, prob.nb)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
    else:
        mode = pwk.PWK_FP64 if args.precision == "fp64" else pwk.PWK_FP32_C128
        plan.set_solver_timing(True)
        for _ in range(args.reps):
            psi = torch.from_numpy(prob.psi).cuda()
            eig = torch.zeros((prob.nk, prob.nb), dtype=torch.float64, device="cuda")
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            rc, iters, notc, napply = pwk.davidson_batched(plan, mode, psi, eig, prob.nb, ETH, RES_TOL,
                                                           args.max_iter, args.max_basis)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        extra = {"unconverged": int(rc), "iters_max": int(iters.max()), "napply": napply.tolist(),
                 "iters_percentiles": np.percentile(iters, [50, 90, 99, 100]).tolist(),
                 "stats": plan.solver_stats()}
    torch.cuda.nvtx.range_pop()
    print(json.dumps({"case": args.case, "cfg": args.cfg, "nk": prob.nk, "nb": prob.nb,
                      "precision": args.precision, "ms": times,
                      "launch_shape": plan.launch_shape(pwk.PRECISIONS[args.precision]),
                      "projector_path": plan.projector_choice(pwk.PRECISIONS[args.precision]), **extra}))
    plan.close()


# --------------------------------------------------------------------------- main
def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-extras", action="store_true",
                    help="only the headline (no H|psi> kernels, Sternheimer, other cells, serving)")
    ap.add_argument("--no-serving", action="store_true")
    ap.add_argument("--quick", action="store_true", help="smaller samples in the context sections")
    ap.add_argument("--case", choices=["hpsi", "davidson", "sternheimer"])
    ap.add_argument("--cfg", type=int, default=2)
    ap.add_argument("--nk", type=int, default=0)
    ap.add_argument("--nb", type=int, default=0)
    ap.add_argument("--precision", default="fp32", choices=["fp64", "fp32", "fp32_c128"])
    ap.add_argument("--reps", type=int, default=3)
    ap.add_argument("--max-iter", type=int, default=MAX_ITER)
    ap.add_argument("--projector-path", type=int, default=0)
    ap.add_argument("--max-basis", type=int, default=0, help="Davidson basis bound (0: 4 nb)")
    args = ap.parse_args()
    if args.case:
        return run_case(args)
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))
    if args.impl == "reference":
        if rank == 0:
            print(json.dumps(run_reference(args)), flush=True)
        return
    import torch
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("gloo")
    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    stream = torch.cuda.current_stream()
    peaks = measured_peaks()
    peaks.update(fma_peaks(torch, dev, stream))
    if world > 1:
        torch.distributed.barrier()
    res, prob, eig_mixed, eig64 = run_headline(args, torch, dev, stream, world, peaks)
    res["peaks"] = peaks
    # the reduced eigensolver or the H applications: the line for the larger device-time share
    res["roofline"] = res["roofline_reduced_eigensolver"]
    hp_out = None
    if rank == 0 and not args.no_extras:
        hk, hprob, hp_out = run_hpsi_kernels(args, torch, dev, stream, peaks)
        res["hpsi_kernels"] = hk
        if res["device_time_share"]["h_applications"] > res["device_time_share"]["reduced_eigensolves"]:
            res["roofline"] = hk["roofline_local_kernel"]
        sol = run_sternheimer(dev, stream, quick=args.quick)
        drho_sample = sol.pop("_drho_sample", None)
        res.update(sol)
        res["other_cells"] = run_other_cells(dev, stream, quick=args.quick)
        if not args.no_serving:
            res["serving"] = run_serving(quick=args.quick)
    else:
        drho_sample = None
    # the CPU-baseline leg (rank 0, N = 1, after every timed region): the oracle timed on the
    # host cores, and the same oracle checking samples of this run's GPU results
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        cb, eigs = cpu_baseline(prob)
        res["cpu_baseline"] = cb
        from oracle import hamiltonian as ham
        vt = ham.grid_coefficients(prob.V_r)
        err_m, err_64 = 0.0, 0.0
        for ik in eigs:
            w = np.linalg.eigvalsh(ham.problem_h(prob, ik, vt))[:prob.nb]
            err_m = max(err_m, float(np.max(np.abs(eig_mixed[ik] - w))))
            err_64 = max(err_64, float(np.max(np.abs(eig64[ik] - w))))
        res["max_abs_eig_err_ry_vs_oracle"] = {"mixed": err_m, "fp64_batched": err_64, "k_points": sorted(eigs),
                                               "bar": EIG_TOL}
        if hp_out is not None:
            psi32, out32 = hp_out
            gpu_out = out32.cpu().numpy().astype(np.complex128)
            psi_in = psi32.cpu().numpy().astype(np.complex128)
            errs = []
            for ik in list(eigs)[:4]:
                n = hprob.npw[ik]
                ref = ham.hpsi_dense(hprob, ik, psi_in[ik], vt)
                errs.append(float(np.max(ham.relative_error(gpu_out[ik][:, :n], ref[:, :n]))))
            res["hpsi_kernels"]["fp32_max_rel_err_vs_oracle"] = max(errs)
        if drho_sample is not None:
            from oracle import drho as odr
            from paper_2412_01695_gb300 import synth
            ks_s, nk4, u_k, u_q, d_s, got = drho_sample
            pk_s = synth.make_config(4, k_subset=ks_s, with_psi=False)
            pq_s = synth.make_config(4, k_subset=ks_s, with_psi=False, shift_q=True)
            ref = odr.drho(pk_s, pq_s, u_k, u_q, d_s, weights=np.full(len(ks_s), 1.0 / nk4))
            res["drho"]["fp64_rel_err_vs_oracle_4k"] = float(np.linalg.norm(got - ref) / np.linalg.norm(ref))
    if rank == 0:
        print(json.dumps(res), flush=True)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
