"""Benchmark of one leapfrog step of the SBP-SAT anisotropic elastic scheme on GB300.

Workload (default): the topography model -- 2 stacked curvilinear blocks of 4001 x 2001 nodes
(16,012,002 nodes), interior order 6, tilted VTI stiffness, traction-free surface, Robin sides,
welded interface, vertical Ricker point force at the surface, FP32 fields.  A "step" is one
leapfrog time step over all blocks (interior stencil, boundary strips, face SAT terms, source).

Prints ONE JSON line (rank 0).  Metric: grid-point updates per second (nodes x steps / s).

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference] [--precision fp32|fp64]

--impl reference times the FP64 CPU oracle (the reference implementation of this build) on a
bounded crop of the same workload, on the host cores.
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import workloads as W  # noqa: E402

METRIC = "grid-pt updates/s"
UNIT = "node-updates/s"
# algorithmic bytes per node of a leapfrog step.  FP64 (two levels): u^n 2, u^{n-1} 2, u^{n+1} 2,
# c 10, 1/(rho J) 1 = 17 words.  FP32 (increment form): u^n 2, d^n 2, d^{n+1} 2, u^{n+1} 2, c 10,
# 1/(rho J) 1 = 19 words
BYTES_PER_NODE = {"fp32": 76, "fp64": 136}
# DRAM bytes per node of one FP32 interior launch (dram__bytes_read.sum + dram__bytes_write.sum of
# k_interior_march_multi<6,3> captured at 2 x 1601x801, scaled by interior nodes).  Set to None whenever that
# kernel changes until it is measured again.
TRAFFIC_BYTES_PER_NODE = {"fp32": 73.0, "fp64": None}
FALLBACK_HBM_GBS = 6800.0
N1, N2 = 4001, 2001
# crop of the workload the oracle is timed on: a 401-column window around the source spanning
# the interface (block 0 top 161 rows, block 1 bottom 161 rows)
CROP = {0: (1800, 2201, N2 - 161, N2), 1: (1800, 2201, 0, 161)}


def workload_name(prec):
    return (f"topography 2x({N1}x{N2}) curvilinear blocks, order 6, tilted VTI, traction-free top, "
            f"Robin sides, interface, Ricker 8 Hz point force, {prec.upper()}")


def peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        try:
            d = json.load(open(p))
            for k in ("hbm_gbs", "hbm_GBs", "hbm"):
                if k in d:
                    v = d[k]
                    return float(v["value"] if isinstance(v, dict) else v), "measured"
        except Exception:
            pass
    return FALLBACK_HBM_GBS, "fallback"


class ClockSampler:
    """nvidia-smi clocks and throttle reasons around and during the timed region.  Samples every
    10 ms (a short timed region still gets samples), plus one query on entry and one on exit."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.idx = gpu_index
        self.proc = None
        self.f = None

    def _once(self):
        try:
            out = subprocess.run(["nvidia-smi", "-i", str(self.idx), f"--query-gpu={self.Q}",
                                  "--format=csv,noheader,nounits"], capture_output=True, text=True, timeout=10)
            return out.stdout.strip().splitlines()
        except Exception:
            return []

    def __enter__(self):
        self.edges = self._once()
        try:
            self.f = tempfile.NamedTemporaryFile("w+", suffix=".csv", delete=False)
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.idx), f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "10"],
                                         stdout=self.f, stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None
        return self

    def __exit__(self, *a):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()
        self.edges += self._once()

    @staticmethod
    def _parse(lines):
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in lines:
            r = [x.strip() for x in line.split(",")]
            try:
                sm.append(float(r[1]))
                mx.append(float(r[2]))
            except Exception:
                continue
            for n, v in zip(names, r[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(n)
        return sm, mx, reasons

    def summary(self):
        if self.proc is None or self.f is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.f.flush()
        loop = [x for x in open(self.f.name).read().strip().splitlines() if x.strip()]
        os.unlink(self.f.name)
        sm, mx, reasons = self._parse(loop)
        esm, emx, ereasons = self._parse(self.edges)
        # the median comes from the samples taken while the timed region ran; the queries on entry
        # and exit (right before and after it) stand in only when a very short region got none
        src = "during" if sm else "edges"
        med = statistics.median(sm) if sm else (statistics.median(esm) if esm else None)
        allmx = mx + emx
        return {"sm_mhz": med, "sm_max_mhz": max(allmx) if allmx else None,
                "reasons": sorted(reasons | ereasons), "samples": len(sm), "edge_samples": len(esm),
                "source": src}


def run_oracle_steps(prec_unused, steps, warmup):
    """Time the FP64 oracle's leapfrog steps on the bounded crop; returns (node-updates/s, detail)."""
    from oracle.scheme import Oracle
    P = W.config3(window=CROP)
    O = Oracle(P)
    dt = O.suggest_dt(0.3)
    u = O.pack(W.smooth_state(P))
    up = u.copy()
    for _ in range(warmup):
        up, u, _ = O.leapfrog(up, u, 0.0, dt, 1)
    t0 = time.perf_counter()
    up, u, _ = O.leapfrog(up, u, 0.0, dt, steps)
    el = time.perf_counter() - t0
    nodes = P.n_nodes
    return nodes * steps / el, dict(nodes=nodes, seconds=el, steps=steps)


def cpu_baseline(target_seconds=12.0):
    """The oracle as it stands, on a bounded crop of the workload (single host thread)."""
    t0 = time.perf_counter()
    rate, d = run_oracle_steps(None, 3, 1)
    # scale the number of timed steps to ~target_seconds of stepping
    per = d["seconds"] / d["steps"]
    n = max(3, min(60, int(target_seconds / max(per, 1e-6))))
    rate, d = run_oracle_steps(None, n, 0)
    return {"value": rate, "unit": UNIT, "cores": 1, "host_cores": os.cpu_count(), "kind": "oracle",
            "sample": f"{d['steps']} leapfrog steps of the FP64 oracle on a crop of the workload: 2 blocks "
                      f"of 401x161 nodes ({d['nodes']} nodes) around the source and interface; "
                      f"{time.perf_counter() - t0:.1f} s incl. assembly"}


class _ShotPrefetch:
    """Client side of the served batch: builds the shots' host inputs (grid, material, source) on
    a few worker threads, at most `ahead` requests beyond the one being admitted (bounded host
    memory), so that the requests reach the engine with their payload."""

    def __init__(self, specs, ahead=12, workers=4):
        from concurrent.futures import ThreadPoolExecutor
        self.specs, self.ahead = specs, ahead
        self.pool = ThreadPoolExecutor(workers)
        self.fut, self.next = {}, 0
        self._top_up(0)

    def _top_up(self, i):
        while self.next < len(self.specs) and self.next <= i + self.ahead:
            _, side, seed, _ = self.specs[self.next]
            self.fut[self.next] = self.pool.submit(W.shot_problem, side, seed)
            self.next += 1

    def get(self, i):
        self._top_up(i)
        return self.fut.pop(i).result()

    def close(self):
        self.pool.shutdown(wait=True)


def serving_bench(nshots=256, side_range=(201, 2001), tick=16, hbm_cap=16e9, sample_every=16):
    """Served batch (config 4 as stated): nshots single-block curvilinear shots, side ~ U(side_range),
    steps = 2 side, admission under an HBM cap (16 GB: admission binds), FP32 continuous batching
    on the persistent tile-queue kernel.  Two runs of the same requests:
      * saturated: every request is waiting at t = 0; solves/s = nshots / makespan is the serving
        path's capacity (the number compared with the one-at-a-time arms);
      * loaded: Poisson arrivals at 0.8 x that capacity; p50 / p99 latency (arrival to result).
    Baselines on a uniform sample (every sample_every-th request) run one solve at a time, back to
    back: the plain FP64 path (the target) and the same path in FP32 (which separates the batching
    gain from the precision gain); their solves/s = sample size / sample time.  Setup (grid,
    material, CFL) and the result read-back are inside every arm; the host-side shot construction
    is not (prefetched on worker threads for the batch, done before each timed solve for the
    baselines)."""
    import numpy as np
    import torch
    from paper_2003_12811_gb300 import Solver
    from paper_2003_12811_gb300.binding import FIELD_CUR
    from paper_2003_12811_gb300.serve import BatchServingEngine, GpuBatchBackend, Request, percentile
    base = W.config4_requests(nshots, side_range, rate=1.0, steps_per_side=2.0, step_multiple=2)
    work = float(np.mean([side * side * n for (_, side, _, n) in base]))
    node_updates = int(sum(side * side * n for (_, side, _, n) in base))

    def serve(arrivals):
        specs = [(a, side, seed, n) for a, (_, side, seed, n) in zip(arrivals, base)]
        pre = _ShotPrefetch(specs)
        reqs = [Request(rid=i, arrival=a, problem=(lambda i=i: pre.get(i)), nsteps=n)
                for i, (a, _, _, n) in enumerate(specs)]
        be = GpuBatchBackend(max_shots=nshots)
        eng = BatchServingEngine(int(hbm_cap), backend=be, tick_steps=tick, max_active=nshots)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        res = eng.run(reqs)
        torch.cuda.synchronize()
        served = time.perf_counter() - t0
        be.close()
        pre.close()
        return served, [r.latency for r in res], eng

    sat_s, sat_lat, sat_eng = serve([0.0] * nshots)
    capacity = nshots / sat_s                            # solves/s at saturation
    rate = 0.8 * capacity                                # arrivals per second of the loaded run
    loaded = W.config4_requests(nshots, side_range, rate=rate, steps_per_side=2.0, step_multiple=2)
    load_s, lat, eng = serve([a for (a, _, _, _) in loaded])

    def one_at_a_time(prec):
        tot = 0.0
        sample = base[::sample_every]
        for (_, side, seed, n) in sample:
            P = W.shot_problem(side, seed)
            torch.cuda.synchronize()
            t1 = time.perf_counter()
            S = Solver(P, prec)                         # state zero at t = 0, as for the batch
            dt = S.suggest_dt(0.3)
            S.sbp_step(n, dt)
            S.sbp_get_field(FIELD_CUR)
            S.close()
            torch.cuda.synchronize()
            tot += time.perf_counter() - t1
        return len(sample) / tot, len(sample), tot

    seq64, n64, t64 = one_at_a_time("fp64")
    seq32, n32, t32 = one_at_a_time("fp32")
    return {"workload": f"served batch (config 4): {nshots} shots, side U{list(side_range)}, steps = 2 side, FP32, "
                        f"HBM cap {hbm_cap / 1e9:.0f} GB, persistent tile-queue kernel, ticks of {tick} graph-replayed "
                        f"steps; saturated run (all requests at t = 0) and loaded run (Poisson arrivals "
                        f"{rate:.2f}/s = 0.8 x the saturated solves/s)",
            "solves_per_s": capacity, "makespan_s": sat_s, "node_updates_per_s": node_updates / sat_s,
            "mean_shot_node_updates": work,
            "loaded": {"arrivals_per_s": rate, "makespan_s": load_s, "solves_per_s": nshots / load_s,
                       "p50_latency_s": percentile(lat, 50), "p99_latency_s": percentile(lat, 99),
                       "peak_active": eng.peak_active, "peak_bytes": eng.peak_bytes, "ticks": eng.ticks},
            "p50_latency_s": percentile(lat, 50), "p99_latency_s": percentile(lat, 99),
            "fp64_one_at_a_time_solves_per_s": seq64, "fp32_one_at_a_time_solves_per_s": seq32,
            "baseline_sample": f"every {sample_every}th request ({n64} shots): FP64 {t64:.1f} s, FP32 {t32:.1f} s",
            "speedup_vs_fp64_one_at_a_time": capacity / seq64,
            "speedup_vs_fp32_one_at_a_time": capacity / seq32,
            "peak_active": sat_eng.peak_active, "peak_bytes": sat_eng.peak_bytes, "ticks": sat_eng.ticks,
            "host_phase_s": {k: round(v, 3) for k, v in sat_eng.phase_s.items()},
            "node_updates": node_updates}


# gradient interior kernel, per node: every level of the segment reads psi_n (2 words) and u_{n+1}
# (2 words; u_n, u_{n-1} stay in registers); once per launch g_c (10 r+w), g_rho (r+w), J (FP64)
# and the first two forward levels (4 words)
GRAD_BYTES_PER_NODE_LEVEL = {"fp32": 16, "fp64": 32}
GRAD_BYTES_PER_NODE_LAUNCH = {"fp32": 22 * 4 + 8 + 16, "fp64": 22 * 8 + 8 + 32}


def adjoint_bench(n=1001, nsteps=2000, prec="fp32"):
    """Misfit gradient (config 5): one curvilinear block n x n, 64 surface receivers, nsteps
    leapfrog steps; observations made by the model with the Gaussian inclusion, gradient of the L2
    misfit at the background model through the checkpointed discrete adjoint (sqrt(nsteps)
    checkpoints).  Also times the forward solve alone and profiles the gradient kernels."""
    import torch
    from paper_2003_12811_gb300 import Solver
    Pb, rec = W.config5(n=n, blob=False)
    Pt, _ = W.config5(n=n, blob=True)
    z = [np.zeros((2, n, n))]
    St = Solver(Pt, prec)
    dt = St.suggest_dt(0.3)
    St.set_state(z, z, 0.0)
    St.sbp_set_receivers(rec)
    obs = St.sbp_record(nsteps, dt)
    St.close()
    S = Solver(Pb, prec)
    S.set_state(z, z, 0.0)
    S.sbp_set_receivers(rec)
    tuning = S.sbp_autotune()
    S.sbp_misfit_gradient(20, dt, obs[:20])                   # warm-up (workspace, adjoint fields)
    S.set_state(z, z, 0.0)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    phi, gr, gc = S.sbp_misfit_gradient(nsteps, dt, obs)     # interval 0: every level kept if it fits
    torch.cuda.synchronize()
    grad_s = time.perf_counter() - t0
    # the memory-lean form: checkpoints every ceil(sqrt(N)) steps, each segment recomputed
    kc = int(math.ceil(math.sqrt(nsteps)))
    S.set_state(z, z, 0.0)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    S.sbp_misfit_gradient(nsteps, dt, obs, checkpoint_every=kc)
    torch.cuda.synchronize()
    grad_ck_s = time.perf_counter() - t0
    # forward alone, same steps
    S.set_state(z, z, 0.0)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    S.sbp_step(nsteps, dt)
    torch.cuda.synchronize()
    fwd_s = time.perf_counter() - t0
    # kernel families of one profiled gradient
    S.set_state(z, z, 0.0)
    S.sbp_profile(True)
    S.sbp_misfit_gradient(nsteps, dt, obs)
    fam_ms, fam_n = S.sbp_profile_read()
    S.sbp_profile(False)
    S.close()
    GS = 12                                                    # gradient interior starts 12 nodes from a face (order 6)
    inner = (n - 2 * GS) ** 2
    k_ms = fam_ms[4] / max(1, fam_n[4])
    levels = nsteps / max(1, fam_n[4])                         # levels per launch (one launch per segment)
    bpn = GRAD_BYTES_PER_NODE_LEVEL[prec] * levels + GRAD_BYTES_PER_NODE_LAUNCH[prec]
    achieved = bpn * inner / (k_ms / 1e3) / 1e9
    peak, src = peaks()
    names = ["interior", "boundary", "faces", "sources", "grad_interior", "grad_strips", "grad_faces_receivers", "misfit_output"]
    return {"workload": f"misfit gradient (config 5): 1 curvilinear block {n}x{n}, order 6, tilted VTI + Gaussian "
                        f"inclusion, 64 surface receivers, {nsteps} steps, {prec.upper()}, every forward level "
                        f"kept on the device ({2 * nsteps * 2 * n * ((n + 31) // 32 * 32) * (4 if prec == 'fp32' else 8) / 1e9:.0f} GB "
                        f"of forward and adjoint levels: no recomputation)",
            "gradients_per_s": 1.0 / grad_s, "ms_per_gradient": 1e3 * grad_s,
            "forward_ms": 1e3 * fwd_s, "gradient_over_forward": grad_s / fwd_s,
            "checkpointed": {"checkpoint_every": kc, "ms_per_gradient": 1e3 * grad_ck_s,
                             "gradient_over_forward": grad_ck_s / fwd_s},
            "tuning": {"rows_per_cta": tuning[0], "strips_concurrent": bool(tuning[1])},
            "misfit": phi, "grad_rho_absmax": float(np.abs(gr[0]).max()), "grad_C_absmax": float(np.abs(gc[0]).max()),
            "family_ms": {k: float(v) for k, v in zip(names, fam_ms)},
            "family_launches": {k: int(v) for k, v in zip(names, fam_n)},
            "roofline": {"kernel": "k_grad_interior", "bound": "hbm", "bytes_per_node": bpn, "levels_per_launch": levels,
                         "units_per_launch": inner,
                         "kernel_ms": k_ms, "achieved": achieved, "peak": peak, "unit": "GB/s",
                         "frac": achieved / peak, "peak_source": src, "traffic": None}}


# algorithmic words per node of the four RK4 stages (rk4_store): U_s (2), c (10), 1/(rho J) (1) each, and of the
# combination v | u, v, a_1 | u, v, a_2 | u, v, a_1, a_2, a_3 in, U_{s+1} and a_s (u_new twice and v_new last) out
RK4_WORDS_PER_STAGE = (4 * 13 + 2 + 6 + 6 + 10 + 3 * 4 + 6) / 4
# the wide operator: FP32 in one march over the interior (the words of the narrow step); FP64 in two passes, fluxes
# u (2) + c (10) -> G (4), divergence G (4), 1/(rho J) (1), u^n (2), u^{n-1} (2) -> u^{n+1} (2)
WIDE_WORDS_IMPLEMENTED = {"fp32": 19, "fp64": 27}


# FP64 operations of k_interior_edges<double, 6, 0, 32, 16> per interior node (ncu thread-level counts
# 2 x DFMA + DADD + DMUL over the 599,778 interior nodes of 2 x 801 x 401), and the FP64 peak
# of the part: 152 SMs x 2 FP64 FMA per clock x 2 flops x 2.07 GHz
FP64_FLOPS_PER_NODE = 227.3
FP64_PEAK_TFLOPS = 152 * 2 * 2 * 2.07e9 / 1e12


def fp64_bench(P, nsteps=20):
    """The FP64 path on the bench workload: node updates/s, the interior kernel's share, and its
    rooflines: HBM at 136 B/node and the FP64 ALU (the bound this path actually meets)."""
    import torch
    from paper_2003_12811_gb300 import Solver
    nodes = P.n_nodes
    S = Solver(P, "fp64")
    dt = S.suggest_dt(0.3)
    zero = [np.zeros((2, b.N2, b.N1)) for b in P.blocks]
    S.set_state(zero, zero, 0.0)
    S.sbp_step(2, dt)
    stream = torch.cuda.current_stream()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    S.sbp_step(nsteps, dt)
    e1.record(stream)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / nsteps
    S.sbp_profile(True)
    S.sbp_step(4, dt)
    fam_ms, fam_n = S.sbp_profile_read()
    S.sbp_profile(False)
    S.close()
    inner = sum((b.N1 - 18) * (b.N2 - 18) for b in P.blocks)
    k_ms = fam_ms[0] / 4
    peak, src = peaks()
    tflops = FP64_FLOPS_PER_NODE * inner / (k_ms / 1e3) / 1e12
    return {"node_updates_per_s": nodes / (ms / 1e3), "ms_per_step": ms, "interior_ms_per_step": k_ms,
            "hbm": {"bytes_per_node": BYTES_PER_NODE["fp64"], "achieved_GBs": BYTES_PER_NODE["fp64"] * inner / (k_ms / 1e3) / 1e9,
                    "frac": BYTES_PER_NODE["fp64"] * inner / (k_ms / 1e3) / 1e9 / peak, "peak_source": src},
            "alu": {"bound": "alu", "kernel": "k_interior_edges<double,6,0>", "flops_per_node": FP64_FLOPS_PER_NODE,
                    "achieved": tflops, "peak": FP64_PEAK_TFLOPS, "unit": "TFLOP/s", "frac": tflops / FP64_PEAK_TFLOPS,
                    "peak_source": "derived: 152 SMs x 2 FP64 FMA per clock x 2 flops x 2.07 GHz"},
            "steps": nsteps}


# 3-D operator: words per node each bulk kernel must move (FP32 words; FP64 doubles them)
#   k3_flux: u (3) and the 27 mixed coefficients in, the 9 fluxes q out            = 39
#   divergence (k3_div with k3_lines): q (9), the 18 narrow coefficients, w, u (3), du (3) in; du, u^{n+1} out = 40
#   one fused pass at the minimum: u, du, 45 coefficients, w in; du, u^{n+1} out     = 58
OP3D_WORDS = {"k3_flux": 39, "divergence": 40, "fused_min": 58}


def bench3d(n=256, nsteps=40, prec="fp32"):
    """The 3-D operator on one curvilinear block of n^3 nodes (order 6; tilted transversely
    isotropic medium with smooth heterogeneity; topography-like top face with traction, five
    displacement faces): leapfrog node updates/s and the rooflines of the two bulk kernels
    (CUDA events on the launch stream)."""
    import torch
    from workloads import box3d as B3
    from paper_2003_12811_gb300 import Solver3D
    N = (n, n, n)
    faces = ("displacement",) * 5 + ("traction",)
    X = B3.block3_coords(N)
    S = Solver3D(X, faces, 6, prec)
    for k0 in range(0, n, 32):
        k1 = min(n, k0 + 32)
        rho, Pm = B3.material3_planes(N, k0=k0, k1=k1)
        S.sbp3_set_material(k0, k1 - k0, rho, Pm)
    # a stable step for the medium: 0.2 x (smallest spacing of the deformed box) / (fastest P speed)
    hmin = min(np.abs(np.diff(X[0], axis=2)).min(), np.abs(np.diff(X[1], axis=1)).min(),
               np.abs(np.diff(X[2], axis=0)).min())
    del X
    dt = 0.2 * hmin / (2.3 * np.sqrt(1.3))
    g1, g2, g3 = B3.ref_grid3(*N)
    u = np.array([np.sin(np.pi * g1) * np.sin(np.pi * g2) * np.sin(np.pi * g3 / 2)] * 3)
    del g1, g2, g3
    S.set_state(u, u)
    del u
    variant, variant_ms = S.sbp3_autotune()           # launch shape of the interior kernel
    stream = torch.cuda.current_stream()
    sh = stream.cuda_stream
    S.step(3, dt, sh)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    S.step(nsteps, dt, sh)
    e1.record(stream)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / nsteps
    S.profile(True)
    S.step(4, dt, sh)
    fam_ms, fam_n = S.profile_read()
    S.profile(False)
    a, b = S.state()
    finite = bool(np.isfinite(b).all())
    S.close()
    nodes = n ** 3
    es = 4 if prec == "fp32" else 8
    peak, src = peaks()
    kern = {}
    for f, name in enumerate(("k3_flux", "k3_div", "k3_lines")):
        kern[name] = {"ms_per_step": fam_ms[f] / 4, "launches": fam_n[f]}
    for name, kms in (("k3_flux", kern["k3_flux"]["ms_per_step"]),
                      ("divergence", kern["k3_div"]["ms_per_step"] + kern["k3_lines"]["ms_per_step"])):
        gbs = OP3D_WORDS[name] * es * nodes / (kms / 1e3) / 1e9
        kern.setdefault(name, {"ms_per_step": kms})
        kern[name].update({"bytes_per_node": OP3D_WORDS[name] * es, "achieved_GBs": gbs, "frac": gbs / peak})
    fused = OP3D_WORDS["fused_min"] * es * nodes / (ms / 1e3) / 1e9
    return {"workload": f"3-D block {n}^3 nodes, order 6, {prec.upper()}, leapfrog in increment form",
            "node_updates_per_s": nodes / (ms / 1e3), "ms_per_step": ms, "kernels": kern,
            "step_vs_fused_minimum": {"bytes_per_node": OP3D_WORDS["fused_min"] * es, "achieved_GBs": fused,
                                      "frac": fused / peak},
            "peak_GBs": peak, "peak_source": src, "launches_per_step": 4, "steps": nsteps, "state_finite": finite,
            "tuning": {"variant": variant, "apply_ms_per_variant": variant_ms}}


def variant_bench(P, prec, nsteps=100):
    """The time integrator and operator variants on the bench workload: RK4 steps (the paper's
    integrator; four fused stage passes per step) and leapfrog steps of the wide-stencil operator,
    node-updates/s with the bandwidth their traffic implies (CUDA events on the launch stream)."""
    import dataclasses
    import torch
    from paper_2003_12811_gb300 import Solver
    es = 4 if prec == "fp32" else 8
    nodes = P.n_nodes
    peak, src = peaks()
    out = {}
    zero = [np.zeros((2, b.N2, b.N1)) for b in P.blocks]
    stream = torch.cuda.current_stream()
    sh = stream.cuda_stream
    # RK4
    S = Solver(P, prec)
    dt = S.suggest_dt(0.5)
    S.sbp_set_state_rk4(zero, zero, 0.0)
    S.sbp_step_rk4(3, dt, sh)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    S.sbp_step_rk4(nsteps, dt, sh)
    e1.record(stream)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / nsteps
    S.close()
    gbs = 4 * RK4_WORDS_PER_STAGE * es * nodes / (ms / 1e3) / 1e9
    out["rk4"] = {"node_updates_per_s": nodes / (ms / 1e3), "ms_per_step": ms, "cfl": 0.5,
                  "bytes_per_node_per_step": 4 * RK4_WORDS_PER_STAGE * es, "achieved_GBs": gbs,
                  "frac_of_peak": gbs / peak, "peak_source": src, "steps": nsteps}
    # wide stencil, leapfrog
    S = Solver(dataclasses.replace(P, stencil="wide"), prec)
    dtw = S.suggest_dt(0.3)
    S.set_state(zero, zero, 0.0)
    S.sbp_step(3, dtw, sh)
    torch.cuda.synchronize()
    e0.record(stream)
    S.sbp_step(nsteps, dtw, sh)
    e1.record(stream)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / nsteps
    S.close()
    bpn = BYTES_PER_NODE[prec]
    out["wide"] = {"node_updates_per_s": nodes / (ms / 1e3), "ms_per_step": ms,
                   "algorithmic_GBs": bpn * nodes / (ms / 1e3) / 1e9,
                   "frac_of_peak_algorithmic": bpn * nodes / (ms / 1e3) / 1e9 / peak,
                   "implemented_words_per_node": WIDE_WORDS_IMPLEMENTED[prec],
                   "implemented_GBs": WIDE_WORDS_IMPLEMENTED[prec] * es * nodes / (ms / 1e3) / 1e9,
                   "peak_source": src, "steps": nsteps}
    return out


def accuracy_table():
    """FP32 against FP64 after each configuration's own step count (configs 1-3 at their stated
    sizes; the FP64 GPU path is the reference: the parity tests hold it to the oracle at 1e-12,
    at full size included), and the l2 error against the manufactured solution where one exists
    (configs 1 and 2).  Norms: the scheme's J H-weighted l2 (sbp_l2_diff, FP64 on the device)."""
    import torch
    from paper_2003_12811_gb300 import Solver
    from paper_2003_12811_gb300.binding import FIELD_CUR

    def run(P, prec, nsteps, dt, up, uc):
        S = Solver(P, prec)
        S.set_state(up, uc, 0.0)
        out = {}
        done = 0
        for mark in sorted(nsteps):
            S.sbp_step(mark - done, dt)
            done = mark
            _, u = S.state()
            t = S.sbp_get_time()
            err_exact = None
            if P.exact is not None:
                e2, _ = S.sbp_l2_diff(FIELD_CUR, [P.exact(b, t) for b in P.blocks])
                err_exact = math.sqrt(e2)
            out[mark] = (u, err_exact)
        return S, out

    table = {}
    cases = [("config 1: 101^2 Cartesian, order 4, manufactured solution", lambda: W.config1(), [200], 0.25, True),
             ("config 2: 4 x 801^2 curvilinear, order 6, manufactured solution", lambda: W.config2(n=801), [1000], 0.25, True),
             ("config 3: 2 x 4001x2001 topography, order 6, Ricker source", lambda: W.config3(), [1000, 5000], 0.3, False)]
    for name, make, marks, cfl, mms in cases:
        P = make()
        S64 = Solver(P, "fp64")
        dt = S64.suggest_dt(cfl)
        S64.close()
        if mms:
            up = [P.exact(b, -dt) for b in P.blocks]
            uc = [P.exact(b, 0.0) for b in P.blocks]
        else:
            up = uc = [np.zeros((2, b.N2, b.N1)) for b in P.blocks]
        t0 = time.perf_counter()
        S64, r64 = run(P, "fp64", marks, dt, up, uc)
        S32, r32 = run(P, "fp32", marks, dt, up, uc)
        rows = {}
        for m in marks:
            u64, e64 = r64[m]
            u32, e32 = r32[m]
            # relative l2 in the scheme's norm: the FP32 field against the FP64 field
            Sref = Solver(P, "fp32")
            Sref.set_state(u32, u32, 0.0)
            e2, r2 = Sref.sbp_l2_diff(FIELD_CUR, u64)
            Sref.close()
            relmax = max(np.abs(a - b).max() for a, b in zip(u32, u64)) / max(np.abs(b).max() for b in u64)
            rows[str(m)] = {"fp32_rel_l2_vs_fp64": math.sqrt(e2 / r2), "fp32_rel_max_vs_fp64": relmax,
                            "l2_error_exact_fp64": e64, "l2_error_exact_fp32": e32}
        S64.close()
        S32.close()
        table[name] = {"dt": dt, "steps": rows, "seconds": time.perf_counter() - t0}
        torch.cuda.synchronize()
    return table


def accuracy3d(n=96, nsteps=(200, 1000)):
    """The 3-D operator in FP32 (increment form) against FP64 on a curvilinear n^3 block (order 6,
    the bench medium and faces), relative l2 of u after each mark; the FP64 path is the reference
    (the parity tests hold it to the 3-D oracle at 1e-12)."""
    from workloads import box3d as B3
    from paper_2003_12811_gb300 import Solver3D
    N = (n, n, n)
    faces = ("displacement",) * 5 + ("traction",)
    X = B3.block3_coords(N)
    rho, P45 = B3.material3_planes(N)
    hmin = min(np.abs(np.diff(X[0], axis=2)).min(), np.abs(np.diff(X[1], axis=1)).min(),
               np.abs(np.diff(X[2], axis=0)).min())
    dt = 0.2 * hmin / (2.3 * np.sqrt(1.3))
    g1, g2, g3 = B3.ref_grid3(*N)
    u0 = np.array([np.sin(np.pi * g1) * np.sin(np.pi * g2) * np.sin(np.pi * g3 / 2),
                   np.sin(2 * np.pi * g1) * np.sin(np.pi * g2) * np.sin(np.pi * g3 / 2),
                   np.sin(np.pi * g1) * np.sin(2 * np.pi * g2) * np.sin(np.pi * g3 / 2)])
    u0 = u0.astype(np.float32).astype(np.float64)
    out = {}
    runs = {}
    for prec in ("fp64", "fp32"):
        S = Solver3D(X, faces, 6, prec)
        S.sbp3_set_material(0, n, rho, P45)
        S.set_state(u0, u0)
        done = 0
        runs[prec] = {}
        for mark in nsteps:
            S.step(mark - done, dt)
            done = mark
            runs[prec][mark] = S.state()[1]
        S.close()
    for mark in nsteps:
        a, b = runs["fp32"][mark], runs["fp64"][mark]
        out[str(mark)] = float(np.sqrt(np.sum((a - b) ** 2) / np.sum(b ** 2)))
    return {"workload": f"3-D block {n}^3, order 6, bench medium and faces, dt = 0.2 h_min / v_max",
            "fp32_vs_fp64_rel_l2": out}


def convergence_table(Ns=(41, 81, 161, 321), T=0.5, cfl=0.25):
    """Sec. 7.1 convergence study on the GPU: the manufactured solution and material on two blocks
    with an interface, traction and displacement faces, to time T; the l2 error (the scheme's J H
    norm, FP64 on the device) against the exact solution and the observed rate between successive
    grids, for RK4 (FP64, the paper's integrator) and leapfrog (FP64 and FP32)."""
    import torch
    from paper_2003_12811_gb300 import Solver
    from paper_2003_12811_gb300.binding import FIELD_CUR
    kinds = ("robin", "displacement", "robin", "displacement")
    out = {}
    for order in (2, 4, 6):
        rows = {}
        for scheme in ("rk4 fp64", "leapfrog fp64", "leapfrog fp32"):
            errs = []
            for N in Ns:
                P = W.mms_problem(N, order, kinds=kinds, two_blocks=True)
                prec = scheme.split()[1]
                S = Solver(P, prec)
                dt = S.suggest_dt(cfl)
                n = int(math.ceil(T / dt))
                dt = T / n
                if scheme.startswith("rk4"):
                    v0 = [np.stack([-W.MMS_W[L] * np.cos(W.MMS_K[L, 0] * b.X[0] + W.MMS_K[L, 1] * b.X[1])
                                    for L in range(2)]) for b in P.blocks]
                    S.sbp_set_state_rk4([P.exact(b, 0.0) for b in P.blocks], v0, 0.0)
                    S.sbp_step_rk4(n, dt)
                else:
                    S.set_state([P.exact(b, -dt) for b in P.blocks], [P.exact(b, 0.0) for b in P.blocks], 0.0)
                    S.sbp_step(n, dt)
                e2, _ = S.sbp_l2_diff(FIELD_CUR, [P.exact(b, S.sbp_get_time()) for b in P.blocks])
                S.close()
                errs.append(math.sqrt(e2))
            rates = [math.log(errs[k] / errs[k + 1]) / math.log((Ns[k + 1] - 1) / (Ns[k] - 1)) for k in range(len(Ns) - 1)]
            rows[scheme] = {"N": list(Ns), "l2_error": errs, "rate": rates}
        out[f"order {order}"] = rows
        torch.cuda.synchronize()
    return out


def batch_profile_run(nshots=8, side=801, nsteps=6, tick=3):
    """A small served batch for profile captures: nshots shots of side^2 held resident, nsteps
    steps in ticks of `tick` persistent launches."""
    import torch
    from paper_2003_12811_gb300 import Batch, Solver
    B = Batch(6, nshots)
    st = torch.cuda.Stream()
    shots = []
    for i in range(nshots):
        S = Solver(W.shot_problem(side, 70 + i), "fp32")
        B.sbp_batch_add(S, nsteps, S.suggest_dt(0.3))
        shots.append(S)
    for _ in range(nsteps // tick):
        B.sbp_batch_step(tick, st.cuda_stream)
    rem = B.sbp_batch_poll(st.cuda_stream)
    for S in shots:
        S.close()
    B.close()
    return {"batch_profile": {"shots": nshots, "side": side, "steps": nsteps, "remaining": list(rem)[:nshots]}}


def replica_times(times, world):
    """Job times of `world` independent replicas (one process per GPU, no data exchange): each
    entry is the slowest rank's (MAX over ranks).  torch.distributed must be initialised when
    world > 1; the reduction runs on the current CUDA device under NCCL, on the CPU under gloo."""
    if world <= 1:
        return [float(x) for x in times]
    import torch
    import torch.distributed as dist
    dev = "cuda" if dist.get_backend() == "nccl" else "cpu"
    t = torch.tensor([float(x) for x in times], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return [float(x) for x in t.tolist()]


def replica_value(nodes, steps, seconds, world):
    """Whole-job node updates per second: every replica advances `nodes` by `steps` steps."""
    return world * nodes * steps / seconds


def reference_arm(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    K, Wm = max(1, args.steps), max(0, args.warmup)
    # keep the whole run within a few minutes: cap the stepping at ~120 s
    rate, d = run_oracle_steps(None, 2, 0)
    per = d["seconds"] / 2
    K = max(1, min(K, int(120 / max(per, 1e-6))))
    Wm = min(Wm, 3)
    rate, d = run_oracle_steps(None, K, Wm)
    line = {"metric": METRIC, "value": rate, "unit": UNIT, "impl": "reference", "n_gpus": args.gpus,
            "steps": K, "warmup": Wm, "ms_per_step": 1e3 * d["seconds"] / K, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": workload_name("fp64") + " -- oracle on a bounded crop", "nodes": d["nodes"]},
            "cpu_baseline": {"value": rate, "unit": UNIT, "cores": 1, "host_cores": os.cpu_count(), "kind": "oracle",
                             "sample": f"{K} steps on a crop of {d['nodes']} nodes (2 blocks of 401x161)"},
            "e2e": {"value": rate, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=2000)
    ap.add_argument("--warmup", type=int, default=10)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--precision", default="fp32", choices=["fp32", "fp64"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--n1", type=int, default=N1, help="nodes per block along x1 (profiling runs use smaller)")
    ap.add_argument("--n2", type=int, default=N2)
    ap.add_argument("--no-serving", action="store_true")
    ap.add_argument("--no-adjoint", action="store_true")
    ap.add_argument("--no-variants", action="store_true", help="skip the RK4 and wide-stencil measurements")
    ap.add_argument("--accuracy", action="store_true",
                    help="print the FP32-against-FP64 accuracy table of configs 1-3 and exit")
    ap.add_argument("--adjoint-only", action="store_true", help="print the misfit-gradient measurement alone")
    ap.add_argument("--batch-profile", action="store_true",
                    help="run a small served batch (8 shots of 801^2, 6 steps) for a profile capture and exit")
    ap.add_argument("--adjoint-steps", type=int, default=2000, help="leapfrog steps of the misfit-gradient workload")
    ap.add_argument("--op3d-only", action="store_true", help="print the 3-D operator measurement alone")
    ap.add_argument("--accuracy3d", action="store_true",
                    help="print the 3-D FP32-against-FP64 accuracy (96^3, 1000 steps) and exit")
    ap.add_argument("--n3d", type=int, default=256, help="nodes per direction of the 3-D operator workload")
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    if args.impl == "reference":
        return reference_arm(args)

    import torch
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    import __graft_entry__
    if rank == 0 or world == 1:
        __graft_entry__.build()
    if world > 1:
        torch.distributed.barrier()
    from paper_2003_12811_gb300 import Solver

    prec = args.precision
    if args.batch_profile:
        print(json.dumps(batch_profile_run()), flush=True)
        return
    if args.accuracy:
        print(json.dumps({"accuracy": accuracy_table(), "convergence": convergence_table()}), flush=True)
        return 0
    if args.adjoint_only:
        print(json.dumps(adjoint_bench(nsteps=args.adjoint_steps, prec=prec)), flush=True)
        return 0
    if args.accuracy3d:
        print(json.dumps({"accuracy3d": accuracy3d()}), flush=True)
        return 0
    if args.op3d_only:
        print(json.dumps(bench3d(n=args.n3d, prec=prec)), flush=True)
        return 0
    P = W.config3(n1=args.n1, n2=args.n2)
    S = Solver(P, prec)
    dt = S.suggest_dt(0.3)
    zero = [np.zeros((2, b.N2, b.N1)) for b in P.blocks]
    S.set_state(zero, zero, 0.0)
    stream = torch.cuda.current_stream()
    sh = stream.cuda_stream
    nodes = P.n_nodes
    interior_nodes = sum((b.N1 - 18) * (b.N2 - 18) for b in P.blocks)

    # launch tuning for this grid (part of the library; chosen by timing operator applications)
    tune_rows, tune_overlap = S.sbp_autotune()
    # warm-up (the first steps also run the source ramp-up)
    S.sbp_step(args.warmup, dt, sh)
    torch.cuda.synchronize()

    def barrier():
        if world > 1:
            torch.distributed.barrier()

    # ---- timed region (value): K steps, CUDA events on the launch stream
    S.sbp_profile(False)
    barrier()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with ClockSampler(local) as clk:
        e0.record(stream)
        S.sbp_step(args.steps, dt, sh)
        e1.record(stream)
        torch.cuda.synchronize()
    barrier()
    ms = e0.elapsed_time(e1)
    _, launches = S.sbp_profile_read()
    ms = replica_times([ms], world)[0]
    ms_per_step = ms / args.steps
    value = replica_value(nodes, args.steps, ms / 1e3, world)

    # ---- per-kernel timing (roofline of the dominant kernel): same K steps with events per family
    S.sbp_profile(True)
    S.sbp_step(args.steps, dt, sh)
    torch.cuda.synchronize()
    fam_ms, _ = S.sbp_profile_read()
    S.sbp_profile(False)
    interior_ms = fam_ms[0] / args.steps         # the interior launches of a step (both blocks)
    units_per_launch = interior_nodes            # one launch covers the interior of both blocks
    bpn = BYTES_PER_NODE[prec]
    achieved = bpn * interior_nodes / (interior_ms / 1e3) / 1e9
    peak, peak_src = peaks()

    # ---- end to end through the C-ABI with host buffers: upload the state, K steps, read back
    up_h = [np.zeros((2, b.N2, b.N1)) for b in P.blocks]
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    S.sbp_set_state(up_h, up_h, 0.0)
    S.sbp_step(args.steps, dt, sh)
    out = S.sbp_get_field(1)
    torch.cuda.synchronize()
    e2e_s = replica_times([time.perf_counter() - t0], world)[0]
    h2d = sum(2 * u.nbytes for u in up_h)
    d2h = sum(o.nbytes for o in out)
    e2e = {"value": replica_value(nodes, args.steps, e2e_s, world), "unit": UNIT,
           "h2d_bytes_per_step": h2d / args.steps, "d2h_bytes_per_step": d2h / args.steps,
           "note": "one request: host->device upload of (u^{n-1}, u^n) as FP64 host arrays, K steps, "
                   "device->host read of u^n; bytes amortised over the K steps"}

    line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms_per_step, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32" if prec == "fp32" else "f64", "data": "synthetic",
            "config": {"workload": workload_name(prec).replace(f"{N1}x{N2}", f"{args.n1}x{args.n2}"), "nodes": nodes, "order": 6, "dt": dt,
                       "parallelism": "replicas" if world > 1 else "single",
                       "tuning": {"rows_per_cta": tune_rows, "strips_concurrent": bool(tune_overlap)},
                       "l2": f"inputs larger than L2 ({bpn * nodes / 1e9:.2f} GB moved per step vs 129 MB L2)"},
            "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
                         "frac": achieved / peak,
                         "traffic": (TRAFFIC_BYTES_PER_NODE[prec] * units_per_launch
                                     if TRAFFIC_BYTES_PER_NODE[prec] else None),
                         "kernel": "k_interior_march_multi" if prec == "fp32" else "k_interior_edges",
                         "peak_source": peak_src,
                         "bytes_per_node": bpn, "units_per_launch": units_per_launch,
                         "kernel_ms_per_step": interior_ms,
                         "family_ms_per_step": {"interior": fam_ms[0] / args.steps, "boundary": fam_ms[1] / args.steps,
                                                "faces": fam_ms[2] / args.steps, "sources": fam_ms[3] / args.steps}},
            "gpu_launches": int(launches.sum()),
            "clocks": clk.summary(),
            "e2e": e2e}
    S.close()
    if rank == 0 and world == 1 and not args.no_variants:
        line["variants"] = variant_bench(P, prec)
        line["variants"]["op3d"] = bench3d(n=args.n3d, prec=prec)
        if prec == "fp32":
            line["variants"]["fp64"] = fp64_bench(P)
    if rank == 0 and world == 1 and not args.no_serving:
        line["serving"] = serving_bench()
    if rank == 0 and world == 1 and not args.no_adjoint:
        line["adjoint"] = adjoint_bench(nsteps=args.adjoint_steps, prec=prec)
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline()
    if rank == 0:
        print(json.dumps(line), flush=True)
    if world > 1:
        torch.distributed.destroy_process_group()
    return 0


if __name__ == "__main__":
    sys.exit(main())
