#!/usr/bin/env python
"""Benchmark of the ORAS-FGMRES Maxwell solve on GB300.

Metric: solves/s of ORAS-preconditioned FGMRES to a true FP64 relative residual of 1e-8
(one solve = one right-hand side).  Workload (default): the layered head-like medium on a
16^3 x 6 tetrahedral grid, degree-2 Nedelec elements (163,424 complex DOFs), 64 subdomains
with 2 overlap layers, FP32 local factors, FP64 outer FGMRES(100), one z-directed dipole.

One step = the numeric work of one request on a fixed mesh: element matrices, global A,
local impedance matrices A_s, the factorisation of every A_s, and the FGMRES solve with the ORAS
preconditioner.  The per-mesh integer set-up (topology, numbering, partition, overlap)
is done once before timing (the imaging loop reuses its mesh); the end-to-end number
`e2e` includes it, through oras_setup with host buffers, every step.

--impl reference times the CPU oracle (test infrastructure, FP64 NumPy/SciPy) on a bounded
sample of the same workload and extrapolates to solves/s.

Multi-GPU (torchrun): every rank solves its own copy of the request (independent problems,
no data-path collective; weak scaling); the only collectives are the timing barrier and the
max over ranks.
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

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import synth  # noqa: E402

METRIC = "ORAS-FGMRES solves/s to true rel-res 1e-8 (FP32 local factors, FP64 outer FGMRES)"
UNIT = "solves/s"
TB = 64
MEASURED = os.path.join(ROOT, "MEASURED_PEAKS.json")
FALLBACK_HBM, FALLBACK_BF16 = 6800.0, 1900.0
TF32_OVER_BF16 = 1.1 / 2.25   # nominal dense tensor-core ratio (tf32 1.1 PF, bf16 2.25 PF)


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="head16",
                    choices=["head16", "cube8", "head8", "krylov24", "batch32", "batch12", "batch8",
                             "head32r3"],
                    help="head16: the benchmark workload; cube8: 8^3 r=1 plane wave (FP64 factors); "
                         "head8: 8^3 r=2 8 subdomains (for kernel profiles); krylov24: "
                         "24^3 r=2 512 subdomains without overlap (464 MB matrix, small factors, for Krylov "
                         "kernel profiles); batch32: 24^3 r=2 256 subdomains, 32 dipoles solved together; "
                         "batch12: 12^3 r=2 32 subdomains, 32 dipoles; batch8: 8^3 r=2 8 subdomains, 32 "
                         "dipoles (for profiles of the multi-right-hand-side apply); head32r3: 32^3 r=3 4096 subdomains without overlap (3.7 M DOFs)")
    ap.add_argument("--block", type=int, default=0,
                    help="1: solve the workload's right-hand sides as one block (block FGMRES)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--e2e-steps", type=int, default=None)
    ap.add_argument("--serve-count", type=int, default=50,
                    help="requests of the serving stream replayed after the main measurement (0: none)")
    ap.add_argument("--serve-slots", type=int, default=4)
    ap.add_argument("--clocks-dir", default=None,
                    help="where the nvidia-smi clock samples of the timed region are written (default: the temp dir)")
    ap.add_argument("--factor-bits", type=int, default=0, choices=[0, 32, 64],
                    help="local factor precision (0: the workload's; 64: the plain FP64 path)")
    ap.add_argument("--ports", type=int, default=1,
                    help="1: also time the 16-port chamber on the 16^3 mesh (metallic bottom, 16 ports "
                         "transmitting together, 16 x 16 scattering matrix, Sec. 5.1)")
    ap.add_argument("--recycling", type=int, default=1,
                    help="1: also time a sequence of three slowly varying systems on the 24^3 Krylov workload "
                         "with FGMRES(50) and with GCRO-DR(50, 10) recycling its subspace (Sec. 6)")
    ap.add_argument("--fp64-path", type=int, default=1,
                    help="1: also time the plain FP64 single-RHS path against the FP32-factor path on the "
                         "small workloads (head8, cube8)")
    ap.add_argument("--serve-max-iter", type=int, default=150,
                    help="FGMRES iteration cap per served request (requests above it report not converged)")
    return ap.parse_args()


def workload(name):
    if name == "head16":
        return synth.config(1)
    if name == "head8":
        w = synth.small(n=8, r=2, nsub=8, overlap=1, restart=100)
        w.name = "head8_r2_s8_d1_profile"
        return w
    if name == "krylov24":
        w = synth.small(n=24, r=2, nsub=512, overlap=0, restart=50)
        w.name = "head24_r2_s512_d0_krylov_profile"
        return w
    if name == "batch32":
        return synth.config(2)
    if name == "batch8":
        w = synth.small(n=8, r=2, nsub=8, overlap=1, nrhs=32, restart=30)
        w.name = "head8_r2_s8_d1_32dipoles_profile"
        return w
    if name == "batch12":
        w = synth.small(n=12, r=2, nsub=32, overlap=1, nrhs=32, restart=100)
        w.name = "head12_r2_s32_d1_32dipoles_profile"
        return w
    if name == "head32r3":
        return synth.config(4)
    return synth.config(0)


def peaks():
    try:
        with open(MEASURED) as f:
            p = json.load(f)
        return float(p["hbm_gbs"]), float(p["bf16_tflops"]), float(p.get("bf16_tflops_sustained", p["bf16_tflops"])), "measured"
    except Exception:
        return FALLBACK_HBM, FALLBACK_BF16, 1700.0, "fallback"


# ------------------------------------------------------------------ distributed plumbing
def dist_init():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch
        import torch.distributed as dist
        backend = "nccl" if torch.cuda.is_available() else "gloo"
        if torch.cuda.is_available():
            torch.cuda.set_device(local)
        dist.init_process_group(backend)
    return world, rank, local


def barrier(world):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def max_over_ranks(x, world):
    """Max of a float over ranks (timing only)."""
    if world == 1:
        return x
    import torch
    import torch.distributed as dist
    dev = "cuda" if dist.get_backend() == "nccl" else "cpu"
    t = torch.tensor([x], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def aggregate(total_ms_max, solves_per_rank, world):
    """Whole-job throughput: units all ranks processed / max time over ranks."""
    return world * solves_per_rank / (total_ms_max / 1000.0)


# ------------------------------------------------------------------ clocks
class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index, directory=None):
        self.proc = None
        self.path = os.path.join(directory or tempfile.gettempdir(), f"clocks_rank{gpu_index}.csv")
        self.gpu = gpu_index

    def start(self):
        try:
            os.makedirs(os.path.dirname(self.path), exist_ok=True)
            self.f = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                                          "-i", str(self.gpu), "-lms", "200"], stdout=self.f, stderr=subprocess.DEVNULL)
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
            for nm, v in zip(names, parts[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
                "samples": len(sm)}


# ------------------------------------------------------------------ algorithmic work
def work_model(O, h, nsub, k, factor_bytes=8):
    """Algorithmic work of the kernels whose roofline is reported.

    LU trailing update: 8 real flops per complex multiply-add; a step of panel k updates
    (nts-k-1)^2 tiles of TB x TB with TB complex MACs each.
    ORAS apply: one pass reads every stored factor entry once (8 B per complex FP32 entry, 16 B
    per FP64 entry, n_s^2 per subdomain), plus per right-hand side of the pass a 4 B index, a 16 B
    gather and a 16 B scatter per local DOF; k = right-hand sides per pass."""
    upd = 0.0
    ns_sq = 0
    ns_sum = 0
    for s in range(nsub):
        n, _, npad = O.oras_subdomain_size(h, s)
        nts = npad // TB
        upd += sum((nts - q - 1) ** 2 for q in range(nts)) * 8.0 * TB ** 3
        ns_sq += n * n
        ns_sum += n
    apply_bytes = float(factor_bytes) * ns_sq + ns_sum * (4 + 16 * 2) * k
    return upd, apply_bytes


def rhs_groups(k, per_pass):
    """Right-hand sides in each launch when k columns go through a kernel per_pass at a time."""
    return [min(per_pass, k - r0) for r0 in range(0, k, per_pass)]


def apply_group_sizes(k, factor_bits, tensor_cores=False):
    """Live right-hand sides of each apply pass: with the tensor-core apply (FP32 factors, 8 or
    more columns) passes of up to 32 (a pass of 8, 16 or 32 lanes, the unused ones zero);
    otherwise CUDA-core groups of up to 4 (FP32 factors) or 2 (FP64), the last one rounded up to a
    power of two (its unused lanes carry zeros)."""
    if tensor_cores and factor_bits == 32 and k >= 8:
        out, r0 = [], 0
        while r0 < k:
            rem = k - r0
            kt = 32 if rem > 16 else (16 if rem > 8 else 8)
            out.append(min(kt, rem))
            r0 += min(kt, rem)
        return out
    maxkr = 4 if factor_bits == 32 else 2
    out, r0 = [], 0
    while r0 < k:
        kr = 1
        while kr < maxkr and kr < k - r0:
            kr *= 2
        out.append(min(kr, k - r0))
        r0 += min(kr, k - r0)
    return out


def front_group_sizes(k, factor_bits):
    """Live right-hand sides of each pass of the apply with sparse factors: up to 32 (FP32) or 2 (FP64)."""
    out, r0 = [], 0
    while r0 < k:
        rem = k - r0
        out.append(min(rem, 2 if factor_bits == 64 else 32))
        r0 += out[-1]
    return out


def front_apply_bytes(arena_bytes, rows, nr):
    """Algorithmic bytes of one pass of the apply with sparse factors: every stored factor entry once,
    and per local unknown a 4 B index and, for each of the nr right-hand sides, a 16 B gather and a
    16 B scatter."""
    return float(arena_bytes) + rows * (4 + 32 * nr)


TRAFFIC = os.path.join(ROOT, "profiles", "roofline_traffic.json")
# the LU schedule and update kernel the committed counters must have been taken on
UPDATE_VERSION = "tcgen05 update with 128x256 and 128x64 blocks, sub-panel schedule (left-looking sub-panels of 8 steps)"


def measured_traffic(kernel, workload, panel):
    """DRAM bytes per launch from the committed ncu capture of this kernel on this workload and
    panel width, taken on the current kernel version (None when there is none)."""
    try:
        with open(TRAFFIC) as f:
            t = json.load(f)[kernel]
        if (t["workload"] == workload and int(t["lu_panel"]) == int(panel)
                and t.get("source_version") == UPDATE_VERSION):
            return float(t["bytes_per_launch"])
    except Exception:
        pass
    return None


FP64_NOMINAL_TFLOPS = 1.25   # GB300 dense FP64, nominal (no measured figure in the peaks file)


def spmv_bytes(n, nnz, k, fp32_input):
    """Algorithmic bytes of one SpMV launch over k right-hand sides: the CSR matrix once (16 B of
    values + 4 B column per entry, 8 B row pointer per row), the input vector entries (8 B complex
    FP32 or 16 B complex FP64) and the FP64 output entries (16 B) per right-hand side."""
    return 20.0 * nnz + 8.0 * (n + 1) + (8.0 if fp32_input else 16.0) * n * k + 16.0 * n * k


def roofline(timings, upd_flops_per_factor, apply_bytes, factors, hbm, bf16_sus, factor_bits=32, spmv=None):
    """Roofline objects of the kernel classes timed with CUDA events inside the step: the
    dominant class (largest device time) first, then the others that have a work model.  The
    TF32 peak is the measured sustained bf16 rate (the update runs inside a seconds-long step)
    times the nominal tf32/bf16 ratio.  spmv = bytes of the Arnoldi SpMV launches (class "spmv":
    FP32-valued vectors) of the timed steps; the FP64 true-residual SpMV is its own class.  The
    panel updates (class "lu_panel") and the trailing updates run the same kernel under one flop
    model, so their times are summed for the update's roofline and for the choice of the dominant
    class."""
    cls = {c: v for c, v in timings.items() if v[1] > 0}
    if "lu_panel" in cls:
        pm, pn = cls.pop("lu_panel")
        um, un = cls.get("lu_update", (0.0, 0))
        cls["lu_update"] = (um + pm, un + pn)
    dom = max(cls, key=lambda c: cls[c][0])
    out = {}
    if "lu_update" in cls and upd_flops_per_factor is not None:
        ms, _ = cls["lu_update"]
        achieved = upd_flops_per_factor * factors / (ms / 1e3) / 1e12
        if factor_bits == 64:
            out["lu_update"] = {"bound": "alu", "achieved": achieved, "peak": FP64_NOMINAL_TFLOPS, "unit": "TFLOP/s",
                                "frac": achieved / FP64_NOMINAL_TFLOPS, "traffic": None,
                                "kernel": "k_lu_update<double> (FP64 CUDA-core trailing and panel updates)",
                                "peak_note": "nominal GB300 dense FP64 (not measured)"}
        else:
            peak = bf16_sus * TF32_OVER_BF16
            out["lu_update"] = {"bound": "tensor", "achieved": achieved, "peak": peak, "unit": "TFLOP/s",
                                "frac": achieved / peak, "traffic": None,
                                "kernel": "k_lu_update_tc (tcgen05 kind::tf32 complex trailing and panel updates)",
                                "peak_note": "TF32 dense = measured bf16 sustained (of measured) x nominal "
                                             "tf32/bf16 ratio 1.1/2.25"}
    if "apply" in cls:
        ms, launches = cls["apply"]
        achieved = apply_bytes * launches / (ms / 1e3) / 1e9
        out["apply"] = {"bound": "hbm", "achieved": achieved, "peak": hbm, "unit": "GB/s", "frac": achieved / hbm,
                        "traffic": None, "kernel": "k_apply / k_apply4 (ORAS preconditioner, one arena pass per launch, or "
                                                   "per pair of concurrent launches when the largest subdomains "
                                                   "take four CTAs)"}
    if "spmv" in cls and spmv:
        ms, _ = cls["spmv"]
        achieved = spmv / (ms / 1e3) / 1e9
        out["spmv"] = {"bound": "hbm", "achieved": achieved, "peak": hbm, "unit": "GB/s", "frac": achieved / hbm,
                       "traffic": None, "kernel": "k_spmv_df (Arnoldi SpMV of the FP32-valued preconditioned "
                                                 "vectors on the FP32 pipes)"}
    if dom not in out:
        out[dom] = {"bound": "hbm", "achieved": None, "peak": hbm, "unit": "GB/s", "frac": None,
                    "traffic": None, "kernel": dom}
    return dom, out


# ------------------------------------------------------------------ CPU oracle baseline
def oracle_estimate(w, iterations, budget_s=20.0, k=1):
    """Time the oracle (as it stands) on a bounded sample of the workload and extrapolate to
    one solve: full global assembly, then local assembly + dense LU + one local solve on the
    smallest subdomains until ~budget_s of CPU work, scaled by sum n_s^3 (LU) and sum n_s^2
    (applies); Krylov vector work from one SpMV and m/2 MGS steps per iteration."""
    import scipy.linalg as sla
    from oracle import assemble, dd, topology
    xyz, tets = w.mesh()
    eps, mu = w.materials(xyz, tets)
    t0 = time.perf_counter()
    topo = topology.build(tets, len(xyz), w.r)
    A = assemble.global_matrix(topo, xyz, eps, mu, w.k0)
    t_asm = time.perf_counter() - t0
    dec = dd.decompose(topo, xyz, w.nsub, w.overlap)
    ns = np.array([len(d) for d in dec.dofs], dtype=np.float64)
    order = np.argsort(ns)
    t_lu = t_sol = 0.0
    sample = []
    spent = 0.0
    for s in order:
        t1 = time.perf_counter()
        As = dd.local_matrix(topo, xyz, eps, mu, w.k0, dec, int(s))
        lu = sla.lu_factor(As, check_finite=False)
        t2 = time.perf_counter()
        v = np.ones(len(dec.dofs[s]), dtype=np.complex128)
        sla.lu_solve(lu, v, check_finite=False)
        t3 = time.perf_counter()
        t_lu += t2 - t1
        t_sol += t3 - t2
        sample.append(int(s))
        spent += t3 - t1
        if spent > budget_s * 0.6:
            break
    smp = ns[sample]
    lu_total = t_lu * (ns ** 3).sum() / (smp ** 3).sum()
    apply_total = t_sol * (ns ** 2).sum() / (smp ** 2).sum()
    v = np.ones(topo.ndof, dtype=np.complex128)
    t4 = time.perf_counter()
    y = A @ v
    for _ in range(w.restart // 2):
        h_ = np.vdot(v, y)
        y = y - h_ * v
    t_kry = time.perf_counter() - t4
    per_solve = (t_asm + lu_total) / k + iterations * (apply_total + t_kry)  # k right-hand sides share A and LU
    return {"value": 1.0 / per_solve, "unit": UNIT, "cores": os.cpu_count(), "kind": "oracle",
            "sample": (f"global assembly in full; local assembly + LU + 1 solve of the {len(sample)} smallest of "
                       f"{w.nsub} subdomains (n_s {int(smp.min())}-{int(smp.max())}), scaled by sum n_s^3 / "
                       f"sum n_s^2; {iterations} iterations (GPU count) of SpMV + {w.restart // 2} MGS steps"),
            "seconds_per_solve_estimate": per_solve}


# ------------------------------------------------------------------ serving replay
def serving_replay(O, count, slots, device=0, max_iter=60):
    """Replays the first `count` requests of the seeded serving stream (Poisson arrivals at
    5/s; grids 8^3-24^3, degree 1-3, 1/8/32 dipole right-hand sides, perturbation radius and
    permittivity drawn per request) through the serving runtime with `slots` worker slots,
    then again with one slot (sequential), and reports solves/s and latency percentiles.
    Meshes and materials are generated before the clock starts; each request's latency runs
    from its submission (at its arrival time) to its result.  Every request is capped at
    `max_iter` FGMRES iterations: the degree-3 requests with 256 subdomains converge far more
    slowly under the zeroth-order impedance transmission condition, and only right-hand sides
    that reach the tolerance count as solves."""
    reqs = synth.serving_requests()[:count]
    prepared = []
    for w in reqs:
        xyz, tets = w.mesh()
        eps, mu = w.materials(xyz, tets)
        dip = np.concatenate([synth.dipole_ring(w.nrhs), np.tile([0.0, 0.0, 1.0], (w.nrhs, 1))], axis=1)
        prepared.append((w, xyz, tets, eps, mu, dip))

    def replay(nslots):
        srv = O.oras_server_create(max_active=nslots, device=device)
        try:
            t0 = time.perf_counter()
            tickets = []
            for w, xyz, tets, eps, mu, dip in prepared:
                delay = t0 + w.arrival_s - time.perf_counter()
                if delay > 0:
                    time.sleep(delay)
                tickets.append(O.oras_submit(srv, xyz, tets, eps, mu, w.k0, w.r, w.nsub, w.overlap, dipoles=dip,
                                             tol=w.tol, restart=w.restart, factor_bits=w.factor_bits,
                                             max_iter=max_iter))
            outs = []
            errors = {}
            for q, (t, (w, *_rest)) in enumerate(zip(tickets, prepared)):
                x, info, rc = O.oras_wait(srv, t)
                rec = O.oras_ticket_info(srv, t)
                outs.append((w, rc, info, rec))
                if rc not in (O.ORAS_OK, O.ORAS_NOT_CONVERGED):
                    errors[q] = O.oras_server_error(srv, t)
            wall = time.perf_counter() - t0
            st = O.oras_server_stats(srv)
        finally:
            O.oras_server_destroy(srv)
        done = [(w, rc, info, rec) for w, rc, info, rec in outs if rc in (O.ORAS_OK, O.ORAS_NOT_CONVERGED)]
        lat = sorted(rec["done_s"] - rec["submit_s"] for _, _, _, rec in done)
        solves = sum(sum(1 for i in info if i["converged"]) for _, _, info, _ in done)
        worst = max((i["relres"] for _, _, info, _ in done for i in info if i["converged"]), default=None)
        first = min(rec["submit_s"] for _, _, _, rec in outs)
        last = max(rec["done_s"] for _, _, _, rec in outs)

        def pct(q):
            return lat[min(len(lat) - 1, int(round(q * (len(lat) - 1))))] if lat else None
        rejections = [dict(index=q, n=w.n, r=w.r, k=w.nrhs, nsub=w.nsub, footprint_gb=rec["footprint"] / 1e9,
                           budget_gb=st["hbm_budget"] / 1e9, reason="footprint (arena + A + Krylov basis) above the "
                                                                      "whole HBM budget")
                      for q, (w, rc, _, rec) in enumerate(outs) if rc == O.ORAS_ERR_REJECTED]
        failures = [dict(index=q, n=w.n, r=w.r, k=w.nrhs, nsub=w.nsub, rc=int(rc), error=errors.get(q, ""))
                    for q, (w, rc, _, rec) in enumerate(outs)
                    if rc not in (O.ORAS_OK, O.ORAS_NOT_CONVERGED, O.ORAS_ERR_REJECTED)]
        return {"slots": nslots, "solves_per_s": solves / (last - first) if last > first else None,
                "rejections": rejections, "failures": failures,
                "requests_per_s": len(done) / (last - first) if last > first else None,
                "solves": solves, "requests_completed": len(done),
                "rejected": sum(1 for _, rc, _, _ in outs if rc == O.ORAS_ERR_REJECTED),
                "failed": sum(1 for _, rc, _, _ in outs if rc not in (O.ORAS_OK, O.ORAS_NOT_CONVERGED,
                                                                      O.ORAS_ERR_REJECTED)),
                "not_converged_requests": sum(1 for _, rc, _, _ in outs if rc == O.ORAS_NOT_CONVERGED),
                "p50_latency_s": pct(0.5), "p99_latency_s": pct(0.99), "makespan_s": last - first,
                "wall_s": wall, "peak_active": st["peak_active"], "hbm_peak_gb": st["hbm_peak"] / 1e9,
                "hbm_budget_gb": st["hbm_budget"] / 1e9, "worst_true_relres": worst}

    mix = replay(slots)
    seq = replay(1)
    return {"stream": f"first {count} of the seeded serving stream (Poisson 5/s; n 8-24, r 1-3, k 1/8/32 dipoles, "
                      "N_sub = 2^ceil(log2(N/2500)), 1 vertex overlap layer, FGMRES(50), FP32 factors, "
                      f"at most {max_iter} iterations per request)",
            "requests": [dict(n=w.n, r=w.r, k=w.nrhs, nsub=w.nsub, arrival_s=round(w.arrival_s, 3)) for w, *_ in prepared],
            "continuous_batching": mix, "sequential_one_slot": seq}


# ------------------------------------------------------------------ ports and scattering matrix
def chamber_ports(beta):
    """16 ports of 0.5 x 0.5 on the four side faces of the unit cube (a 2 x 2 grid on each face),
    the TE10 mode pointing up (z): a synthetic stand-in for the antenna rings of Sec. 5."""
    out = []
    for z0 in (0.0, 0.5):
        for c0 in (0.0, 0.5):
            out.append(((0.0, c0, z0), (0.0, 0.5, 0.0), (0.0, 0.0, 0.5)))
            out.append(((1.0, c0, z0), (0.0, 0.5, 0.0), (0.0, 0.0, 0.5)))
            out.append(((c0, 0.0, z0), (0.5, 0.0, 0.0), (0.0, 0.0, 0.5)))
            out.append(((c0, 1.0, z0), (0.5, 0.0, 0.0), (0.0, 0.0, 0.5)))
    return [(o, u, v, beta) for o, u, v in out]


def ports_measure(O, dev, stream, steps=1, warmup=1):
    """The 16^3 benchmark mesh and medium with a metallic bottom (Sec. 2 eq. metallicbc) and 16
    ports on the side faces (Silver-Mueller condition, eq. wgi, with the TE10 wavenumber of a
    ceramic-filled guide of width 0.5).  One step = oras_factor + oras_solve of the 16 port loads
    together (each port transmitting, eq. wgj), CUDA events on the handle's stream; then the 16 x 16
    scattering matrix (eq. sij) of the fields, timed as a host call (port selection, copy of the
    fields, device integrals and fixed-order sums), and its reciprocity error ||S - S^T|| / ||S||
    (A = A^T and equal ports make S symmetric)."""
    import torch
    w = workload("head16")
    xyz, tets = w.mesh()
    eps, mu = w.materials(xyz, tets)
    nt = len(tets)
    beta_p = float(np.sqrt(w.k0 ** 2 * 59.0 - (np.pi / 0.5) ** 2))
    kind = np.zeros((nt, 4), dtype=np.uint8)
    for q in range(4):  # the face opposite vertex q lies in z = 0
        others = np.stack([xyz[tets[:, j], 2] for j in range(4) if j != q], axis=1)
        kind[np.all(np.abs(others) < 1e-12, axis=1), q] = O.ORAS_FACE_METALLIC
    beta = np.full((nt, 4), beta_p)
    ps = [O.port(*a) for a in chamber_ports(beta_p)]
    h = O.oras_create(xyz, tets, w.r, w.nsub, w.overlap, beta_face=beta, face_kind=kind, restart=w.restart)
    try:
        O.oras_set_stream(h, stream.cuda_stream)
        eps_d = torch.from_numpy(eps).to(dev)
        mu_d = torch.from_numpy(mu).to(dev)
        O.oras_factor(h, eps_d, mu_d, w.k0, mem=O.ORAS_MEM_DEVICE)
        n = O.oras_ndof(h)
        B = np.stack([O.oras_rhs_port(h, p) for p in ps], axis=1)
        k = B.shape[1]
        Bd = torch.from_numpy(np.ascontiguousarray(B.T)).to(dev)      # column-major N x k
        Xd = torch.empty_like(Bd)
        info = None

        def one():
            O.oras_factor(h, eps_d, mu_d, w.k0, mem=O.ORAS_MEM_DEVICE)
            _, inf, rc = O.oras_solve(h, Bd, w.tol, k=k, mem=O.ORAS_MEM_DEVICE, out=Xd)
            if rc != O.ORAS_OK:
                raise RuntimeError("port solve did not converge")
            return inf
        for _ in range(warmup):
            one()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize(dev)
        e0.record(stream)
        for _ in range(steps):
            info = one()
        e1.record(stream)
        torch.cuda.synchronize(dev)
        ms = e0.elapsed_time(e1) / steps
        X = Xd.cpu().numpy().T
        t0 = time.perf_counter()
        S = O.oras_s_matrix(h, ps, X)
        s_ms = (time.perf_counter() - t0) * 1e3
        return {"workload": "16^3 x 6 tets, r = 2, 64 subdomains, 2 layers, head-like medium; metallic bottom; "
                            "16 ports of 0.5 x 0.5 on the side faces, beta = %.3f" % beta_p,
                "ndof": n, "rhs": k, "solves_per_s": k * 1e3 / ms, "ms_per_step": ms,
                "iterations_max": max(i["iterations"] for i in info),
                "worst_true_relres": max(i["relres"] for i in info),
                "s_matrix_ms": s_ms, "reciprocity_error": O.oras_s_error(S, S.T),
                "s_diag_mean_abs": float(np.abs(np.diag(S)).mean()),
                "s_offdiag_max_abs": float(np.abs(S - np.diag(np.diag(S))).max())}
    finally:
        O.oras_destroy(h)


# ------------------------------------------------------------------ subspace recycling
def recycling_measure(O, dev, stream, n_sys=3, m=50, k=10):
    """A sequence of n_sys systems on the 24^3 Krylov workload (512 subdomains without overlap,
    where FGMRES(50) restarts several times) whose permittivity changes slightly from one system to
    the next (eps_t = eps (1 + 2e-3 t xi), xi ~ U(-1, 1) per tet, as in the imaging loop of Sec. 6).
    Each system: oras_factor with its materials + oras_solve of one dipole, CUDA events on the
    handle's stream.  FGMRES(m) against GCRO-DR(m, k), whose handle carries its deflation subspace
    from one system to the next; products = applications of A M^{-1}."""
    import torch
    w = workload("krylov24")
    xyz, tets = w.mesh()
    eps, mu = w.materials(xyz, tets)
    xi = np.random.default_rng(160504521).uniform(-1.0, 1.0, len(tets))
    mats = [torch.from_numpy(eps * (1.0 + 2e-3 * t * xi)).to(dev) for t in range(n_sys)]
    mu_d = torch.from_numpy(mu).to(dev)
    kind, pt, direction = w.sources()[0]
    out = {"workload": f"{w.n}^3 x 6 tets, r = {w.r}, {w.nsub} subdomains, overlap {w.overlap}; "
                       f"{n_sys} systems, eps_t = eps (1 + 2e-3 t xi)", "restart": m, "recycle_k": k}
    for name, opts in (("fgmres", dict(restart=m)), ("gcrodr", dict(restart=m, recycle=k))):
        h = O.oras_create(xyz, tets, w.r, w.nsub, w.overlap, **opts)
        try:
            O.oras_set_stream(h, stream.cuda_stream)
            per = []
            b = x = None
            for t, e_d in enumerate(mats):
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                torch.cuda.synchronize(dev)
                e0.record(stream)
                O.oras_factor(h, e_d, mu_d, w.k0, mem=O.ORAS_MEM_DEVICE)
                if b is None:
                    n = O.oras_ndof(h)
                    b = torch.empty(n, dtype=torch.complex128, device=dev)
                    O.oras_rhs_dipole(h, pt, direction, mem=O.ORAS_MEM_DEVICE, out=b)
                    x = torch.empty_like(b)
                    e0.record(stream)  # the load is not part of the step
                _, info, rc = O.oras_solve(h, b, w.tol, mem=O.ORAS_MEM_DEVICE, out=x)
                e1.record(stream)
                torch.cuda.synchronize(dev)
                per.append({"products": info[0]["iterations"], "ms": e0.elapsed_time(e1),
                            "true_relres": info[0]["relres"], "converged": rc == O.ORAS_OK})
            out[name] = per
        finally:
            O.oras_destroy(h)
    out["products_total"] = {nm: sum(r["products"] for r in out[nm]) for nm in ("fgmres", "gcrodr")}
    out["ms_total"] = {nm: sum(r["ms"] for r in out[nm]) for nm in ("fgmres", "gcrodr")}
    return out


# ------------------------------------------------------------------ plain FP64 path
def fp64_path(O, dev, stream, steps=2, warmup=1):
    """The plain FP64 single-right-hand-side GPU path (FP64 sparse factors on the FP64 pipe, FP64
    apply; the same FGMRES) against the FP32-factor path, one step = oras_factor + oras_solve of one
    right-hand side on device buffers, CUDA events on the handle's stream, on the 8^3 x 6 meshes."""
    import torch
    out = {}
    for name in ("head8", "cube8"):
        w = workload(name)
        xyz, tets = w.mesh()
        eps, mu = w.materials(xyz, tets)
        eps_d = torch.from_numpy(eps).to(dev)
        mu_d = torch.from_numpy(mu).to(dev)
        row = {"ndof": None}
        for bits in (32, 64):
            h = O.oras_create(xyz, tets, w.r, w.nsub, w.overlap, factor_bits=bits, restart=w.restart)
            try:
                O.oras_set_stream(h, stream.cuda_stream)
                O.oras_factor(h, eps_d, mu_d, w.k0, mem=O.ORAS_MEM_DEVICE)
                n = O.oras_ndof(h)
                kind, pt, direction = w.sources()[0]
                b = torch.empty(n, dtype=torch.complex128, device=dev)
                if kind == "plane":
                    O.oras_rhs_plane_wave(h, pt, direction.astype(np.complex128), mem=O.ORAS_MEM_DEVICE, out=b)
                else:
                    O.oras_rhs_dipole(h, pt, direction, mem=O.ORAS_MEM_DEVICE, out=b)
                x = torch.empty_like(b)
                info = None

                def one():
                    O.oras_factor(h, eps_d, mu_d, w.k0, mem=O.ORAS_MEM_DEVICE)
                    _, inf, rc = O.oras_solve(h, b, w.tol, mem=O.ORAS_MEM_DEVICE, out=x)
                    if rc != O.ORAS_OK:
                        raise RuntimeError(f"{name} factor_bits={bits}: solve did not converge")
                    return inf
                for _ in range(warmup):
                    one()
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                torch.cuda.synchronize(dev)
                e0.record(stream)
                for _ in range(steps):
                    info = one()
                e1.record(stream)
                torch.cuda.synchronize(dev)
                ms = e0.elapsed_time(e1) / steps
                row["ndof"] = n
                row[f"factors{bits}"] = {"solves_per_s": 1e3 / ms, "ms_per_solve": ms,
                                         "iterations": info[0]["iterations"], "true_relres": info[0]["relres"]}
            finally:
                O.oras_destroy(h)
        row["speedup_fp32_factors_over_fp64"] = row["factors32"]["solves_per_s"] / row["factors64"]["solves_per_s"]
        out[w.name] = row
    out["note"] = ("one step = oras_factor + oras_solve of one right-hand side to true rel-res 1e-8; factors64 = "
                   "the plain FP64 single-RHS GPU path, factors32 = this library's FP32-factor path")
    return out


# ------------------------------------------------------------------ our arm
def run_ours(args, world, rank, local):
    import torch
    from paper_1605_04521_gb300 import build
    build.build()
    from paper_1605_04521_gb300 import oras as O
    w = workload(args.workload)
    if args.factor_bits:
        w.factor_bits = args.factor_bits
        w.name += f"_factors{args.factor_bits}"
    hbm, bf16, bf16_sus, src = peaks()
    xyz, tets = w.mesh()
    eps, mu = w.materials(xyz, tets)
    dev = torch.device("cuda", local)
    stream = torch.cuda.current_stream(dev)
    t_mesh0 = time.perf_counter()
    opts = dict(restart=w.restart, block=args.block)
    if args.block:
        w.name += "_block_fgmres"
    h = O.oras_create(xyz, tets, w.r, w.nsub, w.overlap, factor_bits=w.factor_bits, **opts)
    t_mesh = time.perf_counter() - t_mesh0
    O.oras_set_stream(h, stream.cuda_stream)
    eps_d = torch.from_numpy(eps).to(dev)
    mu_d = torch.from_numpy(mu).to(dev)
    O.oras_factor(h, eps_d, mu_d, w.k0, mem=O.ORAS_MEM_DEVICE)
    n = O.oras_ndof(h)
    srcs = w.sources()
    krhs = len(srcs)
    b_d = torch.empty(krhs, n, dtype=torch.complex128, device=dev)  # N x k column-major
    for j, (kind, pt, direction) in enumerate(srcs):
        if kind == "plane":
            O.oras_rhs_plane_wave(h, pt, direction.astype(np.complex128), mem=O.ORAS_MEM_DEVICE, out=b_d[j])
        else:
            O.oras_rhs_dipole(h, pt, direction, mem=O.ORAS_MEM_DEVICE, out=b_d[j])
    x_d = torch.empty_like(b_d)
    flush = torch.empty(512 * 1024 * 1024, dtype=torch.uint8, device=dev)

    def step():
        O.oras_factor(h, eps_d, mu_d, w.k0, mem=O.ORAS_MEM_DEVICE)
        _, info, rc = O.oras_solve(h, b_d, w.tol, k=krhs, mem=O.ORAS_MEM_DEVICE, out=x_d)
        if rc != O.ORAS_OK or not all(i["converged"] for i in info):
            raise RuntimeError(f"solve did not converge: {info}")
        return info

    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize(dev)
    O.oras_set_timing(h, 1)
    O.oras_reset_timings(h)
    launches0 = O.oras_launch_count()
    clocks = ClockSampler(local, args.clocks_dir)
    clocks.start()
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    barrier(world)
    torch.cuda.synchronize(dev)
    wall0 = time.perf_counter()
    infos = []
    for q in range(args.steps):
        flush.zero_()                      # L2 flush between timed steps (outside the events)
        ev[q][0].record(stream)
        infos.append(step())
        ev[q][1].record(stream)
    torch.cuda.synchronize(dev)
    barrier(world)
    wall = time.perf_counter() - wall0
    clk = clocks.stop()
    launches = O.oras_launch_count() - launches0
    timings = O.oras_timings(h)
    O.oras_set_timing(h, 0)
    step_ms = [a.elapsed_time(b) for a, b in ev]
    total_ms = max_over_ranks(sum(step_ms), world)
    value = aggregate(total_ms, args.steps * krhs, world)
    # true residual of the last field, FP64, on the host with the library's own A (sanity)
    x_last = x_d.cpu().numpy()
    iters = max(i["iterations"] for i in infos[-1])
    groups = front_group_sizes(krhs, w.factor_bits)
    arena = O.oras_arena_bytes(h)
    rows = sum(O.oras_subdomain_size(h, s)[0] for s in range(w.nsub))
    # bytes of one apply pass, averaged over the passes of a step (groups of right-hand sides)
    apply_bytes = sum(front_apply_bytes(arena, rows, g) for g in groups) / len(groups)
    nnz = O.oras_nnz(h)
    spmv_total = 0.0
    for info in infos:
        it = max(i["iterations"] for i in info)
        cyc = max(i["restarts"] for i in info)
        if w.factor_bits == 32:   # the Arnoldi SpMV (class "spmv"); true residuals are class "spmv64"
            spmv_total += it * sum(spmv_bytes(n, nnz, g, True) for g in rhs_groups(krhs, 8))
    dom, roofs = roofline(timings, None, apply_bytes, args.steps, hbm, bf16_sus, w.factor_bits, spmv_total)
    if "apply" in roofs:
        roofs["apply"]["kernel"] = ("k_fr_fwd / k_fr_bwd (ORAS preconditioner with sparse local factors, one launch per tree "
                                    "level and direction; the bytes count each stored entry once, the two "
                                    "directions read the border entries twice)")
    roof = roofs[dom]
    O.oras_destroy(h)
    # ---------------- end to end through the public API with host buffers
    e2e_steps = args.e2e_steps if args.e2e_steps is not None else max(1, args.steps)
    b_host = torch.from_numpy(b_d.cpu().numpy().T.copy()).pin_memory().numpy()   # (N, k)
    x_host = torch.empty(n, krhs, dtype=torch.complex128).pin_memory().numpy()
    h2d = xyz.nbytes + tets.nbytes + eps.nbytes + mu.nbytes + b_host.nbytes
    d2h = x_host.nbytes
    barrier(world)
    torch.cuda.synchronize(dev)
    e0 = time.perf_counter()
    for _ in range(e2e_steps):
        he = O.oras_setup(xyz, tets, eps, mu, w.k0, w.r, w.nsub, w.overlap, factor_bits=w.factor_bits, **opts)
        xe, info_e, rc = O.oras_solve(he, b_host, w.tol, k=krhs)
        x_host[:] = np.asarray(xe).reshape(n, krhs)
        O.oras_destroy(he)
        if rc != O.ORAS_OK:
            raise RuntimeError("e2e solve did not converge")
    torch.cuda.synchronize(dev)
    e2e_s = max_over_ranks(time.perf_counter() - e0, world)
    e2e_val = world * e2e_steps * krhs / e2e_s
    port_res = None
    if rank == 0 and args.ports:
        try:
            port_res = ports_measure(O, dev, stream)
        except Exception as e:  # noqa: BLE001
            port_res = {"error": f"{type(e).__name__}: {e}"}
    recyc = None
    if rank == 0 and args.recycling:
        try:
            recyc = recycling_measure(O, dev, stream)
        except Exception as e:  # noqa: BLE001
            recyc = {"error": f"{type(e).__name__}: {e}"}
    fp64 = None
    if rank == 0 and args.fp64_path:
        try:
            fp64 = fp64_path(O, dev, stream)
        except Exception as e:  # noqa: BLE001
            fp64 = {"error": f"{type(e).__name__}: {e}"}
    serving = None
    if rank == 0 and args.serve_count > 0:
        # the serving replay is reported beside the main measurement: a failure there is recorded
        # in the line instead of losing the measurement taken above
        try:
            serving = serving_replay(O, args.serve_count, args.serve_slots, device=local,
                                     max_iter=args.serve_max_iter)
        except Exception as e:  # noqa: BLE001
            serving = {"error": f"{type(e).__name__}: {e}"}
    out = None
    if rank == 0:
        cpu = None
        if world == 1 and not args.no_cpu_baseline:
            cpu = oracle_estimate(w, iters, k=krhs)
        out = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": total_ms / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None,
            "dtype": ("c128 factors / c128 Krylov" if w.factor_bits == 64 else "c64 factors / c128 Krylov"), "data": "synthetic",
            "config": {"workload": w.name, "mesh": f"{w.n}^3 x 6 tets (Kuhn)", "degree": w.r, "ndof": n,
                       "nsub": w.nsub, "overlap_layers": w.overlap, "restart": w.restart, "tol": w.tol,
                       "rhs_per_step": krhs, "factor_arena_bytes": arena,
                       "l2": "512 MiB buffer written between timed steps; the step itself streams the "
                             f"{arena / 1e9:.1f} GB of factors",
                       "step": "oras_factor (element matrices, A, A_s, local factorisations) + oras_solve, device buffers",
                       "mesh_setup_s_untimed": t_mesh, "parallelism": f"replicas x{world}",
                       "factors": "sparse block L D L^T"},
            "iterations": iters, "true_relres": max(i["relres"] for i in infos[-1]),
            "phase_ms_per_step": {c: v[0] / args.steps for c, v in timings.items() if v[1] > 0},
            "roofline": roof,
            "roofline_kernels": roofs,
            "cpu_baseline": cpu,
            "e2e": {"value": e2e_val, "unit": UNIT, "h2d_bytes_per_step": int(h2d), "d2h_bytes_per_step": int(d2h),
                    "path": "oras_setup (host mesh + materials) + oras_solve (host rhs -> host x) + oras_destroy"},
            "gpu_launches": int(launches),
            "fp64_path": fp64,
            "ports": port_res,
            "recycling": recyc,
            "serving": serving,
            "clocks": clk,
            "peaks": {"hbm_gbs": hbm, "bf16_tflops": bf16, "bf16_tflops_sustained": bf16_sus, "source": src},
            "wall_s_timed": wall,
        }
        print(json.dumps(out))
    return out


# ------------------------------------------------------------------ reference arm: the oracle
REF_ITERATIONS = {"head16": 17, "head8": 10, "cube8": 11}


def run_reference(args, world, rank):
    if rank != 0:
        return None
    w = workload(args.workload)
    # FGMRES iterations to 1e-8 on these workloads (the GPU path and the oracle agree on them)
    iterations = int(os.environ.get("ORAS_REF_ITERATIONS", str(REF_ITERATIONS.get(args.workload, 40))))
    for _ in range(args.warmup):
        oracle_estimate(w, iterations, budget_s=3.0)
    vals = []
    t0 = time.perf_counter()
    for _ in range(args.steps):
        vals.append(oracle_estimate(w, iterations, budget_s=8.0))
    wall = time.perf_counter() - t0
    v = statistics.median([x["value"] for x in vals])
    cpu = dict(vals[-1])
    cpu["value"] = v
    out = {"impl": "reference", "metric": METRIC, "value": v, "unit": UNIT, "n_gpus": world,
           "steps": args.steps, "warmup": args.warmup, "ms_per_step": wall * 1e3 / args.steps,
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "c128",
           "data": "synthetic", "config": {"workload": w.name, "ndof_closed_form": None},
           "cpu_baseline": cpu,
           "e2e": {"value": v, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
           "note": ("reference arm = the CPU oracle (FP64 NumPy/SciPy) timed on the host cores on a bounded "
                    f"sample and extrapolated; {iterations} FGMRES iterations, the count the solve takes on this workload")}
    print(json.dumps(out))
    return out


def main():
    args = parse()
    world, rank, local = dist_init()
    try:
        if args.impl == "reference":
            run_reference(args, world, rank)
        else:
            run_ours(args, world, rank, local)
    finally:
        if world > 1:
            import torch.distributed as dist
            dist.destroy_process_group()


if __name__ == "__main__":
    main()
