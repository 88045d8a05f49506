#!/usr/bin/env python
"""Throughput of the plane-wave Hamiltonian hot path on one GB300 (or N replicas).

One step = one pass of the hot path over a block of bands of one k-point:
    H C (scatter -> inverse 3-D FFT -> x V -> forward FFT -> gather, kinetic,
    nonlocal P D P^dag C), the density n(r) = sum_b f_b |psi_b|^2, and the
    subspace matrices C^dag H C and C^dag O C,
on the synthetic 128^3 workload: cubic cell L = 20 bohr, E_cut = 30 Ha
(62 759 plane waves at k = (0.1, 0.2, 0.3)), 64 Gaussian atoms, 256
projectors, 256 bands.  Metric: band-applies per second (bands x steps / s).

    python bench.py [--gpus N] [--steps K] [--warmup W] [--prec fp32|fp64|...]
    python bench.py --impl reference     # the FP64 CPU oracle on the host cores

Under torchrun each rank runs its own replica of the workload (independent
problems, no data-path collective); the value is the sum over ranks divided by
the slowest rank's time.
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
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "Hψ band-applies/s & time to |ΔE|<1e-6 Ha: mixed+learned vs FP64, 1 GB300"
UNIT = "band-applies/s"
FP64_NOMINAL_TFLOPS = 1.25


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=60)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    # bf16x3: BF16 hi/lo operand split on the tensor cores; on this workload it
    # is both faster and closer to FP64 than tf32x3 (C^dag H C 1.8e-5 vs 3.7e-5
    # relative; eigenvalues 1.0e-4 vs 2.1e-4 Ha): the FP32 accumulation in
    # tensor memory, not the split, dominates the error of either
    ap.add_argument("--prec", default="bf16x3", choices=["fp64", "fp32", "tf32x3", "bf16x3"])
    ap.add_argument("--no-cg", action="store_true")
    ap.add_argument("--no-batch", action="store_true")
    ap.add_argument("--no-slab", action="store_true", help="skip the 1024-band, 4 k-point slab section")
    ap.add_argument("--no-scf", action="store_true", help="skip the SCF section (Hartree, LDA, Pulay, SCF loop)")
    ap.add_argument("--nbands", type=int, default=0, help="bands of the block (0 = the workload's)")
    ap.add_argument("--workload", default="large")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-fp64", action="store_true")
    ap.add_argument("--cpu-seconds", type=float, default=15.0)
    ap.add_argument("--no-autotune", action="store_true",
                    help="library defaults instead of the autotuned chunk budget and split-K counts (profiling)")
    return ap.parse_args()


# ---------------------------------------------------------------------------
# distributed plumbing
# ---------------------------------------------------------------------------
def dist_setup():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    pg = None
    if world > 1:
        import torch
        import torch.distributed as dist
        backend = "nccl" if torch.cuda.is_available() else "gloo"
        if torch.cuda.is_available():
            torch.cuda.set_device(local)
        dist.init_process_group(backend=backend)
        pg = dist
    return world, rank, local, pg


def barrier(pg):
    if pg is not None:
        pg.barrier()


def _reduce(pg, x: float, op: str) -> float:
    import torch
    t = torch.tensor([x], dtype=torch.float64, device="cuda" if torch.cuda.is_available() else "cpu")
    pg.all_reduce(t, op=getattr(pg.ReduceOp, op))
    return float(t.item())


def max_over_ranks(pg, x: float) -> float:
    return x if pg is None else _reduce(pg, x, "MAX")


def job_totals(pg, local_time: float, local_units: float) -> tuple[float, float]:
    """Whole-job totals over the replicas: the slowest rank's time and the
    units all ranks processed (their sum)."""
    if pg is None:
        return local_time, local_units
    return _reduce(pg, local_time, "MAX"), _reduce(pg, float(local_units), "SUM")


# ---------------------------------------------------------------------------
# clocks during the timed region
# ---------------------------------------------------------------------------
class Clocks:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, local_rank: int):
        vis = os.environ.get("CUDA_VISIBLE_DEVICES")
        self.idx = int(vis.split(",")[local_rank]) if vis else local_rank
        self.proc = None
        self.path = None

    def start(self):
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.idx), f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "100", "-f", self.path],
                                         stdout=subprocess.DEVNULL, stderr=subprocess.DEVNULL)
        except (OSError, ValueError):
            self.proc = None
        time.sleep(0.3)

    def stop(self) -> dict:
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        time.sleep(0.15)
        self.proc.terminate()
        self.proc.wait()
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        with open(self.path) as f:
            for line in f:
                p = [x.strip() for x in line.split(",")]
                if len(p) < 9:
                    continue
                try:
                    sm.append(float(p[1]))
                    smax.append(float(p[2]))
                except ValueError:
                    continue
                for n, v in zip(names, p[5:9]):
                    if v.lower() == "active":
                        reasons.add(n)
        os.unlink(self.path)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(smax) if smax else None,
                "reasons": sorted(reasons), "samples": len(sm)}


# ---------------------------------------------------------------------------
# the workload
# ---------------------------------------------------------------------------
class Problem:
    """Device-resident inputs and outputs of one step, built through the C ABI."""

    def __init__(self, wname: str, prec: str, device, nbands: int = 0, autotune: bool = True):
        import torch

        from paper_1708_03621_gb300 import jdft
        from synth import WORKLOADS, random_coefficients, workload_atoms
        self.jdft = jdft
        self.prec = prec
        w = WORKLOADS[wname]
        self.w = w
        self.dev = device
        atoms = workload_atoms(w)
        self.basis = jdft.Basis(w.R, w.S, w.ecut, w.kfrac, w.weights())
        self.N = int(np.prod(w.S))
        self.npw = self.basis.npw(0)
        self.info = self.basis.info(0)
        V = torch.empty(self.N, dtype=torch.float64, device=device)
        jdft.jdft_gaussian_potential(self.basis, atoms, V)
        jdft.jdft_set_potential(self.basis, V)
        self.nproj = 4 * w.natoms
        P = torch.empty((self.nproj, self.npw), dtype=torch.complex128, device=device)
        jdft.jdft_gaussian_projectors(self.basis, 0, atoms, P)
        D = torch.tensor(np.diag(np.tile([0.5, -0.3, -0.3, -0.3], w.natoms)), device=device)
        jdft.jdft_set_projectors(self.basis, 0, P, D)
        del P, V
        # kinetic energies for the damping of the random block: from the library's own sphere
        iG = self.basis.gvectors(0).astype(np.float64)
        self.nrows = int(iG[:, 0].max() - iG[:, 0].min() + 1)   # i0 rows the sphere touches
        q = (iG + np.asarray(w.kfrac[0])) @ (2 * np.pi * np.linalg.inv(w.R).T).T
        Y = random_coefficients(np.sum(q * q, 1), nbands or w.nbands, w.seed_coeffs)
        Y /= np.sqrt(self.info["omega"] * np.sum(np.abs(Y) ** 2, axis=1, keepdims=True))
        ct = torch.complex128 if prec == "fp64" else torch.complex64
        self.C_host = torch.tensor(Y.astype(np.complex128 if prec == "fp64" else np.complex64)).pin_memory()
        self.C = self.C_host.to(device)
        self.HC = torch.empty_like(self.C)
        self.nb = Y.shape[0]
        self.f = torch.full((self.nb,), 2.0, dtype=torch.float64, device=device)
        self.n = torch.zeros(self.N, dtype=torch.float64, device=device)
        self.CHC = torch.empty((self.nb, self.nb), dtype=torch.complex128, device=device)
        self.COC = torch.empty_like(self.CHC)
        self.ctype = ct
        # the project's autotuner picks the chain's chunk budget and the GEMM
        # split-K schedules for this block before anything is timed
        self.tune = (jdft.jdft_autotune(self.basis, 0, self.C, self.HC, prec)
                     if prec != "fp64" and autotune else None)
        # device status word of the asynchronous orthonormalisation, checked after each timed loop
        self.status = torch.zeros(1, dtype=torch.int32, device=device)

    def buffers(self):
        """A second set of the step's device buffers (the double-buffered end-to-end loop)."""
        import torch
        return {"C": torch.empty_like(self.C), "HC": torch.empty_like(self.HC), "n": torch.empty_like(self.n),
                "CHC": torch.empty_like(self.CHC), "COC": torch.empty_like(self.COC)}

    def own_buffers(self):
        return {"C": self.C, "HC": self.HC, "n": self.n, "CHC": self.CHC, "COC": self.COC}

    def step(self, stream=None, b=None):
        """Rows a1-a9 in one library call (on buffer set b, default the
        problem's own): C^dag O C of the input block, its FP64 Cholesky
        factorisation on the basis's side stream while H C and the density
        run, C^dag H C, then the orthonormalisation C <- C L^-dag.  No host
        wait per step: a failure lands in self.status (see check_status)."""
        j = self.jdft
        b = b or self.own_buffers()
        b["n"].zero_()
        j.jdft_hamiltonian_step(self.basis, 0, b["C"], b["HC"], self.f, b["n"], b["CHC"], b["COC"], self.status,
                                self.prec, stream)

    def check_status(self):
        """Raise if any orthonormalisation since set-up met linearly dependent bands."""
        import torch
        torch.cuda.synchronize()
        if int(self.status.item()) != 0:
            raise RuntimeError(f"orthonormalisation failed (status {int(self.status.item())})")

    def io_bytes(self):
        e = self.C.element_size()
        return (self.nb * self.npw * e,
                self.nb * self.npw * e + 2 * self.nb * self.nb * 16 + self.N * 8)


def kernel_work(p: Problem, name: str, launches: int, nb: int) -> tuple[float, float]:
    """Algorithmic (flops, bytes) of ONE launch of kernel `name`, averaged over the step.

    FFT flops use the nominal 5 n log2 n per complex length-n transform; bytes
    are the minimum DRAM traffic (inputs read once, outputs written once).
    """
    S0, S1, S2 = p.w.S
    ncols = p.info["ncols"]
    nrows = p.nrows
    e = p.C.element_size()
    per_launch_bands = nb / max(1, launches)
    l2 = math.log2
    if name in ("tc_zgemm_cn", "tc_zgemm_nn"):
        return kernel_work(p, name[3:], launches, nb)
    if name == "tcx_cn":
        # the same C^dag B products, from split operands (BF16 hi/lo planes: 8 bytes per complex value)
        return kernel_work(p, "zgemm_cn", launches, nb)
    if name == "tcx_nn":
        return kernel_work(p, "zgemm_nn", launches, nb)
    if name == "tcx_reduce":
        # the split-K partial tiles of one tcx_cn product (128 x 256 FP32 complex per block, one block
        # per (tile, split): the autotuned split count) read once, the nb x nb FP64 output read and written
        tune = getattr(p, "tune", None) or {}
        splits = tune.get("splits_subspace") or 1
        tiles = -(-p.nb // 128)
        return 0.0, splits * tiles * 128 * 256 * 8.0 + 2 * p.nb * p.nb * 16.0
    if name == "split_planes":
        # per step: C, H C (nb rows of npw), C's transpose (npw rows of nb), (D P^dag C)'s and W's
        # transposes (nb rows of nproj, nb); FP32 complex read, four BF16 planes written (8 + 8
        # bytes per value), averaged over the launches
        vals = 3.0 * p.nb * p.npw + p.nb * p.nproj + p.nb * p.nb
        return 0.0, 16.0 * vals / max(1, launches)
    if name in ("plane_apply", "plane_apply_fast", "plane_apply_pair", "plane_apply_density_fast",
                "plane_apply_density_pair"):
        # the fused kernels do the same transforms; their density adds the n(r) update
        fl = 5 * S2 * (2 * nrows * S1 * l2(S1) + 2 * S1 * S0 * l2(S0))
        by = 2 * S2 * ncols * e
        extra = p.N * 16 if "density" in name else 0
        return fl * per_launch_bands, by * per_launch_bands + p.N * (8 if e == 16 else 4) + extra
    if name in ("plane_density", "plane_density_fast"):
        fl = 5 * S2 * (nrows * S1 * l2(S1) + S1 * S0 * l2(S0))
        return fl * per_launch_bands, S2 * ncols * e * per_launch_bands + p.N * 8
    if name in ("zpass_inverse", "zpass_forward"):
        fl = 5 * ncols * S2 * l2(S2)
        by = (p.npw + S2 * ncols) * e + (p.npw * e if name == "zpass_forward" else 0)
        return fl * per_launch_bands, by * per_launch_bands
    if name in ("line_z_inverse", "line_z_forward"):
        return kernel_work(p, "zpass_" + name[7:], launches, nb)
    if name in ("line_rows_inverse", "line_rows_forward"):
        # sphere columns and rows, one read and the other written
        fl = 5 * nrows * S2 * S1 * l2(S1)
        return fl * per_launch_bands, (S2 * ncols + nrows * S1 * S2) * e * per_launch_bands
    if name == "line_columns":
        fl = 2 * 5 * S1 * S2 * S0 * l2(S0)
        return fl * per_launch_bands, 2 * nrows * S1 * S2 * e * per_launch_bands + p.N * (8 if e == 16 else 4)
    if name == "line_density":
        fl = 5 * S1 * S2 * S0 * l2(S0)
        return fl * per_launch_bands, nrows * S1 * S2 * e * per_launch_bands + p.N * 16
    if name in ("sl_mma", "sl_slice"):
        # the FP64 step's five products (those of zgemm_cn and zgemm_nn above) on slices of 36 bytes a complex
        # value; C^dag C needs one operand's.  Averages over the launches, each of both operands for sl_slice.
        cn, nn = [(p.nproj, p.nb), (p.nb, p.nb), (p.nb, 0)], [p.nproj, p.nb]
        vals = sum((M + N) * p.npw for M, N in cn) + sum((p.npw + p.nb) * K for K in nn)
        if name == "sl_slice":
            return 0.0, (16.0 + 36.0) * vals / max(1, launches)
        fl = 3 * kernel_work(p, "zgemm_cn", 3, nb)[0] + 2 * kernel_work(p, "zgemm_nn", 2, nb)[0]
        return fl / max(1, launches), 36.0 * vals / max(1, launches)
    if name == "zgemm_cn":
        # per step: P^dag C (nproj x nb), C^dag HC and C^dag C (nb x nb), over npw (the orthonormaliser
        # reuses the subspace step's C^dag O C)
        per_step = [(p.nproj, p.nb), (p.nb, p.nb), (p.nb, p.nb)]
        fl = sum(8.0 * M * N * p.npw for M, N in per_step) / len(per_step)
        by = sum((M + N) * p.npw * e for M, N in per_step) / len(per_step)
        return fl, by
    if name == "zgemm_nn":
        # per step: HC += P (D P^dag C) (K = nproj) and the orthonormaliser's C L^{-dag} (K = nb)
        fl = 8.0 * p.npw * p.nb * (p.nproj + p.nb) / 2
        by = ((2.0 * p.nb + p.nproj) + (2.0 * p.nb + p.nb)) * p.npw * e / 2
        return fl, by
    return 0.0, 0.0


def roofline_of(k: dict, prec: str, peaks: dict, fp32: dict) -> dict:
    """The roofline that bounds one kernel, with its peak and where that comes from.

    FFT and CUDA-core GEMM kernels: the FP32 arithmetic peak measured on this
    GPU by jdft_measure_fp32_peak (the larger of the scalar and the packed FMA
    chains), or the nominal FP64 rate for FP64 blocks; tensor-core GEMMs: the
    measured BF16 burst (BF16x3 pieces), or TF32 = that x (1.1 / 2.25), the
    nominal TF32/BF16 ratio, against algorithmic 8MNK flops (the 3-term split
    issues 3x that, so 1/3 is that kernel's ceiling; the FP64 products from
    slices 45x); everything else: HBM copy bandwidth.  FP64 transforms run in
    64-bit integers, so their nominal flops can pass the FP64 pipe's rate.
    """
    name = k["name"]
    hbm = peaks.get("hbm_gbs", 6800.0)
    src_hbm = "MEASURED_PEAKS.json hbm_gbs (of measured)" if "hbm_gbs" in peaks else "fallback 6800 GB/s"
    if name.startswith("tc_zgemm") or name in ("tcx_cn", "tcx_nn"):
        bf16 = peaks.get("bf16_tflops", 1900.0)
        src = "of measured" if "bf16_tflops" in peaks else "of fallback"
        if prec == "bf16x3":
            peak, how = bf16, f"measured bf16 burst ({src})"
        else:
            peak, how = bf16 * 1.1 / 2.25, f"measured bf16 burst x nominal tf32/bf16 ratio 1.1/2.25 ({src})"
        return {"bound": "tensor", "achieved": k["achieved_tflops"], "peak": round(peak, 1), "unit": "TFLOP/s",
                "frac": round((k["achieved_tflops"] or 0) / peak, 4), "split_passes": 3, "peak_source": how}
    if name == "sl_mma":
        bf16 = peaks.get("bf16_tflops", 1900.0)
        return {"bound": "tensor", "achieved": k["achieved_tflops"], "peak": round(bf16, 1), "unit": "TFLOP/s",
                "frac": round((k["achieved_tflops"] or 0) / bf16, 4), "split_passes": 45,
                "peak_source": "measured bf16 burst (%s)" % ("of measured" if "bf16_tflops" in peaks else "of fallback")}
    if name.startswith(("plane_", "zgemm", "zpass", "line_")):
        if prec == "fp64":
            alu, how = FP64_NOMINAL_TFLOPS, "FP64 nominal 1.25 TFLOP/s"
        else:
            alu = max(fp32["ffma_tflops"], fp32["ffma2_tflops"])
            how = (f"measured FP32 peak (of measured): FMA chains on all {fp32['sms']} SMs, scalar "
                   f"{fp32['ffma_tflops']:.1f} / packed {fp32['ffma2_tflops']:.1f} TFLOP/s, the larger")
        r_alu = (k["achieved_tflops"] or 0) / alu
        r_hbm = (k["achieved_gbs"] or 0) / hbm
        if r_alu >= r_hbm:
            return {"bound": "alu", "achieved": k["achieved_tflops"], "peak": round(alu, 2), "unit": "TFLOP/s",
                    "frac": round(r_alu, 4), "peak_source": how}
    return {"bound": "hbm", "achieved": k["achieved_gbs"], "peak": hbm, "unit": "GB/s",
            "frac": round((k["achieved_gbs"] or 0) / hbm, 4), "peak_source": src_hbm}


# DRAM bytes (read + write) per band of a kernel, from one ncu capture
# (dram__bytes_read.sum + dram__bytes_write.sum of one 64-band launch on the
# 128^3 workload, --nbands 64), scaled by the bands a launch processes.  ncu
# replays with cold caches, so this bounds the warm traffic from above.  Each
# entry holds the SHA-256 of the kernel's source files at capture time; when
# the sources differ, the figure no longer describes the kernel and the bench
# reports null.
TRAFFIC_SOURCES = {"plane_apply_density_pair": ["csrc/plane_pair.cu", "csrc/fft_pair.cuh", "csrc/fft_reg.cuh",
                                                "csrc/chain.cuh", "csrc/common.cuh", "csrc/tc_ptx.cuh"]}
TRAFFIC_PER_BAND = {
    # 150 366 464 + 85 970 944 bytes over 64 bands (ncu capture of one 64-band launch)
    "plane_apply_density_pair": (3.6928e6, "889ba492c2968694"),
}


def sources_sha(name: str) -> str | None:
    import hashlib
    files = TRAFFIC_SOURCES.get(name)
    if not files:
        return None
    h = hashlib.sha256()
    for f in files:
        with open(os.path.join(ROOT, "paper_1708_03621_gb300", f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


def traffic_per_band(name: str) -> float | None:
    ent = TRAFFIC_PER_BAND.get(name)
    if ent is None or sources_sha(name) != ent[1]:
        return None
    return ent[0]


def run_ours(args, world, rank, local, pg):
    import torch

    from paper_1708_03621_gb300 import jdft
    dev = torch.device("cuda", local)
    torch.cuda.set_device(dev)
    fp32 = jdft.jdft_measure_fp32_peak()  # the FFT kernels' arithmetic roofline, on this GPU
    p = Problem(args.workload, args.prec, dev, args.nbands, autotune=not args.no_autotune)
    tune = p.tune
    stream = torch.cuda.current_stream()
    for _ in range(args.warmup):
        p.step()
    torch.cuda.synchronize()

    # ---- timed region: exactly K steps, events on the launching stream ----
    clocks = Clocks(local)
    clocks.start()
    jdft.jdft_profile_read()
    jdft.jdft_profile_enable(True)
    launches0 = jdft.jdft_launch_count()
    barrier(pg)
    torch.cuda.synchronize()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(args.steps):
        p.step()
    e1.record(stream)
    torch.cuda.synchronize()
    barrier(pg)
    launches = jdft.jdft_launch_count() - launches0
    jdft.jdft_profile_enable(False)
    prof = jdft.jdft_profile_read()
    clk = clocks.stop()
    p.check_status()
    ms = e0.elapsed_time(e1)
    ms_max, units = job_totals(pg, ms, p.nb * args.steps)
    value = units / (ms_max / 1e3)

    # ---- per-kernel roofline from the live events ----
    kernels = []
    for name, (n, kms) in sorted(prof.items(), key=lambda kv: -kv[1][1]):
        per_step_launches = n / args.steps
        fl, by = kernel_work(p, name, per_step_launches, p.nb)
        avg_s = kms / n / 1e3
        kernels.append({"name": name, "launches": n, "ms": round(kms, 3), "share": round(kms / ms, 4),
                        "gflop_per_launch": round(fl / 1e9, 4), "mb_per_launch": round(by / 1e6, 3),
                        "achieved_tflops": round(fl / avg_s / 1e12, 3) if fl else None,
                        "achieved_gbs": round(by / avg_s / 1e9, 1) if by else None})
    peaks = json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json"))) if os.path.exists(
        os.path.join(ROOT, "MEASURED_PEAKS.json")) else {}
    for k in kernels:
        k["roofline"] = roofline_of(k, args.prec, peaks, fp32)
    top = kernels[0]
    roof = dict(top["roofline"])
    roof["kernel"] = top["name"]
    tpb = traffic_per_band(top["name"]) if args.workload == "large" else None
    # per launch, like `achieved`: bytes per band x the bands one launch processes on average
    roof["traffic"] = round(tpb * p.nb * args.steps / top["launches"]) if tpb else None

    # ---- end to end through the public API with host buffers ----
    Bi, Bo = p.io_bytes()
    HC_host = torch.empty_like(p.HC, device="cpu").pin_memory()
    n_host = torch.empty_like(p.n, device="cpu").pin_memory()
    CHC_host = torch.empty_like(p.CHC, device="cpu").pin_memory()
    COC_host = torch.empty_like(p.COC, device="cpu").pin_memory()
    e2e_steps = max(4, args.steps)   # as many pipelined steps as the device-timed region
    # double-buffered: step i+1's input copy (one stream) and step i-1's output
    # copy (another: the two directions use separate copy engines) run while the
    # compute stream runs step i (two device buffer sets)
    sets = [p.own_buffers(), p.buffers()]
    comp, h2d, d2h = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.Stream()
    ev_in = [torch.cuda.Event(), torch.cuda.Event()]
    ev_out = [torch.cuda.Event(), torch.cuda.Event()]
    ev_dn = [torch.cuda.Event(), torch.cuda.Event()]
    torch.cuda.synchronize()
    barrier(pg)
    t0 = time.perf_counter()
    with torch.cuda.stream(h2d):
        sets[0]["C"].copy_(p.C_host, non_blocking=True)
        ev_in[0].record(h2d)
    for i in range(e2e_steps):
        k = i % 2
        if i + 1 < e2e_steps:
            with torch.cuda.stream(h2d):
                if i >= 1:
                    h2d.wait_event(ev_out[1 - k])  # step i-1 is done with that set's C
                sets[1 - k]["C"].copy_(p.C_host, non_blocking=True)
                ev_in[1 - k].record(h2d)
        with torch.cuda.stream(comp):
            comp.wait_event(ev_in[k])
            if i >= 2:
                comp.wait_event(ev_dn[k])  # step i-2's outputs are copied out
            p.step(comp, sets[k])
            ev_out[k].record(comp)
        with torch.cuda.stream(d2h):
            d2h.wait_event(ev_out[k])
            HC_host.copy_(sets[k]["HC"], non_blocking=True)
            n_host.copy_(sets[k]["n"], non_blocking=True)
            CHC_host.copy_(sets[k]["CHC"], non_blocking=True)
            COC_host.copy_(sets[k]["COC"], non_blocking=True)
            ev_dn[k].record(d2h)
    torch.cuda.synchronize()
    e2e_s, e2e_units = job_totals(pg, time.perf_counter() - t0, p.nb * e2e_steps)
    p.check_status()
    # ---- jdft_apply_H alone over the block (rows a1-a6, the scope's band-apply) ----
    apply_reps = max(4, args.steps // 2)
    j0, j1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    jdft.jdft_apply_H(p.basis, 0, p.C, p.HC, p.prec)
    torch.cuda.synchronize()
    j0.record(stream)
    for _ in range(apply_reps):
        jdft.jdft_apply_H(p.basis, 0, p.C, p.HC, p.prec)
    j1.record(stream)
    torch.cuda.synchronize()
    t_apply, apply_units = job_totals(pg, j0.elapsed_time(j1), p.nb * apply_reps)
    apply_h = {"band_applies_per_s": round(apply_units / (t_apply / 1e3), 1),
               "ms_per_call": round(t_apply / apply_reps, 4), "calls": apply_reps,
               "what": "jdft_apply_H over the block: scatter, FFTs, V, gather, kinetic, nonlocal (rows a1-a6)"}

    e2e = {"value": round(e2e_units / e2e_s, 1), "unit": UNIT, "h2d_bytes_per_step": Bi,
           "d2h_bytes_per_step": Bo, "steps": e2e_steps,
           "pipeline": "double-buffered: each step's input copy (pinned host -> device) and output copy "
                       "(device -> pinned host) overlap the neighbouring steps' compute, each direction on a "
                       "stream of its own"}
    del sets

    # ---- the FP64 path on the same workload, for the mixed-vs-FP64 comparison ----
    fp64 = None
    if not args.no_fp64 and args.prec != "fp64":
        del p
        torch.cuda.empty_cache()
        q = Problem(args.workload, "fp64", dev, args.nbands)
        q.step()
        torch.cuda.synchronize()
        k64 = max(2, args.steps // 10)
        a0 = torch.cuda.Event(enable_timing=True)
        a1 = torch.cuda.Event(enable_timing=True)
        a0.record(stream)
        for _ in range(k64):
            q.step()
        a1.record(stream)
        torch.cuda.synchronize()
        q.check_status()
        t64 = a0.elapsed_time(a1)
        fp64 = {"value": round(q.nb * k64 / (t64 / 1e3), 1), "ms_per_step": round(t64 / k64, 3), "steps": k64,
                "mixed_errors_vs_fp64": precision_errors(q)}
        p = q

    batch = None
    if not args.no_batch and world == 1:
        batch = batch_measurements(args.prec, dev)
    cg = None
    if not args.no_cg and world == 1:
        cg = cg_measurements(args.prec if args.prec != "fp64" else "fp32", dev)
    slab = None
    if not args.no_slab and world == 1:
        slab = slab_measurements(args.prec if args.prec != "fp64" else "bf16x3", dev)
    scf_sec = None
    if not args.no_scf and world == 1:
        scf_sec = scf_measurements(dev, fp32)
    out = {
        "metric": METRIC, "value": round(value, 1), "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": round(ms_max / args.steps, 4), "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None,
        "dtype": {"fp64": "f64", "fp32": "f32", "tf32x3": "f32+tf32x3", "bf16x3": "f32+bf16x3"}[args.prec],
        "data": "synthetic (seeded Gaussian atoms, random damped coefficients)",
        "config": {"workload": "cubic L=20 bohr, Ecut=30 Ha, box 128^3, 62759 PW, 64 atoms, 256 projectors, "
                               "256 bands, 1 k-point; step = apply_H + density + subspace + Cholesky orthonormalisation "
                               "(rows a1-a9); the band-CG row a10 is measured under 'cg'",
                   "precision": args.prec, "npw": p.npw, "nbands": p.nb, "nproj": p.nproj,
                   "l2": "working set ~0.5 GB > 126 MB L2 (C, HC, P re-read every step)",
                   "parallelism": f"replicas x{world}", "autotune": tune},
        "clocks": clk, "e2e": e2e, "gpu_launches": int(launches), "roofline": roof, "kernels": kernels,
        "kernel_times_note": "per-launch CUDA-event intervals on each launch's own stream; the overlap "
                             "factorisation runs on a side stream beside the plane pass, so shares add up to "
                             "more than 1",
        "apply_H": apply_h,
        "fp64_path": fp64,
        "cg": cg,
        "batch": batch,
        "slab": slab,
        "scf": scf_sec,
    }
    if rank == 0 and not args.no_cpu_baseline and world == 1:
        out["cpu_baseline"] = cpu_baseline(args.workload, args.cpu_seconds)
        out["cpu_baseline_cg"] = cpu_baseline_cg(args.cpu_seconds)
    if rank == 0:
        print(json.dumps(out), flush=True)


def cg_measurements(prec: str, device, log=lambda *_: None) -> dict:
    """Row a10, the preconditioned band CG, measured two ways.

    * cost of one iteration on the 128^3 workload (256 bands): wall time of
      minimisations stopped after 6 and after 2 iterations, difference / 4
      (each iteration applies H to the 256-band search direction once);
    * time to |dE| < 1e-6 Ha on the 48^3 workload (16 bands) from the seeded
      start, for FP64 + Teter, mixed + Teter and mixed + the learned network
      (committed weights), against E_ref from an FP64 run to residual 1e-10.
    """
    import torch

    from paper_1708_03621_gb300 import jdft, learned
    from synth import WORKLOADS
    out = {}
    w = WORKLOADS["large"]
    b = learned.build_cell(w, device)
    C0 = torch.tensor(learned.start_block(b, w), device=device)
    wall = {}
    for k in (2, 6):
        C = C0.clone()
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        jdft.jdft_minimize_bands(b, 0, C, tol=1e-30, max_iter=k, precond="teter", prec=prec, switch_tol=1e-30,
                                 check=False)
        wall[k] = time.perf_counter() - t0
    per_it = max(1e-9, (wall[6] - wall[2]) / 4)
    out["large_iteration_ms"] = round(per_it * 1e3, 3)
    out["large_iteration_band_applies_per_s"] = round(w.nbands / per_it, 1)
    wts = learned.load_weights()
    net = jdft.Mlp(wts) if wts is not None else None
    out["large_kernels"] = cg_kernel_shares(b, C0, prec, "mlp" if net is not None else "teter", net, iters=6)
    b.close()
    del C0, C
    w = WORKLOADS["small"]
    b = learned.build_cell(w, device)
    C0 = torch.tensor(learned.start_block(b, w), device=device)
    # configuration 1's H C throughput (16 bands, 48^3): FP64 and the mixed precision
    stream = torch.cuda.current_stream()
    for pr, ct in (("fp64", torch.complex128), (prec, torch.complex64)):
        Cx = C0.to(ct)
        Hx = torch.empty_like(Cx)
        for _ in range(5):
            jdft.jdft_apply_H(b, 0, Cx, Hx, pr)
        a0, a1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        reps = 200
        a0.record(stream)
        for _ in range(reps):
            jdft.jdft_apply_H(b, 0, Cx, Hx, pr)
        a1.record(stream)
        torch.cuda.synchronize()
        out[f"small_apply_H_{pr}_band_applies_per_s"] = round(w.nbands * reps / (a0.elapsed_time(a1) / 1e3), 1)
    C = C0.clone()
    ref = jdft.jdft_minimize_bands(b, 0, C, tol=1e-10, max_iter=5000, precond="teter", prec="fp64")
    E_ref = ref["energy"]
    runs = [("fp64", "teter", None), (prec, "teter", None)]
    wts = learned.load_weights()
    mlp = jdft.Mlp(wts) if wts is not None else None
    if mlp is not None:
        runs.append((prec, "mlp", mlp))
    res = {}
    for pr, pc, m in runs:
        best = None
        for _ in range(3):   # best of three (the first includes one-time set-up of kernels)
            C = C0.clone()
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            rep = jdft.jdft_minimize_bands(b, 0, C, tol=1e-6, max_iter=5000, precond=pc, prec=pr, mlp=m)
            dt = time.perf_counter() - t0
            if best is None or dt < best[0]:
                best = (dt, rep)
        dt, rep = best
        res[f"{pr}+{pc}"] = {"seconds": round(dt, 4), "iterations": rep["iterations"],
                             "mixed_iterations": rep["mixed_iterations"],
                             "dE_Ha": float(f"{abs(rep['energy'] - E_ref):.3e}")}
    out["small_time_to_dE_1e-6"] = res
    out["small_E_ref_Ha"] = E_ref
    b.close()
    return out


def scf_measurements(device, fp32: dict) -> dict:
    """The self-consistent field pieces (Hartree, LDA, Pulay) and the SCF loop.

    * Kohn-Sham potential (Hartree chain + LDA, jdft_ks_potential) on the 128^3
      box and one Pulay step (8 stored pairs) over it, CUDA events, after warm-up;
      inputs: a smooth positive density (Gaussians at seeded points);
    * the SCF loop (jdft_scf) on the 48^3 workload ('small', 16 bands) from the
      seeded start, FP64 band solves and BF16x3-then-FP64 band solves, wall time
      to convergence (|dE| < 1e-9 Ha between iterations and density residual
      < 1e-7), against the oracle's converged energy stored in
      tests/golden/scf_small.json.
    """
    import torch

    from paper_1708_03621_gb300 import jdft
    from synth import WORKLOADS, atom_positions, random_coefficients
    out = {}
    stream = torch.cuda.current_stream()
    # ---- field kernels at 128^3 ----
    L, S = 20.0, (128, 128, 128)
    R = np.eye(3) * L
    N = int(np.prod(S))
    b = jdft.Basis(R, S, 1.0, [(0.0, 0.0, 0.0)])
    centres = atom_positions(R, 64, 77)
    g = torch.empty(N, dtype=torch.float64, device=device)
    jdft.jdft_gaussian_potential(b, centres, g, depth=0.01, width=1.2)
    n = (-g).contiguous()
    vion = torch.empty_like(n)
    jdft.jdft_gaussian_potential(b, centres, vion)
    vks = torch.empty_like(n)
    en = torch.zeros(2, dtype=torch.float64, device=device)
    for _ in range(3):
        jdft.jdft_ks_potential(b, n, vion, vks, en)
    reps = 20
    a0, a1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a0.record(stream)
    for _ in range(reps):
        jdft.jdft_ks_potential(b, n, vion, vks, en)
    a1.record(stream)
    torch.cuda.synchronize()
    t_ks = a0.elapsed_time(a1) / reps / 1e3
    flops = 2 * 5.0 * N * math.log2(N)          # two complex 3-D FFTs, nominal 5 n log2 n each
    io = 3 * 8.0 * N                             # read n and V_ion, write V_KS
    passes = 5 * 2 * 16.0 * N                    # five axis passes over the complex box (read + write)
    out["ks_potential_128cubed"] = {
        "ms": round(t_ks * 1e3, 4), "fp64_tflops": round(flops / t_ks / 1e12, 3),
        "fp64_frac_of_nominal": round(flops / t_ks / 1e12 / FP64_NOMINAL_TFLOPS, 3),
        "io_gbs": round(io / t_ks / 1e9, 1), "axis_pass_gbs": round(passes / t_ks / 1e9, 1),
        "work": "V_KS = V_ion + V_H[n] + v_xc[n]: forward and inverse complex FP64 3-D FFTs of the box "
                "(5 n log2 n flops each) in five axis passes, Coulomb kernel and LDA fused; the transforms take the "
                "half box and run in 64-bit integers, so the nominal flops can pass the FP64 pipe's rate"}
    mix = jdft.Pulay(N, 8, 0.5)
    gen = torch.Generator(device=device)
    gen.manual_seed(79)
    preps = 10
    outs = [(n + 1e-3 * torch.randn(N, dtype=torch.float64, device=device, generator=gen)).contiguous()
            for _ in range(preps + 8)]       # independent residuals: every step combines 8 pairs
    nxt = torch.empty_like(n)
    for i in range(8):
        mix.step(n, outs[i], nxt)
    a0.record(stream)
    for i in range(preps):
        mix.step(n, outs[8 + i], nxt)
    a1.record(stream)
    torch.cuda.synchronize()
    t_p = a0.elapsed_time(a1) / preps / 1e3
    used = mix.used()
    by = (4 + (8 - 1) + 2 * 8 + 1) * 8.0 * N     # store (read 2, write 2, other residuals), mix (2 per pair, write)
    out["pulay_step_128cubed"] = {"ms": round(t_p * 1e3, 4), "pairs": used, "gbs": round(by / t_p / 1e9, 1),
                                  "bytes_per_step": by}
    mix.close()
    b.close()
    del n, g, vion, vks, outs, nxt
    # ---- the SCF loop on the 48^3 workload ----
    w = WORKLOADS["small"]
    atoms = atom_positions(w.R, w.natoms, w.seed_atoms)
    gold_path = os.path.join(ROOT, "tests", "golden", "scf_small.json")
    gold = json.load(open(gold_path)) if os.path.exists(gold_path) else None
    from paper_1708_03621_gb300 import learned
    wts = learned.load_weights()
    net = jdft.Mlp(wts) if wts is not None else None
    runs = {}
    cases = [("fp64", 0.0, "teter"), ("bf16x3", 0.0, "teter"), ("fp64", -1.0, "teter")]
    if net is not None:
        cases.append(("bf16x3", 0.0, "mlp"))
    for prec, factor, pc in cases:
        best = None
        for _ in range(2):
            b = jdft.Basis(w.R, w.S, w.ecut, w.kfrac, w.weights())
            vion = torch.empty(int(np.prod(w.S)), dtype=torch.float64, device=device)
            jdft.jdft_gaussian_potential(b, atoms, vion)
            P = torch.empty((4 * w.natoms, b.npw(0)), dtype=torch.complex128, device=device)
            jdft.jdft_gaussian_projectors(b, 0, atoms, P)
            D = torch.tensor(np.diag(np.tile([0.5, -0.3, -0.3, -0.3], w.natoms)), device=device)
            jdft.jdft_set_projectors(b, 0, P, D)
            G = b.gvectors(0).astype(np.float64) + np.asarray(w.kfrac[0])
            Bm = 2 * np.pi * np.linalg.inv(w.R).T
            q = G @ Bm.T
            kin2 = np.einsum("ij,ij->i", q, q)
            C = torch.tensor(random_coefficients(kin2, w.nbands, w.seed_coeffs), device=device)
            dens = torch.empty_like(vion)
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            rep = jdft.jdft_scf(b, [C], vion, dens, tol_energy=1e-9, tol_density=1e-7, band_tol=1e-9, prec=prec,
                                band_tol_factor=factor, precond=pc, mlp=net if pc == "mlp" else None)
            dt = time.perf_counter() - t0
            b.close()
            if best is None or dt < best[0]:
                best = (dt, rep)
        dt, rep = best
        key = prec + ("_fixed_band_tol" if factor < 0 else "") + ("+mlp" if pc == "mlp" else "")
        runs[key] = {"seconds": round(dt, 4), "scf_iterations": rep["iterations"],
                     "band_iterations": rep["band_iterations"], "energy_Ha": rep["energy"],
                     "dE_vs_oracle_Ha": float(f"{abs(rep['energy'] - gold['energy']):.3e}") if gold else None}
    out["small_scf"] = runs
    out["pcm_128cubed"] = pcm_measurements(device)
    out["spinor"] = spinor_measurements(device)
    out["augmented_overlap"] = overlap_measurements(device)
    out["small_scf_workload"] = ("48^3 'small' cell (L=10, Ecut=20, 4259 PW, 8 atoms, 16 bands, f=2), Gaussian "
                                 "V_ion + projectors, LDA (PZ81) + Hartree, Pulay 8 pairs alpha 0.5; band solves "
                                 "Teter-preconditioned CG warm-started each iteration, to max(1e-9, 0.01 x the "
                                 "previous density residual) (the _fixed_band_tol run: 1e-9 throughout; +mlp: the "
                                 "committed network as preconditioner)")
    return out


def overlap_measurements(device) -> dict:
    """The augmented overlap S = Omega + P Q P^dag (Q = diag(0.4, 0.1, 0.1, 0.1)
    per atom): jdft_op_S over the 128^3 workload's 256-band block in BF16x3
    (CUDA events), and the generalised band minimiser on the 48^3 workload
    (16 bands, FP64, Teter, to 1e-8) beside the plain minimiser on the same
    cell without augmentation."""
    import torch

    from paper_1708_03621_gb300 import jdft
    from synth import WORKLOADS, atom_positions, random_coefficients
    out = {}
    stream = torch.cuda.current_stream()
    for wname in ("large", "small"):
        w = WORKLOADS[wname]
        atoms = atom_positions(w.R, w.natoms, w.seed_atoms)
        b = jdft.Basis(w.R, w.S, w.ecut, w.kfrac, w.weights())
        N = int(np.prod(w.S))
        V = torch.empty(N, dtype=torch.float64, device=device)
        jdft.jdft_gaussian_potential(b, atoms, V)
        jdft.jdft_set_potential(b, V)
        P = torch.empty((4 * w.natoms, b.npw(0)), dtype=torch.complex128, device=device)
        jdft.jdft_gaussian_projectors(b, 0, atoms, P)
        D = torch.tensor(np.diag(np.tile([0.5, -0.3, -0.3, -0.3], w.natoms)), device=device)
        jdft.jdft_set_projectors(b, 0, P, D)
        G = b.gvectors(0).astype(np.float64) + np.asarray(w.kfrac[0])
        q = G @ (2 * np.pi * np.linalg.inv(w.R).T).T
        C0 = torch.tensor(random_coefficients(np.einsum("ij,ij->i", q, q), w.nbands, w.seed_coeffs), device=device)
        Q = torch.tensor(np.diag(np.tile([0.4, 0.1, 0.1, 0.1], w.natoms)), device=device)
        if wname == "large":
            jdft.jdft_set_augmentation(b, 0, Q)
            C = C0.to(torch.complex64)
            SC = torch.empty_like(C)
            for _ in range(3):
                jdft.jdft_op_S(b, 0, C, SC, "bf16x3")
            a0, a1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a0.record(stream)
            for _ in range(10):
                jdft.jdft_op_S(b, 0, C, SC, "bf16x3")
            a1.record(stream)
            torch.cuda.synchronize()
            out["op_S_128cubed_256bands_bf16x3_ms"] = round(a0.elapsed_time(a1) / 10, 4)
        else:
            res = {}
            for name, aug in (("plain", False), ("augmented", True)):
                jdft.jdft_set_augmentation(b, 0, Q if aug else None)
                C = C0.clone()
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                if aug:
                    rep = jdft.jdft_minimize_bands_generalized(b, 0, C, tol=1e-8, max_iter=3000)
                else:
                    rep = jdft.jdft_minimize_bands(b, 0, C, tol=1e-8, max_iter=3000, precond="teter", prec="fp64")
                res[name] = {"seconds": round(time.perf_counter() - t0, 4), "iterations": rep["iterations"],
                             "energy_Ha": rep["energy"]}
            out["small_minimise_fp64_teter"] = res
        b.close()
    return out


def spinor_measurements(device) -> dict:
    """Spinor bands in a noncollinear potential (jdft_apply_H_spinor): the 48^3
    workload with 16 spinor bands (FP64 and FP32) and the 128^3 workload with
    64 spinor bands (FP32 transforms; projector products on CUDA cores or as
    BF16x3 tensor-core products), a smooth seeded M(r); CUDA events after warm-up.
    One spinor band-apply = H applied to both components of one band."""
    import torch

    from paper_1708_03621_gb300 import jdft
    from synth import WORKLOADS, atom_positions, random_coefficients
    out = {}
    stream = torch.cuda.current_stream()
    for wname, nb, precs in (("small", 16, ("fp64", "fp32")), ("large", 64, ("fp32", "bf16x3"))):
        w = WORKLOADS[wname]
        atoms = atom_positions(w.R, w.natoms, w.seed_atoms)
        b = jdft.Basis(w.R, w.S, w.ecut, w.kfrac, w.weights())
        N = int(np.prod(w.S))
        V = torch.empty(N, dtype=torch.float64, device=device)
        jdft.jdft_gaussian_potential(b, atoms, V)
        jdft.jdft_set_potential(b, V)
        P = torch.empty((4 * w.natoms, b.npw(0)), dtype=torch.complex128, device=device)
        jdft.jdft_gaussian_projectors(b, 0, atoms, P)
        D = torch.tensor(np.diag(np.tile([0.5, -0.3, -0.3, -0.3], w.natoms)), device=device)
        jdft.jdft_set_projectors(b, 0, P, D)
        G = b.gvectors(0).astype(np.float64) + np.asarray(w.kfrac[0])
        q = G @ (2 * np.pi * np.linalg.inv(w.R).T).T
        C64 = torch.tensor(random_coefficients(np.einsum("ij,ij->i", q, q), 2 * nb, 31), device=device)
        M = torch.empty(3 * N, dtype=torch.float64, device=device)
        for c in range(3):
            jdft.jdft_gaussian_potential(b, atom_positions(w.R, 4, 40 + c), M[c * N:(c + 1) * N], depth=0.2,
                                         width=2.0)
        for prec in precs:
            C = C64 if prec == "fp64" else C64.to(torch.complex64)
            HC = torch.empty_like(C)
            for _ in range(3):
                jdft.jdft_apply_H_spinor(b, 0, M, C, HC, prec)
            a0, a1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            reps = 10
            a0.record(stream)
            for _ in range(reps):
                jdft.jdft_apply_H_spinor(b, 0, M, C, HC, prec)
            a1.record(stream)
            torch.cuda.synchronize()
            ms = a0.elapsed_time(a1) / reps
            out[f"{wname}_{nb}bands_{prec}"] = {"ms_per_call": round(ms, 4),
                                               "spinor_band_applies_per_s": round(nb / (ms / 1e3), 1)}
        b.close()
    return out


def pcm_measurements(device) -> dict:
    """The paper's LinearPCM example on the 128^3 box (L = 20 bohr): a
    solute-shaped dielectric (eps = 1 within ~2 bohr of 64 seeded centres,
    78.4 outside, smooth switch) and the Gaussian charges at those centres;
    jdft_pcm_solve to |r| < 1e-10 |rho~| from phi~ = 0, and one hessian alone
    (CUDA events, after warm-up)."""
    import torch

    from paper_1708_03621_gb300 import jdft
    from synth import atom_positions
    L, S = 20.0, (128, 128, 128)
    R = np.eye(3) * L
    N = int(np.prod(S))
    b = jdft.Basis(R, S, 1.0, [(0.0, 0.0, 0.0)])
    centres = atom_positions(R, 64, 78)
    shape = torch.empty(N, dtype=torch.float64, device=device)
    jdft.jdft_gaussian_potential(b, centres, shape, depth=6.0, width=2.0)
    eps = (1.0 + 77.4 * torch.exp(shape)).contiguous()          # shape <= 0: exp(-sum of Gaussians)
    rho = torch.empty(N, dtype=torch.float64, device=device)
    jdft.jdft_gaussian_potential(b, centres, rho, depth=0.5, width=0.8)
    rho_t = torch.empty(N, dtype=torch.complex128, device=device)
    jdft.jdft_field_J(b, (-rho).to(torch.complex128), rho_t)
    phi = torch.empty_like(rho_t)
    solves = {}
    for prec in ("fp64", "fp32"):
        best = None
        for _ in range(2):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            rep = jdft.jdft_pcm_solve(b, eps, rho_t, phi, tol=1e-10, max_iter=2000, prec=prec)
            wall = time.perf_counter() - t0
            if best is None or wall < best[0]:
                best = (wall, rep)
        wall, rep = best
        solves[prec] = {"iterations": rep["iterations"], "fp64_hessians": rep["fp64_hessians"],
                        "residual": rep["residual"], "A_diel_Ha": rep["A_diel"], "solve_seconds": round(wall, 4),
                        "ms_per_iteration": round(wall / max(1, rep["iterations"]) * 1e3, 4)}
    H = torch.empty_like(phi)
    stream = torch.cuda.current_stream()
    for _ in range(3):
        jdft.jdft_pcm_hessian(b, eps, phi, H)
    a0, a1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    reps = 10
    a0.record(stream)
    for _ in range(reps):
        jdft.jdft_pcm_hessian(b, eps, phi, H)
    a1.record(stream)
    torch.cuda.synchronize()
    t_h = a0.elapsed_time(a1) / reps / 1e3
    flops = 6 * 5.0 * N * math.log2(N)      # three inverse and three forward complex 3-D FFTs
    b.close()
    return {"solve": solves, "hessian_ms": round(t_h * 1e3, 4), "hessian_fp64_tflops": round(flops / t_h / 1e12, 3),
            "hessian_fp64_frac_of_nominal": round(flops / t_h / 1e12 / FP64_NOMINAL_TFLOPS, 3),
            "work": "hessian = 6 complex FP64 3-D FFTs of the box (5 n log2 n each) + gradient, eps product, "
                    "divergence fused into the axis passes; transforms in 64-bit integers, so the nominal flops can pass "
                    "the FP64 pipe's rate"}


def slab_measurements(prec: str, device) -> dict:
    """Configuration 5, the 40 x 20 x 20 bohr slab (box 256 x 128 x 128, 125 k
    plane waves, 256 atoms, 1024 projectors, 1024 bands, 4 k-points):

    * mixed-precision H C + C^dag H C over the band block at every k-point
      (one pass = 4 x 1024 band-applies), CUDA events, after one warm-up pass;
    * the same at k-point 0 on the plain FP64 GPU path, and the mixed result's
      errors against it;
    * one learned-preconditioned mixed band-CG iteration at k-point 0 (wall
      time of 4-iteration minus 2-iteration runs, / 2).

    The band block is drawn on the GPU from a seeded generator with the same
    recipe as the other workloads: complex N(0, 1) / (1 + |k+G|^2), each band
    normalised to Omega sum |C|^2 = 1.
    """
    import torch

    from paper_1708_03621_gb300 import jdft, learned
    from synth import WORKLOADS, workload_atoms
    w = WORKLOADS["slab"]
    atoms = workload_atoms(w)
    b = jdft.Basis(w.R, w.S, w.ecut, w.kfrac, w.weights())
    omega = b.info(0)["omega"]
    V = torch.empty(int(np.prod(w.S)), dtype=torch.float64, device=device)
    jdft.jdft_gaussian_potential(b, atoms, V)
    jdft.jdft_set_potential(b, V)
    del V
    D = torch.tensor(np.diag(np.tile([0.5, -0.3, -0.3, -0.3], w.natoms)), device=device)
    Bm = 2 * np.pi * np.linalg.inv(w.R).T
    blocks = []
    for ik in range(w.nk):
        npw = b.npw(ik)
        P = torch.empty((4 * w.natoms, npw), dtype=torch.complex128, device=device)
        jdft.jdft_gaussian_projectors(b, ik, atoms, P)
        jdft.jdft_set_projectors(b, ik, P, D)
        del P
        q = (b.gvectors(ik).astype(np.float64) + np.asarray(w.kfrac[ik])) @ Bm.T
        damp = torch.tensor(1.0 / (1.0 + np.sum(q * q, 1)), dtype=torch.float32, device=device)
        gen = torch.Generator(device=device)
        gen.manual_seed(w.seed_coeffs * 10 + ik)
        Y = torch.view_as_complex(torch.randn((w.nbands, npw, 2), generator=gen, device=device,
                                              dtype=torch.float32)) * damp[None, :]
        Y /= torch.sqrt(omega * torch.sum(Y.abs() ** 2, dim=1, keepdim=True))
        blocks.append((Y, torch.empty_like(Y)))
    nb = w.nbands
    CHC = torch.empty((nb, nb), dtype=torch.complex128, device=device)

    def mixed_pass():
        for ik, (C, HC) in enumerate(blocks):
            jdft.jdft_apply_H(b, ik, C, HC, prec)
            jdft.jdft_subspace(b, ik, C, HC, CHC, None, prec)

    stream = torch.cuda.current_stream()
    mixed_pass()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    reps = 2
    jdft.jdft_profile_read()
    jdft.jdft_profile_enable(True)
    e0.record(stream)
    for _ in range(reps):
        mixed_pass()
    e1.record(stream)
    torch.cuda.synchronize()
    jdft.jdft_profile_enable(False)
    prof = jdft.jdft_profile_read()
    t_mixed = e0.elapsed_time(e1) / reps
    # the dominant kernel of the pass against its roofline (work model of k-point 0)
    import types
    iG0 = b.gvectors(0)
    sp = types.SimpleNamespace(w=types.SimpleNamespace(S=w.S), info=b.info(0), nrows=int(iG0[:, 0].max() -
                               iG0[:, 0].min() + 1), C=blocks[0][0], N=int(np.prod(w.S)), npw=b.npw(0),
                               nproj=4 * w.natoms, nb=nb)
    fp32 = jdft.jdft_measure_fp32_peak()
    peaks = json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json"))) if os.path.exists(
        os.path.join(ROOT, "MEASURED_PEAKS.json")) else {}
    top_name, (top_n, top_ms) = max(prof.items(), key=lambda kv: kv[1][1])
    fl, by = kernel_work(sp, top_name, top_n / (reps * w.nk), nb)
    avg_s = top_ms / top_n / 1e3
    k = {"name": top_name, "achieved_tflops": round(fl / avg_s / 1e12, 3) if fl else None,
         "achieved_gbs": round(by / avg_s / 1e9, 1) if by else None}
    slab_roof = roofline_of(k, prec, peaks, fp32)
    slab_roof.update({"kernel": top_name, "share": round(top_ms / (t_mixed * reps), 4),
                      "launches_per_pass": round(top_n / reps, 2)})
    out = {"workload": "slab 40x20x20 bohr, Ecut 30, box 256x128x128, 256 atoms, 1024 projectors, "
                       "1024 bands x 4 k-points; pass = H C + C^dag H C at every k",
           "roofline": slab_roof,
           "npw": [b.npw(ik) for ik in range(w.nk)], "precision": prec,
           "mixed_ms_per_pass": round(t_mixed, 3),
           "mixed_band_applies_per_s": round(w.nk * nb / (t_mixed / 1e3), 1)}
    # plain FP64 at k-point 0
    C0, HC0 = blocks[0]
    C64 = C0.to(torch.complex128)
    HC64 = torch.empty_like(C64)
    CHC64 = torch.empty_like(CHC)
    jdft.jdft_apply_H(b, 0, C64, HC64, "fp64")
    torch.cuda.synchronize()
    e0.record(stream)
    jdft.jdft_apply_H(b, 0, C64, HC64, "fp64")
    jdft.jdft_subspace(b, 0, C64, HC64, CHC64, None, "fp64")
    e1.record(stream)
    torch.cuda.synchronize()
    t64 = e0.elapsed_time(e1)
    out["fp64_ms_per_k"] = round(t64, 3)
    out["fp64_band_applies_per_s"] = round(nb / (t64 / 1e3), 1)
    out["mixed_vs_fp64_per_k"] = round((t64 / 1e3) / (t_mixed / 1e3 / w.nk), 2)
    jdft.jdft_apply_H(b, 0, C0, HC0, prec)
    jdft.jdft_subspace(b, 0, C0, HC0, CHC, None, prec)
    torch.cuda.synchronize()
    num = torch.linalg.vector_norm(HC0.to(torch.complex128) - HC64, dim=1)
    den = torch.linalg.vector_norm(HC64, dim=1)
    out["hc_band_rel_max"] = float(f"{float(torch.max(num / den)):.3e}")
    out["chc_rel"] = float(f"{float(torch.max(torch.abs(CHC - CHC64)) / torch.max(torch.abs(CHC64))):.3e}")
    del C64, HC64, CHC64
    # one learned-preconditioned mixed band-CG iteration at k-point 0
    wts = learned.load_weights()
    mlp = jdft.Mlp(wts) if wts is not None else None
    pc = "mlp" if mlp is not None else "teter"
    wall = {}
    for k in (2, 4):
        C = C0.to(torch.complex128)  # the minimiser takes (and returns) an FP64 block
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        jdft.jdft_minimize_bands(b, 0, C, tol=1e-30, max_iter=k, precond=pc, prec=prec, switch_tol=1e-30,
                                 check=False, mlp=mlp)
        wall[k] = time.perf_counter() - t0
        del C
    out["cg_preconditioner"] = pc
    out["cg_iteration_ms"] = round(max(1e-9, (wall[4] - wall[2]) / 2) * 1e3, 3)
    out["cg_kernels"] = cg_kernel_shares(b, C0, prec, pc, mlp, iters=4)
    del blocks
    b.close()
    torch.cuda.empty_cache()
    return out


def cg_kernel_shares(b, C0, prec, precond, mlp, iters: int = 4, top: int = 10) -> dict:
    """Where a band-CG iteration's time goes, per kernel (library tracing, CUDA
    events around every launch), the preconditioner network's kernels
    included: two traced minimisations stopped after 2 and after 2 + iters
    iterations, differenced, so that the set-up of each call and the FP64
    phase's start (orthonormalisation and subspace products on the FP64 block,
    run once per call) cancel."""
    import torch

    from paper_1708_03621_gb300 import jdft
    runs = {}
    for k in (2, 2 + iters):
        C = C0.to(torch.complex128).clone()
        torch.cuda.synchronize()
        jdft.jdft_profile_read()
        jdft.jdft_profile_enable(True)
        t0 = time.perf_counter()
        jdft.jdft_minimize_bands(b, 0, C, tol=1e-30, max_iter=k, precond=precond, prec=prec, switch_tol=1e-30,
                                 check=False, mlp=mlp)
        torch.cuda.synchronize()
        wall = time.perf_counter() - t0
        jdft.jdft_profile_enable(False)
        runs[k] = (wall, jdft.jdft_profile_read())
        del C
    (wa, pa), (wb, pb) = runs[2], runs[2 + iters]
    it_ms = max(1e-9, (wb - wa) / iters * 1e3)
    rows = []
    for name, (n, ms) in pb.items():
        n0, ms0 = pa.get(name, (0, 0.0))
        d = (ms - ms0) / iters
        if d > 0:
            rows.append({"name": name, "launches_per_iteration": round((n - n0) / iters, 2),
                         "ms_per_iteration": round(d, 3), "share_of_iteration": round(d / it_ms, 4)})
    rows.sort(key=lambda r: -r["ms_per_iteration"])
    return {"iterations_differenced": iters, "preconditioner": precond, "iteration_ms": round(it_ms, 3),
            "kernels": rows[:top]}


def precision_errors(q) -> dict:
    """Errors of the mixed modes on the full workload against the FP64 path.

    The FP64 GPU path equals the oracle to 1e-10 (parity tests), so it stands
    in for it at this size.  Per mode: the largest per-band relative error of
    H C, the relative error of C^dag H C (max-abs over max-abs), and the
    largest error of the subspace eigenvalues (Ha), all on the same block.
    """
    import torch

    j = q.jdft
    C64 = q.C.clone()
    j.jdft_orthonormalize(q.basis, 0, C64, "fp64")
    H64 = torch.empty_like(C64)
    j.jdft_apply_H(q.basis, 0, C64, H64, "fp64")
    S64 = torch.empty((q.nb, q.nb), dtype=torch.complex128, device=C64.device)
    j.jdft_subspace(q.basis, 0, C64, H64, S64, None, "fp64")
    e64 = torch.empty(q.nb, dtype=torch.float64, device=C64.device)
    j.jdft_subspace_eigs(S64, e64)
    out = {}
    for prec in ("fp32", "tf32x3", "bf16x3"):
        C = C64.to(torch.complex64)
        H = torch.empty_like(C)
        j.jdft_apply_H(q.basis, 0, C, H, prec)
        S = torch.empty_like(S64)
        j.jdft_subspace(q.basis, 0, C, H, S, None, prec)
        e = torch.empty_like(e64)
        j.jdft_subspace_eigs(S, e)
        dH = (H.to(torch.complex128) - H64).abs().pow(2).sum(1).sqrt() / H64.abs().pow(2).sum(1).sqrt()
        out[prec] = {"hc_band_rel_max": float(f"{dH.max().item():.3e}"),
                     "chc_rel": float(f"{((S - S64).abs().max() / S64.abs().max()).item():.3e}"),
                     "eig_abs_max_Ha": float(f"{(e - e64).abs().max().item():.3e}")}
    return out


def batch_measurements(prec: str, device, reps: int = 3) -> dict:
    """Batched Hamiltonian applications replayed as one CUDA graph each.

    * 32 k-points uniform in the Brillouin zone of the L = 20 bohr, E_cut = 30 Ha
      cell (128^3 box, 64 atoms), 128 bands each: uneven sphere sizes;
    * 8 independent cubic cells, L ~ U[8, 16] bohr, E_cut = 20 Ha, boxes 40^3..80^3,
      16..128 bands, 4..32 atoms.
    Band-applies per second of the graph replay (events on the launch stream).
    """
    import torch

    from paper_1708_03621_gb300 import jdft, learned
    from synth import Workload, random_cells, random_kpoints
    ct = torch.complex128 if prec == "fp64" else torch.complex64
    out = {}
    stream = torch.cuda.current_stream()

    def timed(batch, units):
        batch.launch()
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(reps):
            batch.launch()
        e1.record(stream)
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1) / reps
        return round(units / (ms / 1e3), 1), round(ms, 3)

    kp = tuple(tuple(k) for k in random_kpoints(32, 21))
    wk = Workload("kbatch32", (20.0, 20.0, 20.0), 30.0, (128, 128, 128), kp, 64, 128, 11, 12)
    b = learned.build_cell(wk, device)
    npws = [b.npw(ik) for ik in range(wk.nk)]
    items = []
    for ik in range(wk.nk):
        C = torch.tensor(learned.start_block(b, wk, ik=ik, seed=1000 + ik), device=device).to(ct)
        items.append((b, ik, C, torch.empty_like(C), prec))
    bt = jdft.Batch(items)
    v, ms = timed(bt, wk.nk * wk.nbands)
    out["kpoints32"] = {"band_applies_per_s": v, "ms_per_launch": ms, "nk": wk.nk, "nbands": wk.nbands,
                        "npw_min": min(npws), "npw_max": max(npws)}
    bt.close()
    del items
    b.close()
    torch.cuda.empty_cache()
    cells = random_cells(8, 29)
    items, bases = [], []
    for w in cells:
        bc = learned.build_cell(w, device)
        bases.append(bc)
        C = torch.tensor(learned.start_block(bc, w), device=device).to(ct)
        items.append((bc, 0, C, torch.empty_like(C), prec))
    bt = jdft.Batch(items)
    units = sum(w.nbands for w in cells)
    v, ms = timed(bt, units)
    out["cells8"] = {"band_applies_per_s": v, "ms_per_launch": ms, "bands": units,
                     "boxes": [w.S[0] for w in cells], "nbands": [w.nbands for w in cells]}
    bt.close()
    return out


def oracle_sample_step(o, C):
    """The oracle's version of one step on a sample of bands (band-major C)."""
    from oracle import planewave as pw
    HC = o.apply_H(C)
    pw.density(o.basis, C.T, np.full(C.shape[0], 2.0))
    pw.subspace(o.basis, C.T, HC.T)
    pw.lowdin(C.T, o.basis.Omega)
    return HC


def cpu_baseline(wname: str, seconds: float) -> dict:
    """The FP64 oracle as it stands, on the host cores, on a bounded sample of bands."""
    from oracle import cfft
    from tests.systems import OracleSystem, workload
    o = OracleSystem(workload(wname))
    C = o.coeffs()
    t0 = time.perf_counter()
    done = 0
    while True:
        oracle_sample_step(o, C[done % C.shape[0]:done % C.shape[0] + 1])
        done += 1
        if time.perf_counter() - t0 > seconds or done >= C.shape[0]:
            break
    dt = time.perf_counter() - t0
    return {"value": round(done / dt, 4), "unit": UNIT, "cores": cfft.num_threads(), "kind": "oracle",
            "sample": f"{done} of {C.shape[0]} bands, one band per oracle call (apply_H + density + "
                      f"subspace row + orthonormalisation), {dt:.1f} s"}


def cpu_baseline_cg(seconds: float) -> dict:
    """The oracle's band CG (FP64, Teter) on the 48^3 system, as it stands, on
    the host cores: iterations from the seeded start within a bounded time."""
    from oracle import cfft
    from oracle import minimize as mn
    from oracle import planewave as pw
    from tests.systems import OracleSystem, workload
    o = OracleSystem(workload("small"))
    C0 = pw.lowdin(o.coeffs(16).T, o.basis.Omega)
    happly = lambda X: pw.apply_H(o.basis, o.V, X, o.P, o.D)
    its = 2
    while True:
        t0 = time.perf_counter()
        mn.minimize_bands(o.basis, happly, C0, tol=1e-30, max_iter=its)
        dt = time.perf_counter() - t0
        if dt > seconds / 3 or its >= 64:
            break
        its *= 2
    return {"value": round(its / dt, 4), "unit": "CG iterations/s", "cores": cfft.num_threads(), "kind": "oracle",
            "sample": f"{its} Teter-preconditioned iterations of the 48^3, 16-band minimisation from the seeded "
                      f"start, {dt:.1f} s (the GPU run takes 82-125 iterations to |dE| < 1e-6 Ha)"}


def run_reference(args, world, rank):
    """The oracle timed as the reference arm (rank 0 only)."""
    if rank != 0:
        return
    from oracle import cfft
    from tests.systems import OracleSystem, workload
    o = OracleSystem(workload(args.workload))
    C = o.coeffs()
    per_step = 1
    for i in range(args.warmup):
        oracle_sample_step(o, C[i % C.shape[0]:i % C.shape[0] + per_step])
    t0 = time.perf_counter()
    for i in range(args.steps):
        oracle_sample_step(o, C[i % C.shape[0]:i % C.shape[0] + per_step])
    dt = time.perf_counter() - t0
    value = per_step * args.steps / dt
    out = {"metric": METRIC, "value": round(value, 4), "unit": UNIT, "n_gpus": world, "steps": args.steps,
           "warmup": args.warmup, "ms_per_step": round(dt / args.steps * 1e3, 2), "higher_is_better": True,
           "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic", "impl": "reference",
           "config": {"workload": "cubic L=20 bohr, Ecut=30 Ha, box 128^3, 62759 PW, 64 atoms, 256 projectors, "
                                  "256 bands, 1 k-point; step = apply_H + density + subspace + orthonormalisation",
                      "sample": f"{per_step} band per step (bounded sample of the 256-band block)"},
           "cpu_baseline": {"value": round(value, 4), "unit": UNIT, "cores": cfft.num_threads(), "kind": "oracle",
                            "sample": f"{per_step} band per step, {args.steps} steps"},
           "e2e": {"value": round(value, 4), "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(out), flush=True)


def main():
    args = parse()
    world, rank, local, pg = dist_setup()
    if args.impl == "reference":
        run_reference(args, world, rank)
    else:
        run_ours(args, world, rank, local, pg)
    if pg is not None:
        pg.destroy_process_group()


if __name__ == "__main__":
    main()
