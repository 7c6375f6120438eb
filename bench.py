#!/usr/bin/env python3
"""Benchmark of the cluster-TEBD iteration at chi_max = 1024 (cfg4 workload).

Workload: the 500-qubit, 100-layer Clifford+T (20% T) random-structured
circuit of the chi_max=1024 configuration (cutoff 1e-8, k_max 4,
Q_max = 24), run from a synthetic saturated state: every interior bond at
chi = 1024 (Haar-random right isometries, Porter-Thomas spectra), i.e. the
regime in which the iteration spends its time.  A "step" is one cluster-TEBD
iteration (partition + all cluster updates of the iteration, batched).  The
metric is cluster updates (clusters with k >= 2) per second.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

One JSON line on rank 0.  For N > 1 (torchrun), every rank runs an
independent replica (the path has no exchange step): value = units of all
ranks / max time over ranks, scaling "weak".
"""
from __future__ import annotations

import argparse
import hashlib
import json
import math
import os
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "cluster updates/s and TFLOP/s (% TC peak) at χ=1024 vs plain FP64 GPU path"
UNIT = "cluster updates/s"

# DRAM traffic of the FP32 round update (k_eig_apply_f32) per algorithmic flop,
# from one ncu capture of run_apply_traffic at n = 60 (G and V of the launch
# about 1 GB, eight times L2).  The figure holds for the kernel source it was
# taken on: the reported traffic is null once that text changes.  The round
# update reads and writes each tile once per 64^3 complex product, so its bytes
# grow with its flops and the per-flop figure scales to any launch.
APPLY_TRAFFIC = {
    "bytes_per_flop": (474915328 + 552583168) / 39868956672.0,
    "source_sha256": "d3f456cd52e33ea1c998d4cca88a5959cb948bf7050a961d0b27711949bd845f",
    "capture": "ncu dram__bytes_read.sum + dram__bytes_write.sum of the first k_eig_apply_f32 launch of "
               "'bench.py --workload apply-traffic --n 60' on a GB300 (15 problems, widths up to 2048, "
               "about 1 GB of G and V): 474,915,328 + 552,583,168 B for 3.987e10 algorithmic flops, "
               "scaled to this launch's flops",
}


# DRAM traffic of the bidiagonalisation (k_bidiag) per algorithmic flop, from one
# ncu capture of run_bidiag_traffic at n = 32: one level of a saturated chi =
# 1024 iteration, the cluster sizes of the default workload.  Null once the
# kernel's source changes.
BIDIAG_TRAFFIC = {
    "bytes_per_flop": (117199380992 + 189555739648) / 462066898261.3,
    "source_sha256": "9bd3cec63e13aec51b5aa411346ad27f44b7b1e5a3782f34db7c6b38c6015a22",
    "capture": "ncu dram__bytes_read.sum + dram__bytes_write.sum of the first k_bidiag launch of "
               "'bench.py --workload bidiag-traffic --n 32' on a GB300 (2048 columns and 512, 2048, 2048, 4096 and "
               "8192 rows; the launch keeps its rows in global memory): 117,199,380,992 + 189,555,739,648 B for "
               "4.621e11 algorithmic flops, scaled to this launch's flops",
}


def bidiag_kernel_digest() -> str:
    """sha256 of the bidiagonalisation kernel's source text (comment and body)
    and of its launch plan."""
    src = open(os.path.join(ROOT, "paper_2502_19289_gb300", "csrc", "svd_direct.cu")).read()
    a = src.index("// One Golub-Kahan step per column k.")
    b = src.index("\n}\n", src.index("k_bidiag(const DirProb*", a)) + 3
    c = src.index("// Launch shape of a class of problems")
    d = src.index("\n}\n", c) + 3
    return hashlib.sha256((src[a:b] + src[c:d]).encode()).hexdigest()


def apply_kernel_digest() -> str:
    """sha256 of the FP32 round-update kernel's source text (comment, tile
    constants and kernel body)."""
    src = open(os.path.join(ROOT, "paper_2502_19289_gb300", "csrc", "kernels.cu")).read()
    a = src.index("// FP32 apply, one 64 x 64")
    b = src.index("\n}\n", src.index("k_eig_apply_f32(const EigProb*", a)) + 3
    return hashlib.sha256(src[a:b].encode()).hexdigest()


def traffic_per_launch(kernel: str, flops_per_launch: float):
    """(bytes, note) for a launch of the given algorithmic flops."""
    known = {"eig_apply": (APPLY_TRAFFIC, apply_kernel_digest), "bidiag": (BIDIAG_TRAFFIC, bidiag_kernel_digest)}
    if kernel not in known:
        return None, "no capture of this kernel"
    t, digest = known[kernel]
    if t["bytes_per_flop"] is None:
        return None, "no capture"
    if t["source_sha256"] != digest():
        return None, "kernel changed since the capture"
    return t["bytes_per_flop"] * flops_per_launch, t["capture"]


def peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        d = json.load(open(p))
        d["source"] = "measured"
        return d
    return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0,
            "sm_max_mhz": 2070.0, "source": "fallback"}


def measure_compute_peaks(P, torch, device):
    """FP32 CUDA-core and TF32 tensor-core throughput measured on this device.

    FP32: the library's FMA-loop probe (best and mean of 5 launches).  TF32:
    torch.matmul of 8192^3 fp32 operands with TF32 enabled (cuBLAS), best of 10
    back-to-back (burst) and a ~4 s back-to-back loop (sustained).  The SM count
    is the device's own."""
    best, mean, sms = P.measure_fma(5)
    out = {"fp32_simt_tflops": best, "fp32_simt_tflops_mean": mean, "n_sm": sms,
           "fp32_source": "measured: FMA-loop probe (4 x 256 threads per SM, 8 chains), best of 5"}
    prev = torch.backends.cuda.matmul.allow_tf32
    try:
        torch.backends.cuda.matmul.allow_tf32 = True
        n = 8192
        a = torch.randn(n, n, device=device, dtype=torch.float32)
        b = torch.randn(n, n, device=device, dtype=torch.float32)
        c = a @ b
        torch.cuda.synchronize()
        ts = []
        for _ in range(10):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            c = a @ b
            e1.record()
            e1.synchronize()
            ts.append(e0.elapsed_time(e1) / 1e3)
        burst = 2.0 * n ** 3 / min(ts) / 1e12
        reps, t0 = 0, time.perf_counter()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        while time.perf_counter() - t0 < 4.0:
            for _ in range(8):
                c = a @ b
            reps += 8
            torch.cuda.synchronize()
        e1.record()
        e1.synchronize()
        sustained = 2.0 * n ** 3 * reps / (e0.elapsed_time(e1) / 1e3) / 1e12
        out.update({"tf32_tflops": burst, "tf32_tflops_sustained": sustained,
                    "tf32_source": "measured: torch.matmul fp32 8192^3 with TF32 (cuBLAS), best of 10 "
                                   "and a 4 s loop"})
        del a, b, c
        torch.cuda.empty_cache()
    finally:
        torch.backends.cuda.matmul.allow_tf32 = prev
    return out


class Clocks:
    """nvidia-smi sampling during the timed region."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.idx = gpu_index
        self.p = None
        fd, self.out = tempfile.mkstemp(prefix="ctebd_clocks_", suffix=".csv")
        os.close(fd)

    def __enter__(self):
        try:
            self.f = open(self.out, "w")
            self.p = subprocess.Popen(["nvidia-smi", f"--id={self.idx}", f"--query-gpu={self.Q}",
                                       "--format=csv,noheader,nounits", "-lms", "200"],
                                      stdout=self.f, stderr=subprocess.DEVNULL)
        except Exception:
            self.p = None
        return self

    def __exit__(self, *a):
        if self.p:
            self.p.terminate()
            try:
                self.p.wait(5)
            except Exception:
                self.p.kill()
            self.f.close()

    def summary(self):
        if not self.p or not os.path.exists(self.out):
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.out):
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax.append(float(parts[2]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[5:9]):
                if v.lower() == "active":
                    reasons.add(nm)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        return {"sm_mhz": float(np.median(sm)), "sm_max_mhz": float(max(smax)),
                "reasons": sorted(reasons), "samples": len(sm)}


def saturated_state(P, mps, n, chi, seed, device):
    import torch

    import synth
    chis, sites, lams = synth.random_right_canonical_device(n, chi, seed, device=device,
                                                            dtype=torch.complex64)
    lam_arrays = [np.ascontiguousarray(l, dtype=np.float64) for l in lams]
    torch.cuda.synchronize()     # sites are produced on torch's stream; the copy runs on ours
    mps.load_device(chis.astype(np.int32), [s.data_ptr() for s in sites],
                    [l.ctypes.data for l in lam_arrays])
    del sites
    torch.cuda.empty_cache()
    return chis


def profile_rows(P, mps):
    import ctypes as C
    rows = np.zeros(5 * 32)
    nk = C.c_int(0)
    P._check(P.lib.ctebd_profile_read(mps._h, rows.ctypes.data_as(C.POINTER(C.c_double)), 32,
                                      C.byref(nk)), "profile_read")
    out = {}
    for k in range(nk.value):
        buf = C.create_string_buffer(64)
        P.lib.ctebd_kernel_name(k, buf, 64)
        out[buf.value.decode()] = dict(zip(("launches", "ms", "flops", "bytes", "tc_launches"),
                                           rows[5 * k:5 * k + 5]))
    return out


# ---------------------------------------------------------------------------
# plain FP64 GPU comparator: complex128 merge / U / torch.linalg.svd, one
# cluster at a time, no batching, no sketch (the path the target compares to)
# ---------------------------------------------------------------------------
def plain_fp64_update(torch, sites, lams, q0, k, U, chi_max, cutoff):
    dev = next(iter(sites.values())).device
    t = sites[q0].to(torch.complex128)
    for j in range(1, k):
        t = torch.tensordot(t, sites[q0 + j].to(torch.complex128), dims=([t.dim() - 1], [0]))
    cl, cr = t.shape[0], t.shape[-1]
    th = t.reshape(cl, 1 << k, cr)
    Ut = torch.as_tensor(U, dtype=torch.complex128, device=dev)
    th = torch.einsum("st,atb->asb", Ut, th)
    lamL = torch.as_tensor(lams[q0], dtype=torch.float64, device=dev)
    R = th.reshape(-1)
    rdim = cr
    fs = []
    for j in range(k - 1, 0, -1):
        m, n = cl << j, 2 * rdim
        Mb = R.reshape(m, n)
        w = lamL.repeat_interleave(1 << j).to(torch.complex128)
        Usv, S, Vh = torch.linalg.svd(w[:, None] * Mb, full_matrices=False)
        S2 = (S * S).double()
        W = S2.sum()
        tail = torch.flip(torch.cumsum(torch.flip(S2, [0]), 0), [0])
        ok = tail <= cutoff * W
        r = int(torch.nonzero(ok)[0].item()) if bool(ok.any()) else S.numel()
        r = max(1, min(r, chi_max))
        kept = S2[:r].sum()
        fs.append(float(kept / W))
        R = (Mb @ Vh[:r].conj().T / torch.sqrt(kept)).reshape(-1)
        rdim = r
    torch.cuda.synchronize()
    return fs


def method_flops(clusters, chi, log):
    """The method's own work for one iteration, in real flops with 8 per complex
    multiply-add, from the actual shapes: the merge chain (Sec. III.A exact
    contraction), the cluster unitary on the physical index, and per split j
    the randomized truncated SVD of the target design -- sketch and projection
    products 8 m n l each, CholeskyQR2 of Y and of B^H (16 m l^2 + 16 n l^2),
    write-back 8 (m + n) l r -- with sketch width l = min(n, r + 8), no power
    iteration and the O(l^3) small-SVD term left out.  chi: bond dimensions
    before the iteration; log: the iteration's split log (m, n, r in columns
    3-5)."""
    fm = fu = fs = 0.0
    for cl in clusters:
        q0, k = cl.q0, cl.k
        cL, cR = float(chi[q0]), float(chi[q0 + k])
        for j in range(1, k):
            fm += 8.0 * cL * 2 ** j * float(chi[q0 + j]) * 2.0 * float(chi[q0 + j + 1])
        fu += 8.0 * 4.0 ** k * cL * cR
    for row in np.asarray(log).reshape(-1, 14):
        m, n, r = float(row[3]), float(row[4]), float(row[5])
        l = min(n, r + 8.0)
        fs += 2 * 8.0 * m * n * l + 16.0 * m * l * l + 16.0 * n * l * l + 8.0 * (m + n) * l * r
    return fm, fu, fs


class PlainFP64:
    """The plain FP64 GPU cluster update, one cluster at a time: complex128
    merge and unitary with torch, every split a full cuSOLVER SVD
    (torch.linalg.svd) of the Schmidt-weighted matrix, the same truncation rule
    and gauge as the library (right-canonical sites, unweighted remainder,
    renormalised spectra), no batching and no sketch."""

    def __init__(self, torch, sites, lams, device):
        self.t = torch
        self.dev = device
        self.sites = [torch.as_tensor(s, device=device).to(torch.complex128) for s in sites]
        self.lams = [np.asarray(l, dtype=np.float64).copy() for l in lams]
        self.logF = 0.0

    def chi(self):
        return np.array([1] + [int(s.shape[2]) for s in self.sites], dtype=np.int32)

    def apply_1q(self, q, u):
        ut = self.t.as_tensor(u, dtype=self.t.complex128, device=self.dev)
        self.sites[q] = self.t.einsum("st,atb->asb", ut, self.sites[q])

    def update(self, q0, k, U, chi_max, cutoff, floor=1e-13):
        t = self.t
        th = self.sites[q0]
        for j in range(1, k):
            th = t.tensordot(th, self.sites[q0 + j], dims=([th.dim() - 1], [0]))
        cl, cr = th.shape[0], th.shape[-1]
        th = t.einsum("st,atb->asb", t.as_tensor(U, dtype=t.complex128, device=self.dev),
                      th.reshape(cl, 1 << k, cr))
        lamL = t.as_tensor(self.lams[q0], dtype=t.float64, device=self.dev)
        R, rdim, fs = th.reshape(-1), cr, []
        for j in range(k - 1, 0, -1):
            m, n = cl << j, 2 * rdim
            Mb = R.reshape(m, n)
            w = lamL.repeat_interleave(1 << j).to(t.complex128)
            _, S, Vh = t.linalg.svd(w[:, None] * Mb, full_matrices=False)
            s = S.double().cpu().numpy()
            s2 = s * s
            W = float(s2.sum())
            r = len(s)
            if cutoff > 0:
                tail = np.cumsum(s2[::-1])[::-1]
                over = np.nonzero(tail[1:] > cutoff * W)[0]
                r = int(over[-1]) + 2 if len(over) else 1
            r = max(1, min(r, int(np.sum(s > floor * s[0])), chi_max))
            kept = float(s2[:r].sum())
            fs.append(kept / W)
            self.logF += math.log(kept / W)
            self.sites[q0 + j] = Vh[:r].reshape(r, 2, rdim).contiguous()
            self.lams[q0 + j] = s[:r] / math.sqrt(kept)
            R = (Mb @ Vh[:r].conj().T / math.sqrt(kept)).reshape(-1)
            rdim = r
        self.sites[q0] = R.reshape(cl, 2, rdim).contiguous()
        return fs


def mps_overlap(torch, a_sites, b_sites):
    """<a|b> / (|a| |b|) of two MPS given as lists of (chi, 2, chi) tensors."""
    def inner(x, y):
        E = torch.ones((1, 1), dtype=torch.complex128, device=x[0].device)
        for A, B in zip(x, y):
            E = torch.einsum("ab,asc,bsd->cd", E, A.conj(), B)
        return E.reshape(-1)[0]
    ab = inner(a_sites, b_sites)
    return float(abs(ab) / math.sqrt(abs(inner(a_sites, a_sites)) * abs(inner(b_sites, b_sites))))


def run_compare(args):
    """The same iterations three ways from one state: the library's FP32 path
    (batched, tensor cores), the library's FP64 mode (same kernels and
    batching in complex128) and the plain FP64 GPU path
    (PlainFP64).  Workload: the chi_max = 1024 workload's circuit statistics on
    an n-qubit state saturated at chi; every arm runs `steps` iterations after
    one untimed warm-up iteration; device time of the updates with CUDA events.
    Reports updates/s of every arm and the final fidelity products.  With
    --plain-sample 0 the plain path is left out (at chi = 1024 it takes over
    ten seconds per cluster update) and the FP64 mode is the reference arm."""
    import torch

    import paper_2502_19289_gb300 as P
    import synth
    device = "cuda:0"
    w = synth.WORKLOADS[4]
    n, chi, kmax = args.n, args.chi, args.kmax
    q_max = kmax + 2 * int(math.log2(chi))
    c = synth.random_structured(n, w.n_layers, p1=w.p1, p2=w.p2, one_q=w.one_q, two_q=w.two_q, seed=4100)
    circ = P.Circuit(n, c.gates, c.params)
    chis, sites, lams = synth.random_right_canonical(n, chi, seed=4100, dtype=np.complex64)
    stream = torch.cuda.Stream(device=device)
    out = {}
    final_sites = {}

    def iterate(step_fn, chi_fn, one_q_fn, start):
        chi_now = chi_fn()
        clusters, stop = P.cluster_partition(circ.gates, circ.n_gates, start, chi_now, cfgs["fp32"])
        used = set(q for cl in clusters for q in range(cl.q0, cl.q0 + cl.k))
        singles = [(q, P.cluster_unitary(circ.gates, circ.n_gates, P.Cluster(q, 1, start, stop)))
                   for q in range(n) if q not in used]
        one_q_fn(clusters, start, stop, singles)
        Us = [P.cluster_unitary(circ.gates, circ.n_gates, cl) for cl in clusters]
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        with torch.cuda.stream(stream):
            step_fn(clusters, Us)
        e1.record(stream)
        e1.synchronize()
        return stop, len(clusters), e0.elapsed_time(e1) / 1e3

    cfgs = {"fp32": P.make_config(n, chi, w.cutoff, q_max, 0, kmax, P.FP32),
            "fp64": P.make_config(n, chi, w.cutoff, q_max, 0, kmax, P.FP64)}
    arms = ("fp32", "fp64", "plain_fp64") if args.plain_sample > 0 else ("fp32", "fp64")
    for arm in arms:
        if arm == "plain_fp64":
            m = PlainFP64(torch, sites, lams, device)

            def step_fn(clusters, Us, m=m):
                for cl, U in zip(clusters, Us):
                    m.update(cl.q0, cl.k, U, chi, w.cutoff)

            def one_q_fn(clusters, lo, hi, singles, m=m):
                for q, u in singles:
                    m.apply_1q(q, u)
            chi_fn = m.chi
            F = lambda m=m: math.exp(m.logF)
        else:
            m = P.MPS(cfgs[arm], stream.cuda_stream)
            m.load(chis, [s.astype(np.complex128) for s in sites], lams)

            def step_fn(clusters, Us, m=m):
                m.step(clusters, Us)

            def one_q_fn(clusters, lo, hi, singles, m=m):
                m.apply_singletons(circ.gates, circ.n_gates, clusters, lo, hi)
            chi_fn = m.bond_dims
            F = m.fidelity
        start, _, _ = iterate(step_fn, chi_fn, one_q_fn, 0)       # warm-up iteration
        updates, dev_s = 0, 0.0
        for _ in range(args.steps):
            start, nu, dt = iterate(step_fn, chi_fn, one_q_fn, start)
            updates += nu
            dev_s += dt
        out[arm] = {"updates_per_s": updates / dev_s, "updates": updates, "device_s": dev_s,
                    "F_final": F(), "chi_max_reached": int(max(chi_fn()))}
        if arm == "plain_fp64":
            final_sites[arm] = m.sites
        else:
            final_sites[arm] = [torch.as_tensor(m.site(q), device=device) for q in range(n)]
            m.close()
        torch.cuda.empty_cache()
    line = {"metric": "cluster updates/s at equal final fidelity: FP32 tensor-core path vs FP64 paths",
            "unit": "cluster updates/s", "higher_is_better": True, "n_gpus": 1, "dtype": "c64 / c128",
            "data": "synthetic (seeded circuit + random saturated MPS)",
            "config": {"workload": f"n={n}, chi_max={chi} (state saturated at chi), chi_max=1024 workload's "
                                   f"circuit statistics, cutoff 1e-8, k_max={kmax}, Q_max={q_max}; "
                                   f"{args.steps} timed iterations after 1 warm-up, same state for every arm"},
            "arms": out,
            "speedup_fp32_vs_fp64_mode": out["fp32"]["updates_per_s"] / out["fp64"]["updates_per_s"],
            "abs_dF_fp32_vs_fp64_mode": abs(out["fp32"]["F_final"] - out["fp64"]["F_final"]),
            "overlap_fp32_vs_fp64_mode": mps_overlap(torch, final_sites["fp32"], final_sites["fp64"])}
    if "plain_fp64" in out:
        line.update({
            "speedup_fp32_vs_plain": out["fp32"]["updates_per_s"] / out["plain_fp64"]["updates_per_s"],
            "abs_dF_fp32_vs_plain": abs(out["fp32"]["F_final"] - out["plain_fp64"]["F_final"]),
            "abs_dF_fp64_vs_plain": abs(out["fp64"]["F_final"] - out["plain_fp64"]["F_final"]),
            "overlap_fp32_vs_plain": mps_overlap(torch, final_sites["fp32"], final_sites["plain_fp64"]),
            "overlap_fp64_vs_plain": mps_overlap(torch, final_sites["fp64"], final_sites["plain_fp64"])})
    print(json.dumps(line))


def run_apply_traffic(args):
    """Small case for the dominant kernel's DRAM traffic per algorithmic flop:
    one saturated chi = 1024 iteration on n qubits (host-generated state) by the
    Jacobi solver (a sweep cap below the direct solver's, host-driven sweep
    rounds so that every launch is visible to a profiler).
    Prints the eigenproblems of the first eigen-solve and the algorithmic flops
    of its first round update, in which every pair of column blocks rotates:
    one 64^3 complex product per V tile and two per upper G tile.  Captured as

        python bench.py --workload apply-traffic --n 60 &&
        ncu --metrics dram__bytes_read.sum,dram__bytes_write.sum,gpu__time_duration.sum
            --clock-control none -k regex:k_eig_apply_f32 -c 1 --csv
            python bench.py --workload apply-traffic --n 60"""
    import paper_2502_19289_gb300 as P
    import synth
    n = args.n
    if args.tensor_cores is not None:   # 2: the Jacobi round updates on tcgen05 as well
        P.set_tensor_cores(args.tensor_cores)
    w = synth.WORKLOADS[4]
    cfg = P.make_config(n, 1024, w.cutoff, 24, 0, 4, P.FP32)
    c = synth.random_structured(n, w.n_layers, p1=w.p1, p2=w.p2, one_q=w.one_q, two_q=w.two_q, seed=4000)
    circ = P.Circuit(n, c.gates, c.params)
    chis, sites, lams = synth.random_right_canonical(n, 1024, seed=4000, dtype=np.complex64)
    mps = P.MPS(cfg)
    mps.load(chis, sites, lams)
    P.set_sweep_graphs(0)
    P.set_max_sweeps(11)
    clusters, stop = P.cluster_partition(circ.gates, circ.n_gates, 0, mps.bond_dims(), cfg)
    Us = [P.cluster_unitary(circ.gates, circ.n_gates, cl) for cl in clusters]
    widths = [2 * int(chis[cl.q0 + cl.k]) for cl in clusters]   # of the first splits
    try:
        mps.step(clusters, Us)
    except P.CtebdError:   # a solve that needs more sweeps than the cap; the first round is what is captured
        pass
    h = [(n + 63) // 64 for n in widths]   # pairs of 32-wide blocks
    flops = sum(8.0 * 64 ** 3 * (2 * (x * (x + 1) // 2) + x * x) for x in h)
    print(json.dumps({"problems": len(h), "widths": sorted(set(widths)),
                      "first_round_flops": flops, "source_sha256": apply_kernel_digest()}))


def run_bidiag_traffic(args):
    """The same iteration by the direct solver: prints the splits of the first
    level's widest launch class and the algorithmic flops of their
    bidiagonalisation, 16 (m n k - (m + n) k^2 / 2 + k^3 / 3) with k = min(m, n).
    Captured as

        python bench.py --workload bidiag-traffic --n 32 &&
        ncu --metrics dram__bytes_read.sum,dram__bytes_write.sum,gpu__time_duration.sum
            --clock-control none -k regex:k_bidiag -c 1 --csv
            python bench.py --workload bidiag-traffic --n 32"""
    import paper_2502_19289_gb300 as P
    import synth
    n = args.n
    w = synth.WORKLOADS[4]
    cfg = P.make_config(n, 1024, w.cutoff, 24, 0, 4, P.FP32)
    c = synth.random_structured(n, w.n_layers, p1=w.p1, p2=w.p2, one_q=w.one_q, two_q=w.two_q, seed=4000)
    circ = P.Circuit(n, c.gates, c.params)
    chis, sites, lams = synth.random_right_canonical(n, 1024, seed=4000, dtype=np.complex64)
    mps = P.MPS(cfg)
    mps.load(chis, sites, lams)
    clusters, stop = P.cluster_partition(circ.gates, circ.n_gates, 0, mps.bond_dims(), cfg)
    mps.step(clusters, [P.cluster_unitary(circ.gates, circ.n_gates, cl) for cl in clusters])
    level1 = [(int(r[3]), int(r[4])) for r in mps.split_log() if int(r[2]) == int(r[0]) + int(r[1]) - 1]
    wide = [(a, b) for a, b in level1 if 1024 < b <= 2048]
    flops = sum(16.0 * (a * b * min(a, b) - (a + b) * min(a, b) ** 2 / 2 + min(a, b) ** 3 / 3) for a, b in wide)
    print(json.dumps({"splits": wide, "flops": flops, "source_sha256": bidiag_kernel_digest()}))


def run_cfg5(args):
    """cfg5: independent random-structured Clifford+T circuits (n ~ U[50, 300],
    layers ~ U[40, 100], T density ~ U[5%, 25%] of the one-qubit gates,
    CNOT/CZ on nearest-neighbour bonds with p = 0.3), chi_max = 1024, cutoff
    1e-8, k_max = 4, from |0...0>.  All circuits are packed side by side on one
    MPS and advance together: every iteration steps the clusters of all
    unfinished circuits in the same batched launches (FP32 path).  Timed: the
    whole packed simulation, wall clock (host partition included).  Then every
    circuit runs alone in the library's FP64 mode, and its final bond
    dimensions, fidelity product and state are compared with its slice of the
    packed run."""
    import torch

    import paper_2502_19289_gb300 as P
    import synth
    rng = np.random.default_rng(5000)
    circs, spec = [], []
    for i in range(args.circuits):
        n = int(rng.integers(50, 301))
        layers = int(rng.integers(40, 101))
        t = float(rng.uniform(0.05, 0.25))
        circs.append(synth.random_structured(n, layers, p1=0.5, p2=0.3,
                                             one_q={synth.T: t, synth.H: (1 - t) / 2, synth.S: (1 - t) / 2},
                                             two_q=(synth.CNOT, synth.CZ), seed=5000 + i))
        spec.append((n, layers, t))
    k_max, chi, cut = 4, 1024, 1e-8
    q_max = k_max + 2 * 10
    stream = torch.cuda.Stream()
    packed = [(c.n_qubits, c.gates, c.params) for c in circs]
    cfg = P.make_config(1, chi, cut, q_max, 0, k_max, P.FP32)
    warm, _ = P.simulate_packed(packed[:2], cfg, stream.cuda_stream)   # untimed: first launches
    warm.close()
    counts = {"updates": 0, "iterations": 0}

    def count(cl):
        counts["updates"] += len(cl)
        counts["iterations"] += 1

    torch.cuda.synchronize()
    t0 = time.perf_counter()
    mps, pk = P.simulate_packed(packed, cfg, stream.cuda_stream, callback=count)
    stream.synchronize()
    wall = time.perf_counter() - t0
    chis = mps.bond_dims()
    logF_packed = float(math.log(mps.fidelity()))
    rows, logF_sum = [], 0.0
    t64 = 0.0
    for c, off in zip(circs, pk.offsets):
        n = c.n_qubits
        cfg64 = P.make_config(n, chi, cut, q_max, 0, k_max, P.FP64)
        a = time.perf_counter()
        ref = P.simulate(P.Circuit(n, c.gates, c.params), cfg64, stream.cuda_stream)
        t64 += time.perf_counter() - a
        lf64 = float(math.log(ref.fidelity()))
        logF_sum += lf64
        prof64 = [int(x) for x in ref.bond_dims()]
        prof32 = [int(x) for x in chis[off:off + n + 1]]
        a_sites = [torch.as_tensor(mps.site(off + q)).to(torch.complex128) for q in range(n)]
        b_sites = [torch.as_tensor(ref.site(q)).to(torch.complex128) for q in range(n)]
        ov = mps_overlap(torch, a_sites, b_sites)
        rows.append({"n": n, "max_chi": max(prof64), "chi_profile_equal": prof32 == prof64, "logF_fp64": lf64,
                     "overlap": ov})
        ref.close()
    mps.close()
    d_logF = abs(logF_packed - logF_sum)
    line = {"metric": "cluster updates/s, packed circuits (cfg5) vs each circuit's FP64-mode run",
            "value": counts["updates"] / wall, "unit": "cluster updates/s", "higher_is_better": True,
            "n_gpus": 1, "dtype": "c64", "data": "synthetic (seeded circuits from |0...0>)",
            "config": {"workload": f"cfg5: {args.circuits} Clifford+T circuits, n ~ U[50, 300] "
                                   f"(total {sum(x[0] for x in spec)} qubits), layers ~ U[40, 100], "
                                   "T density ~ U[5%, 25%], chi_max=1024, cutoff 1e-8, k_max=4, packed per step",
                       "timing": "wall clock of the whole packed simulation, host partition included"},
            "updates": counts["updates"], "iterations": counts["iterations"], "wall_s": wall,
            "fp64_mode_alone_s": t64, "fp64_updates_per_s": counts["updates"] / t64,
            "agreement": {"circuits": len(rows),
                          "chi_profiles_equal": int(sum(r["chi_profile_equal"] for r in rows)),
                          "min_overlap": min(r["overlap"] for r in rows),
                          "abs_dlogF_total": d_logF,
                          "max_chi": max(r["max_chi"] for r in rows),
                          "truncated_circuits": int(sum(r["logF_fp64"] < -1e-6 for r in rows))},
            "circuits": rows}
    print(json.dumps(line))


def run_latency(args):
    """Where latency dominates: cfg1 (n=12, exact, FP64), cfg3's gate
    statistics at n=40 (Clifford, chi_max 512, cutoff 1e-12) and cfg2's at
    n=100 over 20 layers, each from |0...0> through the whole circuit.  Per
    configuration: the wall time of the step calls, and the summed device time
    of the library's kernels in a second, identical run with per-launch CUDA
    events.  Their ratio is the fraction of the step the GPU is busy; the rest
    is host work, launch gaps and the per-level reads, the most that capturing
    a whole step into one graph could remove."""
    import torch

    import paper_2502_19289_gb300 as P
    import synth

    def run(w, base, profile):
        n, chi = w.n_qubits, w.chi_max
        q_max = w.k_max + 2 * int(math.log2(chi))
        prec = P.FP64 if w.precision == "fp64" else P.FP32
        cfg = P.make_config(n, chi, w.cutoff, q_max, 0, w.k_max, prec)
        c = w.circuit(0, base)
        circ = P.Circuit(n, c.gates, c.params)
        stream = torch.cuda.Stream()
        mps = P.MPS(cfg, stream.cuda_stream)
        if profile:
            P._check(P.lib.ctebd_profile(mps._h, 1), "ctebd_profile")
        start, steps, upd, t_step = 0, 0, 0, 0.0
        torch.cuda.synchronize()
        while start < circ.n_layers:
            cl, stop = P.cluster_partition(circ.gates, circ.n_gates, start, mps.bond_dims(), cfg)
            mps.apply_singletons(circ.gates, circ.n_gates, cl, start, stop)
            if cl:
                Us = [P.cluster_unitary(circ.gates, circ.n_gates, x) for x in cl]
                t0 = time.perf_counter()
                mps.step(cl, Us)
                t_step += time.perf_counter() - t0
                steps += 1
                upd += len(cl)
            start = stop
        out = {"steps": steps, "updates": upd, "step_wall_s": t_step, "max_chi": int(max(mps.bond_dims())),
               "logF": float(math.log(mps.fidelity()))}
        if profile:
            cls = profile_rows(P, mps)
            out["kernel_ms"] = float(sum(v["ms"] for v in cls.values()))
            out["launches"] = int(sum(v["launches"] for v in cls.values()))
            out["classes"] = cls
        mps.close()
        return out

    res = {}
    for name, base, w in (("cfg1: n=12, 10 layers, exact, FP64", 1, synth.WORKLOADS[1]),
                          ("cfg3 statistics: n=40, 100 layers, Clifford, chi_max 512", 3, synth.reduced(3, 40, 100)),
                          ("cfg2 statistics: n=100, 20 layers", 2, synth.reduced(2, 100, 20))):
        run(w, base, False)   # warm-up
        plain = run(w, base, False)
        prof = run(w, base, True)
        ns = max(prof["steps"], 1)
        top = sorted(prof["classes"].items(), key=lambda kv: -kv[1]["ms"])[:5]
        res[name] = {"updates_per_s": plain["updates"] / plain["step_wall_s"], "steps": plain["steps"],
                     "step_ms": 1e3 * plain["step_wall_s"] / max(plain["steps"], 1),
                     "kernel_ms_per_step": prof["kernel_ms"] / ns,
                     "kernel_ms_per_step_by_class": {k: round(v["ms"] / ns, 4) for k, v in top},
                     "launches_per_step": prof["launches"] / ns,
                     "gpu_busy_frac": prof["kernel_ms"] / 1e3 / plain["step_wall_s"],
                     "max_chi": plain["max_chi"]}
    print(json.dumps({"metric": "GPU-busy fraction of the step on latency-bound configurations",
                      "unit": "fraction", "n_gpus": 1, "data": "synthetic (seeded circuits from |0...0>)",
                      "configs": res}))


def run_tebd(args):
    """Cluster-TEBD against standard TEBD on the same circuits (Sec. IV.B,
    Figs. 8-9).  Random-structured circuits from the paper's generator
    (Sec. IV.A: every slot filled, a two-qubit gate with p = 0.5), with the
    Clifford and the non-Clifford gate sets of App. A, run from |0...0>
    through the whole circuit at one chi_max in the FP32 path.  Standard TEBD
    is the special case of one layer per iteration and two-qubit clusters
    (L_max = 1, k_max = 2).  Cluster-TEBD contracts as many layers per
    iteration as its clusters allow under the memory bound (Eq. 7), with
    Q_max = 3 + 2 log2 chi_max: the paper's runs at chi_max = 4096 used
    Q_max = 27, the same three qubits of headroom between two saturated
    bonds.  Clusters are also capped at k_max qubits (default 8), because
    every cluster unitary is built as a dense 2^k x 2^k matrix.  Per
    circuit: the wall time of each whole run (host partition and cluster
    unitaries included), their ratio, and each run's fidelity product."""
    import torch

    import paper_2502_19289_gb300 as P
    import synth
    chi, k_max, cut = args.chi, args.kmax, 1e-8
    lg = int(math.log2(chi))
    stream = torch.cuda.Stream()

    def run(c, cluster):
        n = c.n_qubits
        cfg = (P.make_config(n, chi, cut, 3 + 2 * lg, 0, k_max, P.FP32) if cluster else
               P.make_config(n, chi, cut, 2 + 2 * lg, 1, 2, P.FP32))
        circ = P.Circuit(n, c.gates, c.params)
        counts = [0, 0]

        def count(s, e, cl, f):
            counts[0] += 1
            counts[1] += len(cl)

        torch.cuda.synchronize()
        t0 = time.perf_counter()
        mps = P.simulate(circ, cfg, stream.cuda_stream, callback=count)
        stream.synchronize()
        wall = time.perf_counter() - t0
        out = {"s": wall, "F": float(mps.fidelity()), "iterations": counts[0], "updates": counts[1],
               "max_chi": int(max(mps.bond_dims())), "layers": circ.n_layers}
        mps.close()
        return out

    warm = synth.paper_random_structured(12, 10, clifford=False, seed=1)
    run(warm, True)    # untimed: first launches, graph and kernel setup
    run(warm, False)
    rows = []
    for clifford in (True, False):
        for n, layers in ((40, 40), (40, 80), (100, 40), (100, 80)):
            c = synth.paper_random_structured(n, layers, clifford=clifford,
                                              seed=9000 + n + layers + (0 if clifford else 500))
            t = run(c, False)
            ct = run(c, True)
            rows.append({"gates": "Clifford" if clifford else "non-Clifford", "n": n, "layers": t["layers"],
                         "tebd_s": t["s"], "ctebd_s": ct["s"], "speedup": t["s"] / ct["s"],
                         "F_tebd": t["F"], "F_ctebd": ct["F"], "iterations": [t["iterations"], ct["iterations"]],
                         "updates": [t["updates"], ct["updates"]], "max_chi": [t["max_chi"], ct["max_chi"]]})
    summary = {g: {"min": min(r["speedup"] for r in rows if r["gates"] == g),
                   "max": max(r["speedup"] for r in rows if r["gates"] == g)}
               for g in ("Clifford", "non-Clifford")}
    print(json.dumps({"metric": "cluster-TEBD speed-up over standard TEBD (wall-time ratio, same circuit)",
                      "unit": "x", "higher_is_better": True, "n_gpus": 1, "dtype": "c64",
                      "data": "synthetic (the paper's random-structured generator, seeded; from |0...0>)",
                      "config": {"workload": f"paper generator, Clifford and non-Clifford sets, n in (40, 100), "
                                             f"40 and 80 layers, chi_max={chi}, cutoff 1e-8; cluster-TEBD "
                                             f"k_max={k_max}, Q_max={3 + 2 * lg}; standard TEBD L_max=1, "
                                             "k_max=2",
                                 "timing": "wall clock of each whole simulation"},
                      "speedup": summary, "circuits": rows}))


def run_shor(args):
    """Cluster-TEBD against standard TEBD on Shor's order-finding circuit
    (Sec. IV.B, Fig. 10): Beauregard's construction for N with base a, t
    counting qubits (default: the phase-estimation size for the precision the
    paper used for that N), every long-range gate routed through
    nearest-neighbour SWAPs.  Both modes run from |0...0> through the whole
    circuit in the FP32 path; standard TEBD is L_max = 1, k_max = 2, and
    cluster-TEBD takes Q_max = 3 + 2 log2 chi_max with clusters of at most
    k_max qubits (default 8).  For t <= 10 and at most 24 qubits, the counting
    register's distribution from each final state is compared with its closed
    form, sum_z |2^-t sum_{C : a^C = z mod N} exp(-2 pi i y C / 2^t)|^2."""
    import torch

    import paper_2502_19289_gb300 as P
    from synth.shor import counting_qubits, shor_build, shor_circuit
    eps = {15: 1e-3, 21: 1e-4, 35: 1e-5, 91: 1e-5, 221: 1e-9}
    N, a = args.shor_n, args.shor_a
    t = args.shor_t if args.shor_t > 0 else counting_qubits(N, eps.get(N, 1e-3))
    chi, k_max, cut = args.chi, args.kmax, 1e-8
    lg = int(math.log2(chi))
    c, regs = shor_build(N, a, t, routing=args.shor_routing)
    cpos = regs["c"]   # chain position of counting qubit c_j
    n = c.n_qubits
    circ = P.Circuit(n, c.gates, c.params)
    stream = torch.cuda.Stream()

    def run(circuit, nq, cluster):
        cfg = (P.make_config(nq, chi, cut, 3 + 2 * lg, 0, k_max, P.FP32) if cluster else
               P.make_config(nq, chi, cut, 2 + 2 * lg, 1, 2, P.FP32))
        counts = [0, 0]

        def count(s, e, cl, f):
            counts[0] += 1
            counts[1] += len(cl)

        torch.cuda.synchronize()
        t0 = time.perf_counter()
        mps = P.simulate(circuit, cfg, stream.cuda_stream, callback=count)
        stream.synchronize()
        return mps, {"s": time.perf_counter() - t0, "F": float(mps.fidelity()), "iterations": counts[0],
                     "updates": counts[1], "max_chi": int(max(mps.bond_dims()))}

    def counting_error(mps):
        if t > 10 or n > 24:
            return None
        v = np.ones((1, 1), dtype=np.complex128)
        for q in range(n):
            s = mps.site(q)
            v = np.einsum("ia,asb->isb", v, s).reshape(-1, s.shape[2])
        p = np.abs(v.reshape((2,) * n)) ** 2
        pc = p.sum(axis=tuple(i for i in range(n) if i not in cpos))   # axes in chain order
        axes = sorted(cpos)
        got = np.zeros(1 << t)
        for idx in np.ndindex(*(2,) * t):
            bit = dict(zip(axes, idx))
            got[sum(bit[cpos[t - 1 - k]] << k for k in range(t))] += pc[idx]
        C = np.arange(1 << t)
        z = np.array([pow(a, int(k), N) for k in C])
        ref = np.array([sum(abs(np.exp(-2j * np.pi * y * C[z == u] / (1 << t)).sum() / (1 << t)) ** 2
                            for u in np.unique(z)) for y in range(1 << t)])
        return float(np.max(np.abs(got / got.sum() - ref)))

    warm = shor_circuit(15, 2, 1)
    for cl in (True, False):   # untimed: first launches, graph and kernel setup
        m, _ = run(P.Circuit(warm.n_qubits, warm.gates, warm.params), warm.n_qubits, cl)
        m.close()
    out = {}
    for name, cl in (("tebd", False), ("cluster_tebd", True)):
        m, r = run(circ, n, cl)
        r["counting_register_max_abs_error"] = counting_error(m)
        m.close()
        out[name] = r
    print(json.dumps({"metric": "cluster-TEBD speed-up over standard TEBD on Shor's circuit (wall-time ratio)",
                      "value": out["tebd"]["s"] / out["cluster_tebd"]["s"], "unit": "x",
                      "higher_is_better": True, "n_gpus": 1, "dtype": "c64",
                      "data": "synthetic (Beauregard's order-finding circuit, SWAP-routed; from |0...0>)",
                      "config": {"workload": f"Shor order finding N={N}, a={a}, t={t} counting qubits, {n} qubits, "
                                             f"{args.shor_routing} routing, "
                                             f"{circ.n_gates} gates in {circ.n_layers} layers; chi_max={chi}, cutoff "
                                             f"1e-8; cluster-TEBD k_max={k_max}, Q_max={3 + 2 * lg}; standard TEBD "
                                             "L_max=1, k_max=2",
                                 "timing": "wall clock of each whole simulation"},
                      "qubits": n, "gates": circ.n_gates, "layers": circ.n_layers, "arms": out}))


def aggregate(dev_s: float, wall_s: float, units: int, device=None):
    """Whole-job figures over all ranks: max of the times, sum of the units.

    Replicas share nothing on the data path; this is the only collective."""
    import torch
    import torch.distributed as dist
    if not (dist.is_available() and dist.is_initialized()) or dist.get_world_size() == 1:
        return dev_s, wall_s, units
    t = torch.tensor([dev_s, wall_s], dtype=torch.float64, device=device)
    u = torch.tensor([float(units)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    dist.all_reduce(u, op=dist.ReduceOp.SUM)
    return float(t[0]), float(t[1]), int(round(float(u[0])))


def run_ours(args, rank, world, local_rank):
    import torch

    import paper_2502_19289_gb300 as P
    import synth

    torch.cuda.set_device(local_rank)
    device = f"cuda:{local_rank}"
    stream = torch.cuda.Stream(device=device)
    if args.tensor_cores is not None:
        P.set_tensor_cores(args.tensor_cores)
    w = synth.WORKLOADS[4]
    n, chi, kmax = args.n, args.chi, args.kmax
    q_max = kmax + 2 * int(math.log2(chi))
    cfg = P.make_config(n, chi, w.cutoff, q_max, 0, kmax, P.FP32, seed=4000 + rank)
    c = synth.random_structured(n, w.n_layers, p1=w.p1, p2=w.p2, one_q=w.one_q, two_q=w.two_q,
                                seed=4000 + rank)
    circ = P.Circuit(n, c.gates, c.params)
    mps = P.MPS(cfg, stream.cuda_stream)
    saturated_state(P, mps, n, chi, seed=4000 + rank, device=device)

    start = 0
    totals = {"updates": 0, "dev_ms": 0.0, "wall_s": 0.0, "h2d": 0, "d2h": 0, "flops": 0.0,
              "f_merge": 0.0, "f_u": 0.0, "f_split": 0.0}
    step_f = []
    sweeps = []   # Jacobi sweeps (pass 1, pass 2) of every split of the timed steps

    def one_step(timed):
        nonlocal start
        if start >= circ.n_layers:
            start = 0
        t0 = time.perf_counter()
        chi_now = mps.bond_dims()
        clusters, stop = P.cluster_partition(circ.gates, circ.n_gates, start, chi_now, cfg)
        mps.apply_singletons(circ.gates, circ.n_gates, clusters, start, stop)
        Us = [P.cluster_unitary(circ.gates, circ.n_gates, cl) for cl in clusters]
        ev0 = torch.cuda.Event(enable_timing=True)
        ev1 = torch.cuda.Event(enable_timing=True)
        ev0.record(stream)
        f = mps.step(clusters, Us)
        ev1.record(stream)
        chi_after = mps.bond_dims()          # device->host result read (bond dims, f)
        ev1.synchronize()
        t1 = time.perf_counter()
        if timed:
            totals["updates"] += len(clusters)
            totals["dev_ms"] += ev0.elapsed_time(ev1)
            totals["wall_s"] += t1 - t0
            totals["h2d"] += sum(16 * U.size for U in Us)
            totals["d2h"] += 8 * len(f) + 4 * len(chi_after)
            log = mps.split_log()
            fm, fu, fs = method_flops(clusters, chi_now, log)
            if len(log):
                sweeps.append(log[:, 12:14])
            totals["f_merge"] += fm
            totals["f_u"] += fu
            totals["f_split"] += fs
            step_f.append((len(clusters), sum(cl.k for cl in clusters), float(np.prod(f))))
        start = stop
        return clusters, Us

    for _ in range(args.warmup):
        one_step(False)
    torch.cuda.synchronize()
    if world > 1:
        import torch.distributed as dist
        dist.barrier()
    # timed region: the library's default path, no per-launch events; its launch
    # and flop counters still accumulate
    P._check(P.lib.ctebd_profile(mps._h, 0), "profile")
    with Clocks(local_rank) as clk:
        for _ in range(args.steps):
            one_step(True)
        torch.cuda.synchronize()
    counts = profile_rows(P, mps)
    # one more iteration with per-launch CUDA events: kernel times and shares
    P._check(P.lib.ctebd_profile(mps._h, 1), "profile")
    one_step(False)
    torch.cuda.synchronize()
    prof = profile_rows(P, mps)
    P._check(P.lib.ctebd_profile(mps._h, 0), "profile")
    res = dict(totals)
    res["prof"] = prof
    res["counts"] = counts
    res["clocks"] = clk.summary()
    res["steps_detail"] = step_f
    sw = np.concatenate(sweeps) if sweeps else np.zeros((0, 2))
    capped, capped_moved = mps.solver_stats()
    direct = int((sw[:, 0] == 0).sum())   # direct and narrow splits make no sweeps
    sw = sw[sw[:, 0] > 0]
    res["jacobi_sweeps"] = {"splits": int(len(sw)), "splits_without_jacobi": direct, "cap": P.max_sweeps(),
                            "refinements_accepted_at_cap": capped, "their_max_moved_rel": capped_moved,
                            "pass1_mean": float(sw[:, 0].mean()) if len(sw) else 0.0,
                            "pass1_max": int(sw[:, 0].max()) if len(sw) else 0,
                            "pass2_mean": float(sw[:, 1].mean()) if len(sw) else 0.0,
                            "pass2_max": int(sw[:, 1].max()) if len(sw) else 0} if len(sw) else None
    res["peaks"] = measure_compute_peaks(P, torch, device)

    # plain FP64 comparator on a sample of the next iteration's clusters
    if rank == 0 and args.plain_sample > 0:
      try:
            chi_now = mps.bond_dims()
            clusters, stop = P.cluster_partition(circ.gates, circ.n_gates, start, chi_now, cfg)
            big = sorted(clusters, key=lambda c: -(int(chi_now[c.q0]) * int(chi_now[c.q0 + c.k]) << c.k))
            sample = sorted(big[: args.plain_sample], key=lambda c: c.q0)
            sites = [torch.as_tensor(mps.site(q), device=device) for q in
                     sorted({cl.q0 + j for cl in sample for j in range(cl.k)})]
            idx = sorted({cl.q0 + j for cl in sample for j in range(cl.k)})
            smap = {q: s for q, s in zip(idx, sites)}
            lams = {cl.q0: mps.lam(cl.q0) for cl in sample}
            Us = [P.cluster_unitary(circ.gates, circ.n_gates, cl) for cl in sample]
            t0 = time.perf_counter()
            fplain = []
            for cl, U in zip(sample, Us):
                fplain.append(plain_fp64_update(torch, smap, lams, cl.q0, cl.k, U, chi, w.cutoff))
            t_plain = time.perf_counter() - t0
            # ours on exactly the same sample, one launch batch
            t0 = time.perf_counter()
            fours = mps.step(sample, Us)
            torch.cuda.synchronize()
            t_ours = time.perf_counter() - t0
            fp = np.concatenate([np.array(x) for x in fplain])
            res["plain"] = {"updates": len(sample), "s": t_plain, "ours_s": t_ours,
                            "max_abs_df": float(np.max(np.abs(fp - np.asarray(fours)))) if len(fp) == len(fours) else None,
                            "F_plain": float(np.prod(fp)), "F_ours": float(np.prod(fours))}
      except Exception as e:  # the comparator must not hide the main measurement
        res["plain"] = {"error": repr(e)}
    return res


def _oracle_worker(args):
    """One host process: single-threaded oracle cluster updates of the chi_max =
    1024 workload's circuit over a reduced-chi synthetic saturated state, for
    about `seconds`.  Imports only the oracle and the input generators."""
    chi, nsites, seconds, seed = args
    if ROOT not in sys.path:
        sys.path.insert(0, ROOT)
    import oracle
    import synth
    w = synth.WORKLOADS[4]
    c = synth.random_structured(nsites, w.n_layers, p1=w.p1, p2=w.p2, one_q=w.one_q,
                                two_q=w.two_q, seed=4000)
    layer, nl = oracle.asap_layers(nsites, c.gates)
    chis, sites, lams = synth.random_right_canonical(nsites, chi, seed=seed)
    m = oracle.MPS.from_arrays(sites, lams)
    q_max = w.k_max + 2 * int(math.log2(chi))
    done, t0, start = 0, time.perf_counter(), 0
    while time.perf_counter() - t0 < seconds:
        if start >= nl:
            start = 0
        clusters, stop = oracle.partition(nsites, c.gates, layer, nl, start, m.chi(), q_max, 0, w.k_max)
        for q0, k in clusters:
            U = oracle.cluster_unitary(q0, k, c, layer, start, stop)
            m.cluster_update(q0, k, U, chi, w.cutoff)
            done += 1
            if time.perf_counter() - t0 >= seconds:
                break
        start = stop
    return done, time.perf_counter() - t0


def host_cores() -> int:
    try:
        return len(os.sched_getaffinity(0))
    except Exception:
        return os.cpu_count() or 1


def cpu_baseline(seconds=12.0, chi=128, nsites=16, workers=None):
    """The FP64 CPU oracle, as it stands, on all host cores: one spawned
    process per core, each running single-threaded cluster updates of the
    chi_max = 1024 workload's circuit on a 16-qubit chi = 128 synthetic
    saturated state (chi = 1024 oracle updates take about an hour each).  The
    per-update cost grows as chi^3 (merge and SVD), so the chi = 1024 rate is
    reported as the measured rate x (128/1024)^3, labelled as extrapolated."""
    import concurrent.futures as cf
    import multiprocessing as mp
    workers = workers or host_cores()
    ctx = mp.get_context("spawn")
    # one thread per process: the oracle is single-threaded and numpy's BLAS
    # pool would otherwise put cores x cores threads on the host
    saved = {k: os.environ.get(k) for k in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS")}
    os.environ.update({k: "1" for k in saved})
    try:
        with cf.ProcessPoolExecutor(max_workers=workers, mp_context=ctx) as ex:
            res = list(ex.map(_oracle_worker, [(chi, nsites, seconds, 4000 + i) for i in range(workers)]))
    finally:
        for k, v in saved.items():
            if v is None:
                os.environ.pop(k, None)
            else:
                os.environ[k] = v
    done = sum(r[0] for r in res)
    rate = sum(r[0] / r[1] for r in res)          # processes run side by side
    ext = rate * (chi / 1024.0) ** 3
    return {"value": ext, "unit": UNIT, "cores": workers, "kind": "oracle",
            "value_basis": f"extrapolated to chi=1024 from the measured chi={chi} rate x ({chi}/1024)^3",
            "measured_value": rate, "measured_chi": chi, "per_core_measured": rate / workers,
            "sample": f"{done} cluster updates (k=2..4) of the chi_max=1024 workload's circuit (cfg4 gate "
                      f"statistics) on a {nsites}-qubit chi={chi} synthetic saturated state, FP64 oracle, "
                      f"{workers} single-threaded processes x {seconds:.0f} s"}


def run_cfg2(args):
    """Sketched split (randomized range finder + CholeskyQR + Rayleigh-Ritz, with
    the tail check) against the full split, from |0...0> through the circuit.

    ``--workload cfg2``: n=100, 50 layers of random-structured Clifford+T (10% T,
    10% long-range pairs), chi_max=256, cutoff 1e-10, k_max=6.
    ``--workload sketch-cfg4``: the cfg4 gate statistics (20% T, chi_max=1024,
    cutoff 1e-8, k_max=4) on ``--n`` qubits (default 100) for ``--layers``
    layers (default 30): the growing phase, where the bonds climb to chi_max.
    Three modes: full split; sketch sized by the Eq. 9 bound; sketch sized by
    the learned rank predictor (trained in the same run on six smaller circuits
    of the same gate statistics).  Device time of the cluster updates (CUDA
    events on the library's stream) and wall time; the modes must agree on log
    F and the bond dimensions."""
    import torch

    import paper_2502_19289_gb300 as P
    import paper_2502_19289_gb300.rank_model as R
    import synth
    base = 4 if args.workload == "sketch-cfg4" else 2
    w = synth.WORKLOADS[base]
    if base == 4:
        w = synth.reduced(4, args.n, args.layers or 30)
    elif args.layers:   # same gate statistics, deeper circuit (bonds grow towards chi_max)
        w = synth.reduced(2, w.n_qubits, args.layers)
    n, chi, over = w.n_qubits, w.chi_max, 8
    q_max = w.k_max + 2 * int(math.log2(chi))
    c = w.circuit(0, base)
    stream = torch.cuda.Stream()

    t0 = time.perf_counter()
    small = synth.reduced(base, 40, 60 if base == 2 else 22)
    Xs, rs, bs = [], [], []
    for seed in range(1, 7):
        cc = small.circuit(seed, base)
        X, r, b = R.collect((cc.gates, cc.params), small.n_qubits, chi, w.cutoff, q_max, w.k_max,
                            stream.cuda_stream)
        Xs.append(X); rs.append(r); bs.append(b)
    X, r, b = np.concatenate(Xs), np.concatenate(rs), np.concatenate(bs)
    params, hist = R.train(X, R.bucket_of(r, b), epochs=150, lr=3e-3, batch=256, seed=0)
    train_s = time.perf_counter() - t0

    def run(oversample, learned):
        circ = P.Circuit(n, c.gates, c.params)
        cfg = P.make_config(n, chi, w.cutoff, q_max, 0, w.k_max, P.FP32, sketch_oversample=oversample)
        mps = P.MPS(cfg, stream.cuda_stream)
        hint = R.make_hint_fn(mps, circ, cfg, params) if learned else None
        start, updates, dev_ms, work, splits = 0, 0, 0.0, 0.0, 0
        torch.cuda.synchronize()
        w0 = time.perf_counter()
        while start < circ.n_layers:
            chi_now = mps.bond_dims()
            clusters, stop = P.cluster_partition(circ.gates, circ.n_gates, start, chi_now, cfg)
            if oversample > 0 and clusters:
                hints = (hint(clusters, chi_now) if hint else
                         [P.cluster_rank_bounds(circ.gates, circ.n_gates, cl, chi_now) for cl in clusters])
                for cl, h in zip(clusters, hints):
                    for j, v in enumerate(h[:11]):
                        cl.rank_hint[j] = int(v)
            mps.apply_singletons(circ.gates, circ.n_gates, clusters, start, stop)
            if clusters:
                Us = [P.cluster_unitary(circ.gates, circ.n_gates, cl) for cl in clusters]
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record(stream)
                mps.step(clusters, Us)
                e1.record(stream)
                e1.synchronize()
                dev_ms += e0.elapsed_time(e1)
                updates += len(clusters)
                log = mps.split_log()
                work += float(np.sum(log[:, 9] ** 3))
                splits += len(log)
            start = stop
        wall = time.perf_counter() - w0
        sk, fb = mps.sketch_stats()
        out = {"updates_per_s": updates / (dev_ms / 1000.0), "e2e_updates_per_s": updates / wall,
               "updates": updates, "device_s": dev_ms / 1000.0, "logF": float(math.log(mps.fidelity())),
               "splits": splits, "sketched": sk, "fell_back": fb, "eigen_work_sum_ne3": work,
               "max_chi": int(max(mps.bond_dims())), "wall_s": wall}
        dims = list(mps.bond_dims())
        mps.close()
        return out, dims

    full, d_full = run(0, False)
    eq9, d_eq9 = run(over, False)
    learned, d_l = run(over, True)
    if base == 4:
        desc = (f"cfg4 gate statistics from |0...0>: n={n}, {w.n_layers}-layer random-structured Clifford+T "
                f"(20% T), chi_max=1024, cutoff 1e-8, k_max=4, Q_max={q_max}, sketch oversampling 8")
        trained = f"trained on 6 cfg4-shaped circuits (n=40, 22 layers)"
    else:
        desc = (f"cfg2: n=100, {w.n_layers}-layer random-structured Clifford+T (10% T, 10% long-range pairs), "
                f"chi_max=256, cutoff 1e-10, k_max=6, Q_max={q_max}, sketch oversampling 8")
        trained = "trained on 6 cfg2-shaped circuits (n=40, 60 layers)"
    line = {"metric": f"cluster updates/s, {'cfg4 growing phase' if base == 4 else 'cfg2 workload'}: "
                      "full split vs sketched split (Eq. 9 and learned sizes)",
            "unit": "cluster updates/s", "higher_is_better": True, "n_gpus": 1, "dtype": "c64",
            "data": "synthetic (seeded circuit from |0...0>)",
            "config": {"workload": desc,
                       "rank_model": f"{trained}, {len(X)} splits, "
                                     f"loss {hist[0]:.3f} -> {hist[-1]:.3f}, {train_s:.1f} s"},
            "modes": {"full": full, "sketch_eq9": eq9, "sketch_learned": learned},
            "speedup_eq9": eq9["updates_per_s"] / full["updates_per_s"],
            "speedup_learned": learned["updates_per_s"] / full["updates_per_s"],
            "wall_speedup_eq9": full["wall_s"] / eq9["wall_s"],
            "wall_speedup_learned": full["wall_s"] / learned["wall_s"],
            "agreement": {"max_abs_dlogF": max(abs(eq9["logF"] - full["logF"]),
                                              abs(learned["logF"] - full["logF"])),
                          "bond_dims_equal": d_full == d_eq9 == d_l}}
    print(json.dumps(line))


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--n", type=int, default=None,
                    help="qubits (default: 500 for cfg4, 60 for compare, 24 for apply-traffic, 100 for sketch-cfg4)")
    ap.add_argument("--chi", type=int, default=None, help="chi_max (default: 256 for tebd, else 1024)")
    ap.add_argument("--kmax", type=int, default=None,
                    help="largest cluster (default 8 for tebd, with Q_max = 3 + 2 log2 chi; else 4, "
                         "with Q_max = kmax + 2 log2 chi: 6 lets k = 3..6 clusters form)")
    ap.add_argument("--plain-sample", type=int, default=2)
    ap.add_argument("--cpu-seconds", type=float, default=12.0)
    ap.add_argument("--workload", default="cfg4", choices=["cfg4", "cfg2", "sketch-cfg4", "cfg5", "compare", "apply-traffic",
                             "bidiag-traffic", "latency", "tebd", "shor"],
                    help="cfg4: the headline (saturated chi=1024, full split); cfg2, sketch-cfg4: full vs "
                         "sketched split (cfg2, and cfg4's growing phase); "
                         "compare: FP32 path, FP64 mode and the plain FP64 path over the same iterations; "
                         "apply-traffic, bidiag-traffic: small cases for the round update's and the "
                         "bidiagonalisation's DRAM traffic; latency: GPU-busy "
                         "fraction of the step on small configurations; cfg5: packed circuits, each "
                         "checked against its FP64-mode run; tebd: cluster-TEBD against standard "
                         "TEBD on the paper's generator; shor: the same on Shor's order-finding circuit")
    ap.add_argument("--circuits", type=int, default=64, help="cfg5: number of packed circuits")
    ap.add_argument("--shor-n", type=int, default=15, help="shor: the number to factor")
    ap.add_argument("--shor-a", type=int, default=2, help="shor: the base (coprime with N)")
    ap.add_argument("--shor-t", type=int, default=0,
                    help="shor: counting qubits (default: phase-estimation size for the paper's precision)")
    ap.add_argument("--shor-routing", default="return", choices=["return", "lazy"],
                    help="shor: SWAP routing (return: every routed qubit moves back; lazy: it stays)")
    ap.add_argument("--tensor-cores", type=int, default=None, choices=[0, 1, 2],
                    help="tensor-core policy (default 1, the size policy; 0 never; 2 always, "
                         "including the Jacobi round updates)")
    ap.add_argument("--layers", type=int, default=0,
                    help="cfg2 / sketch-cfg4: circuit depth (default: 50 / 30)")
    args = ap.parse_args()
    if args.n is None:
        args.n = {"compare": 60, "apply-traffic": 24, "bidiag-traffic": 32, "sketch-cfg4": 100}.get(args.workload, 500)
    if args.chi is None:
        args.chi = {"tebd": 256, "shor": 256}.get(args.workload, 1024)
    if args.kmax is None:
        args.kmax = 8 if args.workload in ("tebd", "shor") else 4
    if args.workload == "tebd":
        run_tebd(args)
        return
    if args.workload == "shor":
        run_shor(args)
        return
    if args.workload in ("cfg2", "sketch-cfg4"):
        run_cfg2(args)
        return
    if args.workload == "compare":
        run_compare(args)
        return
    if args.workload == "latency":
        run_latency(args)
        return
    if args.workload == "cfg5":
        run_cfg5(args)
        return
    if args.workload == "bidiag-traffic":
        run_bidiag_traffic(args)
        return
    if args.workload == "apply-traffic":
        run_apply_traffic(args)
        return
    rank = int(os.environ.get("RANK", 0))
    world = int(os.environ.get("WORLD_SIZE", 1))
    local_rank = int(os.environ.get("LOCAL_RANK", 0))
    pk = peaks()
    workload = (f"cfg4: n={args.n}, 100-layer random-structured Clifford+T (20% T), "
                f"chi_max={args.chi}, cutoff 1e-8, k_max={args.kmax}, "
                f"Q_max={args.kmax + 2 * int(math.log2(args.chi))}; "
                "synthetic saturated state (all interior bonds at chi_max)")
    config = {"workload": workload, "precision": "complex64 contractions, fp64 spectra/weights",
              "l2": "inputs larger than L2 (theta/Gram per step >> 129 MB)", "replicas": world}
    if args.tensor_cores is not None:
        config["tensor_cores"] = {0: "never", 1: "size policy", 2: "always, Jacobi round updates included"}[
            args.tensor_cores]

    if args.impl == "reference":
        if rank != 0:
            return
        vals = []
        for _ in range(args.warmup):
            cpu_baseline(seconds=2.0)
        t0 = time.perf_counter()
        for _ in range(args.steps):
            vals.append(cpu_baseline(seconds=max(args.cpu_seconds / max(args.steps, 1), 3.0)))
        dt = time.perf_counter() - t0
        v = float(np.mean([x["value"] for x in vals]))
        cb = dict(vals[-1])
        cb["value"] = v
        cb["measured_value"] = float(np.mean([x["measured_value"] for x in vals]))
        line = {"impl": "reference", "metric": METRIC, "value": v, "unit": UNIT, "n_gpus": 1,
                "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1000 * dt / args.steps,
                "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
                "data": "synthetic", "config": config, "cpu_baseline": cb,
                "e2e": {"value": v, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
        print(json.dumps(line))
        return

    import torch
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    res = run_ours(args, rank, world, local_rank)
    dev_s = res["dev_ms"] / 1000.0
    units = res["updates"]
    wall = res["wall_s"]
    if world > 1:
        dev_s, wall, units = aggregate(dev_s, wall, units, device=f"cuda:{local_rank}")
    if rank != 0:
        if world > 1:
            import torch.distributed as dist
            dist.destroy_process_group()
        return
    prof = res["prof"]
    clocks = res["clocks"]
    mp = res["peaks"]
    # dominant kernel class by device time
    dom_name, dom = max(prof.items(), key=lambda kv: kv[1]["ms"])
    alu_peak = mp["fp32_simt_tflops"]
    tc_peak = mp["tf32_tflops"]
    if dom.get("tc_launches", 0) > 0 and dom["flops"] > 0:
        achieved = dom["flops"] / (dom["ms"] / 1000.0) / 1e12
        roof = {"kernel": dom_name, "bound": "tensor", "achieved": achieved, "peak": tc_peak / 3.0,
                "unit": "TFLOP/s", "frac": achieved / (tc_peak / 3.0), "traffic": None,
                "peak_source": "measured TF32 burst / 3 (three TF32 products per FP32-accurate product)",
                "launches": dom["launches"], "avg_launch_ms": dom["ms"] / max(dom["launches"], 1)}
    elif dom["flops"] > 0:
        achieved = dom["flops"] / (dom["ms"] / 1000.0) / 1e12
        traffic, t_note = traffic_per_launch(dom_name, dom["flops"] / max(dom["launches"], 1))
        roof = {"kernel": dom_name, "bound": "alu", "achieved": achieved, "peak": alu_peak,
                "unit": "TFLOP/s", "frac": achieved / alu_peak, "traffic": traffic,
                "traffic_unit": "bytes per launch", "traffic_source": t_note,
                "peak_source": mp["fp32_source"] + f"; {mp['n_sm']} SMs",
                "launches": dom["launches"], "avg_launch_ms": dom["ms"] / max(dom["launches"], 1)}
    else:
        achieved = dom["bytes"] / (dom["ms"] / 1000.0) / 1e9
        roof = {"kernel": dom_name, "bound": "hbm", "achieved": achieved, "peak": pk["hbm_gbs"],
                "unit": "GB/s", "frac": achieved / pk["hbm_gbs"], "traffic": None,
                "peak_source": pk["source"], "launches": dom["launches"]}
    counts = res["counts"]
    total_flops = sum(v["flops"] for v in counts.values())
    tflops = total_flops / dev_s / 1e12 if dev_s > 0 else 0.0
    f_method = res["f_merge"] + res["f_u"] + res["f_split"]
    tflops_method = f_method / dev_s / 1e12 * world if dev_s > 0 else 0.0
    tc_cls = {k: v for k, v in prof.items() if v.get("tc_launches", 0) > 0}
    tc_ms = sum(v["ms"] for v in tc_cls.values())
    tc_achieved = sum(v["flops"] for v in tc_cls.values()) / (tc_ms / 1000.0) / 1e12 if tc_ms > 0 else 0.0
    tensor_cores = {"classes": sorted(tc_cls), "tc_launches": int(sum(v["tc_launches"] for v in tc_cls.values())),
                    "achieved": tc_achieved, "peak": tc_peak, "unit": "TFLOP/s", "frac": tc_achieved / tc_peak,
                    "share_of_step": tc_ms / max(sum(v["ms"] for v in prof.values()), 1e-9),
                    "peak_source": mp["tf32_source"],
                    "note": "algorithmic complex-GEMM flops; the pipe runs 3 TF32 products per product "
                            "(hi/lo split) for FP32 accuracy"}
    flops = {
        "method": {"tflops": tflops_method, "tc_frac": tflops_method / tc_peak,
                   "per_step_tflop": {"merge": res["f_merge"] / 1e12 / max(args.steps, 1),
                                      "apply_u": res["f_u"] / 1e12 / max(args.steps, 1),
                                      "split": res["f_split"] / 1e12 / max(args.steps, 1)},
                   "definition": "the method's work from the actual shapes: merge chain + U + per split the "
                                 "randomized truncated SVD of the target design (sketch width l = r + 8, "
                                 "q = 0, CholeskyQR2, write-back; the l^3 small-SVD term excluded)"},
        "executed": {"tflops": tflops * world, "tc_frac": tflops * world / tc_peak,
                     "definition": "algorithmic flops of the kernels this implementation runs (bidiagonalisation, "
                                   "divide and conquer, back-transformation, projections, merge, U)"},
        "tc_peak": tc_peak, "tc_peak_source": mp["tf32_source"],
    }
    gpu_launches = int(sum(v["launches"] for v in counts.values()))
    value = units / dev_s if dev_s > 0 else 0.0
    cpu = cpu_baseline(seconds=args.cpu_seconds) if args.cpu_seconds > 0 else None
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": 1000.0 * dev_s / max(args.steps, 1),
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "c64",
        "data": "synthetic (seeded circuit + random saturated MPS)", "config": config,
        "tflops_algorithmic": tflops * world,
        "tc_frac": tflops_method / tc_peak,
        "flops": flops,
        "peaks_measured": mp,
        "tensor_cores": tensor_cores,
        "roofline": roof,
        "kernels": {k: {"launches": int(v["launches"]), "ms": round(v["ms"], 3),
                        "share": round(v["ms"] / max(sum(x["ms"] for x in prof.values()), 1e-9), 4)}
                    for k, v in prof.items() if v["launches"] > 0},
        "kernels_note": "per-launch CUDA events of one further iteration; the timed iterations run without events",
        "cpu_baseline": cpu,
        "e2e": {"value": units / wall if wall > 0 else 0.0, "unit": UNIT,
                "h2d_bytes_per_step": int(res["h2d"] / max(args.steps, 1)),
                "d2h_bytes_per_step": int(res["d2h"] / max(args.steps, 1))},
        "gpu_launches": gpu_launches,
        "clocks": clocks,
        "updates": units,
        "steps_detail": res["steps_detail"],
    }
    if res["jacobi_sweeps"]:   # splits that took the Gram matrix and Jacobi
        line["jacobi_sweeps"] = res["jacobi_sweeps"]
    if "plain" in res and "error" in res["plain"]:
        line["plain_fp64"] = res["plain"]
    elif "plain" in res:
        pl = res["plain"]
        line["plain_fp64"] = {"updates_per_s": pl["updates"] / pl["s"],
                              "ours_same_sample_updates_per_s": pl["updates"] / pl["ours_s"],
                              "speedup": (pl["s"] / pl["ours_s"]) if pl["ours_s"] > 0 else None,
                              "max_abs_df": pl["max_abs_df"], "F_plain": pl["F_plain"],
                              "F_ours": pl["F_ours"], "sample_updates": pl["updates"]}
    print(json.dumps(line))
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
