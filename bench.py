"""Benchmark of the exact-exchange apply (Vx psi and E_x) on one GB300.

A step is one kx_vx_apply over the whole workload: the 96^3 isolated-box system
(Dirichlet, unscreened, 12th-order FD, h = 0.25 bohr, 64 orbitals, 2080
symmetric pair solves), inputs resident in HBM.  The metric is pair-solves/s of
the split-precision tensor-core path; the float64 GPU path, the error against
it, an end-to-end host-buffer run and the FP64 CPU oracle are reported beside.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl kronx|reference]

Under torchrun (N > 1) every rank runs an independent replica of the workload
(weak scaling, no data-path collective); rank 0 prints one JSON line.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import workloads  # noqa: E402

METRIC = "pair-solves/s and Vx*psi time, split-precision vs FP64 on 1 GB300 at stated error"
UNIT = "pair-solves/s"
SYS = workloads.C2
WORKLOAD = ("96x96x96 isolated box, Dirichlet, unscreened f=-4pi/lambda, 12th-order FD, h=0.25 bohr, "
            "64 orbitals, 2080 symmetric pair solves + Vx*psi + E_x per step")
DATA = "synthetic: seeded s/p Gaussian-sum orbitals on 24 random atom centres, FP64 CholeskyQR2-orthonormalised"


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=30)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", choices=["kronx", "reference"], default="kronx")
    ap.add_argument("--no-extras", action="store_true", help="skip FP64/e2e/oracle legs (profiling runs)")
    ap.add_argument("--no-tune", action="store_true",
                    help="skip the launch-shape tuner (profiling runs: keeps its trial launches out of a capture)")
    ap.add_argument("--profile-case", choices=["small", "ace", "multipole", "fft", "kpoints", "fp64"], default=None,
                    help="small: one apply of a small case of the same kernels (96^3, 8 orbitals); ace: three "
                         "ACE operator applies at 96^3 with 64 + 64 vectors; multipole: two applies of the "
                         "headline system with boundary values to order 4; fft: the first 64 pairs of the "
                         "80^3 periodic system on a KX_FFT32 plan, twice; kpoints: Vx of the 64^3 slab's "
                         "16 bands at one k-point of its 2 x 2 grid, twice; all for ncu captures")
    return ap.parse_args()


def run_profile_case(which="small"):
    """small: one split-precision apply at 96^3 with 8 orbitals (36 pairs): the
    same kernels as the bench workload on inputs of about L2 size, so that an
    ncu capture with many passes stays short.  ace: three kx_ace_apply calls on
    the headline system's tensor-core plan with 64 seeded vectors xi (scaled by
    1e-3) and 64 orbitals phi (1.4 GB on the device)."""
    import torch
    import paper_2406_16998_gb300 as kx
    from paper_2406_16998_gb300 import build
    build.build()
    if which == "fft":
        sysd = workloads.C3
        plan = kx.Plan.for_system(sysd, precision=kx.KX_FFT32)
        psi = torch.from_numpy(np.ascontiguousarray(workloads.make_orbitals(sysd).T)).cuda()
        for _ in range(2):
            vx, ex = kx.kx_vx_apply_pairs(plan, psi, 0, 64)
        torch.cuda.synchronize()
        print(json.dumps({"profile_case": "fft", "e_x": ex.item(), "status": plan.status()}), flush=True)
        return
    if which == "kpoints":
        kd = workloads.K1
        theta, wk = workloads.kpoint_grid(kd, workloads.K1_KGRID)
        psi = torch.from_numpy(np.ascontiguousarray(
            np.transpose(workloads.make_bloch_orbitals(kd, theta), (0, 2, 1)))).cuda()
        plan = kx.Plan.for_system(kd, precision=kx.KX_F16X3)
        for _ in range(2):
            out = kx.kx_vx_apply_kpoint(plan, theta, wk, psi, 1, psi[1])
        torch.cuda.synchronize()
        print(json.dumps({"profile_case": "kpoints", "maxabs": out.abs().max().item(), "status": plan.status()}),
              flush=True)
        return
    if which == "fp64":
        # the float64 path (the speed-up denominator) on the small case below
        case = workloads.System(n=(96, 96, 96), h=(0.25,) * 3, bc=(workloads.DIRICHLET,) * 3,
                                kernel=workloads.UNSCREENED, n_orb=8, n_centres=4, seed=5, name="profile-small")
        psi = torch.from_numpy(np.ascontiguousarray(workloads.make_orbitals(case).T)).cuda()
        plan = kx.Plan.for_system(case, precision=kx.KX_FP64)
        vx, ex = kx.kx_vx_apply(plan, psi)
        torch.cuda.synchronize()
        print(json.dumps({"profile_case": "fp64", "e_x": ex.item(), "status": plan.status()}), flush=True)
        return
    if which == "multipole":
        plan = kx.Plan.for_system(SYS, precision=kx.KX_F16X3)
        plan.set_multipole(4)
        psi = torch.from_numpy(np.ascontiguousarray(workloads.make_orbitals(SYS).T)).cuda()
        for _ in range(2):
            vx, ex = kx.kx_vx_apply(plan, psi)
        torch.cuda.synchronize()
        print(json.dumps({"profile_case": "multipole", "e_x": ex.item(), "status": plan.status()}), flush=True)
        return
    if which == "ace":
        plan = kx.Plan.for_system(SYS, precision=kx.KX_F16X3)
        xi = torch.from_numpy(np.ascontiguousarray(workloads.random_field(plan.N, 64, 3).T) * 1e-3).cuda()
        phi = torch.from_numpy(np.ascontiguousarray(workloads.make_orbitals(SYS).T)).cuda()
        out = torch.empty_like(phi)
        for _ in range(3):
            kx.kx_ace_apply(plan, xi, phi, out=out)
        torch.cuda.synchronize()
        print(json.dumps({"profile_case": "ace", "max_abs": float(out.abs().max())}), flush=True)
        return
    case = workloads.System(n=(96, 96, 96), h=(0.25,) * 3, bc=(workloads.DIRICHLET,) * 3,
                            kernel=workloads.UNSCREENED, n_orb=8, n_centres=4, seed=5, name="profile-small")
    psi = torch.from_numpy(np.ascontiguousarray(workloads.make_orbitals(case).T)).cuda()
    plan = kx.Plan.for_system(case, precision=kx.KX_F16X3)
    vx, ex = kx.kx_vx_apply(plan, psi)
    torch.cuda.synchronize()
    status = plan.status()
    print(json.dumps({"profile_case": "small", "e_x": ex.item(), "status": status}), flush=True)
    if status != kx.KX_OK:
        raise SystemExit(1)


def peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), float(d["bf16_tflops"]), float(d.get("bf16_tflops_sustained", d["bf16_tflops"])), "measured"
    except Exception:
        return 6800.0, 1900.0, 1700.0, "fallback"


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled every 100 ms while running."""
    FIELDS = ["clocks.sm", "clocks.max.sm", "power.draw", "clocks_event_reasons.hw_slowdown",
              "clocks_event_reasons.hw_thermal_slowdown", "clocks_event_reasons.sw_thermal_slowdown",
              "clocks_event_reasons.sw_power_cap"]

    def __init__(self, index):
        self.index = index
        self.rows = []
        self.proc = None

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.index}", "--query-gpu=" + ",".join(self.FIELDS),
                                          "--format=csv,noheader,nounits", "-lms", "100"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
            time.sleep(0.5)
        except Exception:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            parts = [p.strip() for p in line.split(",")]
            if len(parts) == len(self.FIELDS):
                self.rows.append(parts)

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        sm = [float(r[0]) for r in self.rows if r[0].replace(".", "").isdigit()]
        mx = [float(r[1]) for r in self.rows if r[1].replace(".", "").isdigit()]
        reasons = set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for r in self.rows:
            for k, nm in enumerate(names):
                if r[3 + k].lower().startswith("active"):
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": sorted(reasons), "samples": len(self.rows)}


def dist_setup(n_gpus):
    import torch
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if n_gpus > 1 and world != n_gpus:
        raise SystemExit(f"--gpus {n_gpus} needs torchrun with {n_gpus} ranks (WORLD_SIZE={world})")
    if torch.cuda.is_available():
        torch.cuda.set_device(local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl" if torch.cuda.is_available() else "gloo")
    return world, rank, local


def barrier(world):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def max_over_ranks(x, world):
    if world == 1:
        return x
    import torch
    import torch.distributed as dist
    t = torch.tensor([x], dtype=torch.float64, device="cuda")
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def cpu_baseline(psi, budget_s=12.0):
    """The FP64 oracle as it stands, on a bounded sample of the workload's pairs
    (the first pairs of the library's pair list, so that the same partial sums
    can be compared with the split path's).  Returns the timing line and the
    oracle's partial (Vx psi, E_x) over those pairs."""
    import oracle
    from paper_2406_16998_gb300 import shard
    op = oracle.Plan(SYS.n, SYS.h, SYS.bc, SYS.kernel, SYS.omega)
    n_orb = psi.shape[1]
    pairs = shard.pair_list(n_orb)
    done, dt = 0, 0.0
    vx_sum, ex_sum = None, 0.0
    while done < len(pairs):
        chunk = pairs[done:done + 4]
        t0 = time.perf_counter()
        vx, ex = oracle.vx_apply(op, psi, pairs=chunk)
        dt += time.perf_counter() - t0  # the oracle's own time; summing the samples is not counted
        vx_sum = vx if vx_sum is None else vx_sum + vx
        ex_sum += ex
        done += len(chunk)
        if dt > budget_s:
            break
    line = {"value": done / dt, "unit": UNIT, "cores": len(os.sched_getaffinity(0)), "kind": "oracle",
            "sample": f"first {done} of {len(pairs)} symmetric pairs of the workload (pair product, f(L) by "
                      f"mode products, both accumulations), {dt:.1f} s of NumPy FP64"}
    return line, done, vx_sum, ex_sum


def run_reference(args):
    """Reference arm: the oracle (FP64 NumPy, host cores) on bounded samples of the same workload."""
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    import oracle
    psi = workloads.make_orbitals(SYS)
    op = oracle.Plan(SYS.n, SYS.h, SYS.bc, SYS.kernel, SYS.omega)
    pairs = oracle.pair_list(SYS.n_orb, ordered=False)
    per_step = 4
    for w in range(args.warmup):
        oracle.vx_apply(op, psi, pairs=pairs[w * per_step:(w + 1) * per_step])
    t0 = time.perf_counter()
    for s in range(args.steps):
        k0 = ((args.warmup + s) * per_step) % len(pairs)
        oracle.vx_apply(op, psi, pairs=pairs[k0:k0 + per_step])
    dt = time.perf_counter() - t0
    value = per_step * args.steps / dt
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * dt / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": DATA, "config": {"workload": WORKLOAD, "sample": f"{per_step} pair solves per step"},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": len(os.sched_getaffinity(0)), "kind": "oracle",
                             "sample": f"{per_step} symmetric pairs of the workload per step, {args.steps} steps"},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


# algorithmic work per item of each pass (useful flops; fp32 scratch / input / output bytes)
def pass_model(n):
    n1, n2, n3 = n
    N = n1 * n2 * n3
    return {
        "X3F": (2.0 * N * n3, 4.0 * N + 8.0 * N),      # rho from two fp32 orbitals, write mode-3 coefficients
        "X2F": (2.0 * N * n2, 8.0 * N),
        "X1": (4.0 * N * n1, 8.0 * N),                  # forward + inverse mode 1 in one pass
        "X2I": (2.0 * N * n2, 8.0 * N),
        "slab": (4.0 * N * (n1 + n2), 8.0 * N),         # X2F + X1 + X2I fused per k3 slice
        "X3I": (2.0 * N * n3, 8.0 * N),                 # read coefficients, write phi
        "acc": (4.0 * N, 7.0 * N),                       # read phi; one orbital block exchanged per group
    }


# DRAM bytes per unit of a kernel, from the ncu summaries under profiles/: a
# line "traffic: <kernel> <bytes per unit> <unit> sha256=<hash of the kernel's
# source text when the capture was taken>".  The figure is used only while the
# source still has that hash; otherwise the traffic is reported as null.
# The hash covers the kernel's own source text: from `start` up to `end`.
TRAFFIC_SOURCES = {"slab": ("profiles/tc_slab_kernel_96cube_8orb_full.md", "paper_2406_16998_gb300/csrc/kx_tc.cu",
                            "struct SlabArgs {", "// Accumulation of one chunk")}


def kernel_source_hash(kind):
    import hashlib
    _, source, start, end = TRAFFIC_SOURCES[kind]
    text = open(os.path.join(ROOT, source)).read()
    a = text.index(start)
    return hashlib.sha256(text[a:text.index(end, a)].encode()).hexdigest()


def measured_traffic(kind, units_per_launch):
    if kind not in TRAFFIC_SOURCES:
        return None, "no ncu capture for this kernel"
    summary = os.path.join(ROOT, TRAFFIC_SOURCES[kind][0])
    try:
        sha = kernel_source_hash(kind)
        for line in open(summary):
            f = line.split()
            if len(f) >= 5 and f[0] == "traffic:" and f[1] == kind:
                if f[4] != "sha256=" + sha:
                    return None, "kernel source changed since the ncu capture"
                return float(f[2]) * units_per_launch, f"ncu dram__bytes_read+write per {f[3]} x units per launch"
    except OSError:
        pass
    return None, "no ncu capture for this kernel"


def other_workloads(kx, torch, stream, hbm, bf16, steps=3):
    """Context lines beside the headline: the split path on the 80^3 periodic
    screened 256-orbital system (32896 pairs), the same system through the FFT
    variant, the batch of eight systems (26400 pairs) replayed as one CUDA graph,
    and the Bloch k-point path on the 64^3 slab (4096 pair solves)."""
    res = {}
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    sysd = workloads.C3
    psi = torch.from_numpy(np.ascontiguousarray(workloads.make_orbitals(sysd).T)).cuda()
    plan = kx.Plan.for_system(sysd, precision=kx.KX_F16X3)
    vx = torch.empty_like(psi)
    ex = torch.empty(1, dtype=torch.float64, device="cuda")
    kx.kx_vx_apply(plan, psi, out=vx, e_x=ex)
    e0.record(stream)
    for _ in range(steps):
        kx.kx_vx_apply(plan, psi, out=vx, e_x=ex)
    e1.record(stream)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / steps
    P3 = sysd.n_orb * (sysd.n_orb + 1) // 2
    res["c3_80cube_periodic_screened_256orb"] = {"ms_per_apply": ms, "pair_solves_per_s": P3 / (ms / 1e3),
                                                 "pairs": P3, "status": plan.status()}
    # the same system through the FFT variant (KX_FFT32: float32 DFTs on the CUDA cores);
    # its passes move half spectra, h = (n1 / 2 + 1) / n1 of the complex values: 32 h N + 4 N
    # bytes per pair (pass A writes 8 h N, B reads and writes 16 h N, C reads 8 h N and writes 4 N)
    plan_f = kx.Plan.for_system(sysd, precision=kx.KX_FFT32)
    vx_f = torch.empty_like(vx)
    ex_f = torch.empty(1, dtype=torch.float64, device="cuda")
    kx.kx_vx_apply(plan_f, psi, out=vx_f, e_x=ex_f)
    e0.record(stream)
    kx.kx_vx_apply(plan_f, psi, out=vx_f, e_x=ex_f)
    e1.record(stream)
    torch.cuda.synchronize()
    ms_f = e0.elapsed_time(e1)
    plan_f.profile(True)
    kx.kx_vx_apply(plan_f, psi, out=vx_f, e_x=ex_f)
    pr = plan_f.profile_read()
    plan_f.profile(False)
    fft_ms = pr["fft"][0]
    fft_bytes = (32.0 * (sysd.n[0] // 2 + 1) / sysd.n[0] + 4.0) * plan_f.N
    gbs = fft_bytes * P3 / (fft_ms / 1e3) / 1e9
    res["c3_fft_variant"] = {
        "ms_per_apply": ms_f, "pair_solves_per_s": P3 / (ms_f / 1e3), "fft_passes_ms": fft_ms,
        "kronecker_speedup": ms_f / ms, "status": plan_f.status(),
        "vx_psi_maxrel_vs_kronecker": float((vx_f - vx).abs().max() / vx.abs().max()),
        "e_x_rel_vs_kronecker": abs(ex_f.item() - ex.item()) / abs(ex.item()),
        "fft_roofline": {"bound": "hbm", "achieved": gbs, "peak": hbm, "unit": "GB/s", "frac": gbs / hbm,
                         "algorithmic_bytes_per_pair": fft_bytes}}
    del psi, vx, plan, plan_f, vx_f
    plans, psis, outs, P4 = [], [], [], 0
    for sd in workloads.C4:
        plans.append(kx.Plan.for_system(sd, precision=kx.KX_F16X3))
        psis.append(torch.from_numpy(np.ascontiguousarray(workloads.make_orbitals(sd).T)).cuda())
        outs.append(torch.empty_like(psis[-1]))
        P4 += sd.n_orb * (sd.n_orb + 1) // 2
    t0 = time.perf_counter()
    batch = kx.Batch(plans, [sd.n_orb for sd in workloads.C4])  # tunes each plan (400 ms budget)
    create_s = time.perf_counter() - t0
    exs = torch.empty(len(plans), dtype=torch.float64, device="cuda")
    batch.run(psis, outs, e_x=exs, stream=stream)
    e0.record(stream)
    for _ in range(steps):
        batch.run(psis, outs, e_x=exs, stream=stream)
    e1.record(stream)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / steps
    useful = sum(workloads.useful_flops_per_pair(sd.n) * sd.n_orb * (sd.n_orb + 1) // 2 for sd in workloads.C4)
    tf = useful / (ms / 1e3) / 1e12
    # per system: orbital 0's row of Vx psi (its pair solves with every orbital)
    # against the oracle, and E_x against 1/2 dV sum_i <psi_i, (Vx psi)_i>
    import oracle
    errs, t_or = [], 0.0
    for k, sd in enumerate(workloads.C4):
        psi_h = psis[k].cpu().numpy().T
        op = oracle.Plan(sd.n, sd.h, sd.bc, sd.kernel, sd.omega, sd.fd_order)
        t1 = time.perf_counter()
        ref, _ = oracle.vx_apply(op, psi_h, ordered=True, pairs=[(0, j) for j in range(sd.n_orb)])
        t_or += time.perf_counter() - t1
        got = outs[k][0].cpu().numpy()
        vxh = outs[k].cpu().numpy()
        e_id = 0.5 * sd.dV * float(np.einsum("ij,ij->", psis[k].cpu().numpy(), vxh))
        errs.append({"system": sd.name, "row0_vx_maxrel_vs_oracle": float(np.max(np.abs(got - ref[:, 0])) /
                                                                            np.max(np.abs(ref[:, 0]))),
                     "e_x": exs[k].item(), "e_x_rel_vs_identity": abs(exs[k].item() - e_id) / abs(e_id),
                     "tuning": plans[k].tuning()})
    res["c4_batch_8_systems"] = {"ms_per_batch": ms, "pair_solves_per_s": P4 / (ms / 1e3), "pairs": P4,
                                 "status": [p.status() for p in plans], "batch_create_s": create_s,
                                 "useful_tflops": tf,
                                 "roofline": {"bound": "tensor", "achieved": tf, "peak": bf16 / 3.0, "unit": "TFLOP/s",
                                              "frac": tf / (bf16 / 3.0),
                                              "peak_source": "measured bf16_tflops / 3 (three fp16 products)"},
                                 "per_system": errs, "oracle_rows_s": t_or}
    batch.close()
    del psis, outs, plans
    # Bloch k-points: the 64^3 slab (periodic x1 and x2, vacuum along x3), 16 bands
    # on a 2 x 2 k-grid; Vx psi at every k-point needs the pair blocks (k, q),
    # q >= k (10 of 16: a reversed block is the conjugate solve), 16 x 16 pair
    # solves each, six complex mode products per solve on the tensor cores (axes
    # of 64 points): each reads and writes the solve's complex float32 grid
    # vector once, 16 N bytes, so 96 N bytes per solve (the HBM roofline);
    # 16 N (n1 + n2 + n3) useful flops per solve (float64 plan for the error)
    kd = workloads.K1
    theta, wk = workloads.kpoint_grid(kd, workloads.K1_KGRID)
    psi_np = workloads.make_bloch_orbitals(kd, theta)
    psi_k = torch.from_numpy(np.ascontiguousarray(np.transpose(psi_np, (0, 2, 1)))).cuda()
    plan_k = kx.Plan.for_system(kd, precision=kx.KX_F16X3)
    vx_k = torch.empty_like(psi_k)
    ex_k = torch.empty(1, dtype=torch.float64, device="cuda")
    kx.kx_vx_kpoints(plan_k, theta, wk, psi_k, out=vx_k, e_x=ex_k, stream=stream)
    e0.record(stream)
    for _ in range(steps):
        kx.kx_vx_kpoints(plan_k, theta, wk, psi_k, out=vx_k, e_x=ex_k, stream=stream)
    e1.record(stream)
    torch.cuda.synchronize()
    ms_k = e0.elapsed_time(e1) / steps
    plan_k.profile(True)
    kx.kx_vx_kpoints(plan_k, theta, wk, psi_k, out=vx_k, e_x=ex_k, stream=stream)
    pr = plan_k.profile_read()
    plan_k.profile(False)
    PK = len(wk) * (len(wk) + 1) // 2 * kd.n_orb ** 2
    flops_pair = 16.0 * kd.N * sum(kd.n)
    bytes_pair = 40.0 * kd.N  # forward pair writes, middle and inverse pairs read and write, complex64
    tf = flops_pair * PK / (pr["bloch"][0] / 1e3) / 1e12
    gbs_k = bytes_pair * PK / (pr["bloch"][0] / 1e3) / 1e9
    # the same apply with the CUDA-core products (KX_BLOCH_TC=0), for comparison
    vx_cc = torch.empty_like(psi_k)
    os.environ["KX_BLOCH_TC"] = "0"
    try:
        kx.kx_vx_kpoints(plan_k, theta, wk, psi_k, out=vx_cc, stream=stream)
        plan_k.profile(True)
        kx.kx_vx_kpoints(plan_k, theta, wk, psi_k, out=vx_cc, stream=stream)
        pr_cc = plan_k.profile_read()
        plan_k.profile(False)
    finally:
        del os.environ["KX_BLOCH_TC"]
    cc_rel = float((vx_cc - vx_k).abs().max() / vx_k.abs().max())
    del vx_cc
    e0.record(stream)
    e_only = kx.kx_energy_kpoints(plan_k, theta, wk, psi_k, stream=stream)
    e1.record(stream)
    torch.cuda.synchronize()
    ms_e = e0.elapsed_time(e1)
    plan_k64 = kx.Plan.for_system(kd, precision=kx.KX_FP64)
    vx_64, ex_64 = kx.kx_vx_kpoints(plan_k64, theta, wk, psi_k, stream=stream)
    torch.cuda.synchronize()
    # the oracle as it stands on a bounded sample, beside it: Vx of band 0 at
    # k-point 1 (its pair solves with every band of every k-point), which is
    # also a full-size parity check of that band
    import oracle
    base = oracle.Plan(kd.n, kd.h, kd.bc, kd.kernel, kd.omega, kd.fd_order)
    t0 = time.perf_counter()
    ref_band = oracle.vx_apply_kpoint(base, theta, wk, psi_np, None, 1, psi_np[1][:, :1])[:, 0]
    dt_o = time.perf_counter() - t0
    got_band = vx_k[1, 0].cpu().numpy()
    n_sample = len(wk) * kd.n_orb
    res["k1_kpoints_slab_64cube_16bands_2x2"] = {
        "ms_per_apply": ms_k, "pair_solves_per_s": PK / (ms_k / 1e3), "pairs": PK,
        "pairs_of_the_k_sum": len(wk) ** 2 * kd.n_orb ** 2,
        "mode_products_ms": pr["bloch"][0], "mode_product_launches": pr["bloch"][1],
        "cuda_core_mode_products_ms": pr_cc["bloch"][0], "cuda_core_vx_maxrel_vs_tensor_core": cc_rel,
        "other_kernels_ms": pr["bloch_other"][0], "e_x": ex_k.item(), "status": plan_k.status(),
        "energy_only_ms": ms_e, "energy_only_rel_vs_vx_path": abs(e_only.item() - ex_k.item()) / abs(ex_k.item()),
        "vx_maxrel_vs_fp64_plan": float((vx_k - vx_64).abs().max() / vx_64.abs().max()),
        "vs_oracle_sampled": {"vx_band_maxrel": float(np.max(np.abs(got_band - ref_band)) / np.max(np.abs(ref_band)))},
        "cpu_baseline": {"value": n_sample / dt_o, "unit": "pair-solves/s", "cores": len(os.sched_getaffinity(0)),
                         "kind": "oracle",
                         "sample": f"Vx of band 0 at k-point 1: its {n_sample} pair solves with every band of every "
                                   f"k-point, {dt_o:.1f} s of NumPy FP64"},
        "e_x_rel_vs_fp64_plan": abs(ex_k.item() - ex_64.item()) / abs(ex_64.item()),
        "useful_tflops": tf,
        "roofline": {"bound": "hbm", "achieved": gbs_k, "peak": hbm, "unit": "GB/s", "frac": gbs_k / hbm,
                     "algorithmic_bytes_per_pair": bytes_pair}}
    return res


def ace_legs(kx, torch, stream, plan, psi, vx, hbm, steps=5):
    """The ACE tail and the compressed operator on the headline system: xi from
    (psi, Vx psi) with kx_ace, then V_ACE applied to the orbitals with
    kx_ace_apply.  The apply reads xi and phi for the projections and xi again
    for the combination and writes out: 16 N (n_xi + n_vec) bytes, its HBM
    roofline.  Errors are against the float64 plan on the same xi and psi, and
    the ACE property V_ACE psi = Vx psi."""
    n_orb, N = psi.shape
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    xi, _ = kx.kx_ace(plan, psi, vx)  # first call reserves the workspace
    t0 = time.perf_counter()
    for _ in range(steps):
        xi, _ = kx.kx_ace(plan, psi, vx)  # synchronises (reads the Cholesky flag)
    ms_ace = 1e3 * (time.perf_counter() - t0) / steps
    out = torch.empty_like(psi)
    kx.kx_ace_apply(plan, xi, psi, out=out, stream=stream)
    torch.cuda.synchronize()
    e0.record(stream)
    for _ in range(steps):
        kx.kx_ace_apply(plan, xi, psi, out=out, stream=stream)
    e1.record(stream)
    torch.cuda.synchronize()
    ms_apply = e0.elapsed_time(e1) / steps
    plan.profile(True)
    kx.kx_ace_apply(plan, xi, psi, out=out, stream=stream)
    prof = plan.profile_read()
    plan.profile(False)
    kernels = {"projection_ms": prof["ace"][0], "combination_ms": prof["ace_comb"][0],
               "launches": prof["ace"][1] + prof["ace_comb"][1]}
    plan64 = kx.Plan.for_system(SYS, precision=kx.KX_FP64)
    out64 = torch.empty_like(psi)
    kx.kx_ace_apply(plan64, xi, psi, out=out64, stream=stream)
    torch.cuda.synchronize()
    e0.record(stream)
    kx.kx_ace_apply(plan64, xi, psi, out=out64, stream=stream)
    e1.record(stream)
    torch.cuda.synchronize()
    ms64 = e0.elapsed_time(e1)
    bytes_apply = 16.0 * N * (n_orb + n_orb)
    gbs = bytes_apply / (ms_apply / 1e3) / 1e9
    return {"ace_build_ms": ms_ace,
            "ace_apply_ms": ms_apply, "ace_apply_kernels": kernels, "ace_apply_fp64_ms": ms64,
            "speedup_vs_fp64": ms64 / ms_apply,
            "ace_apply_roofline": {"bound": "hbm", "achieved": gbs, "peak": hbm, "unit": "GB/s", "frac": gbs / hbm,
                                   "algorithmic_bytes": bytes_apply},
            "ace_apply_maxrel_vs_fp64_gpu": float((out - out64).abs().max() / out64.abs().max()),
            "ace_psi_vs_vx_psi_maxrel": float((out - vx).abs().max() / vx.abs().max()),
            "n_xi": n_orb, "n_vec": n_orb}


FP32_ALU_PEAK_TFLOPS = 152 * 128 * 2 * 2.07e9 / 1e12  # SMs x FP32 lanes x flops per FMA x max SM clock


def multipole_legs(kx, torch, stream, plan, psi, ms_zero, bf16, steps=3):
    """Vx psi of the headline system with Dirichlet values from the multipole
    expansion (orders 2 and 4) instead of zero boundary values: time per apply,
    the correction kernels' time, and their tensor roofline: the weighted
    moments of the pair densities and the k-weighted combination each take
    K n^2 N multiply-adds (K = (l_max + 1)^2), issued as three fp16 products on
    the tensor cores for up to 64 orbitals, so the bound is the measured bf16
    peak / 3 in useful flops."""
    res = {}
    n_orb, N = psi.shape
    vx = torch.empty_like(psi)
    ex = torch.empty(1, dtype=torch.float64, device="cuda")
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    for l_max in (2, 4):
        t0 = time.perf_counter()
        plan.set_multipole(l_max)
        setup_s = time.perf_counter() - t0
        kx.kx_vx_apply(plan, psi, out=vx, e_x=ex, stream=stream)
        torch.cuda.synchronize()
        e0.record(stream)
        for _ in range(steps):
            kx.kx_vx_apply(plan, psi, out=vx, e_x=ex, stream=stream)
        e1.record(stream)
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1) / steps
        plan.profile(True)
        kx.kx_vx_apply(plan, psi, out=vx, e_x=ex, stream=stream)
        prof = plan.profile_read()
        plan.profile(False)
        mp_ms = prof["multipole"][0]
        K = (l_max + 1) ** 2
        flops = 4.0 * K * n_orb * n_orb * N
        ach = flops / (mp_ms / 1e3) / 1e12
        tensor = n_orb <= 64
        pk = bf16 / 3.0 if tensor else FP32_ALU_PEAK_TFLOPS
        res[f"l_max_{l_max}"] = {
            "ms_per_apply": ms, "overhead_ms": ms - ms_zero, "correction_ms": mp_ms, "setup_s": setup_s,
            "e_x": ex.item(), "status": plan.status(),
            "correction_roofline": {
                "bound": "tensor" if tensor else "alu", "achieved": ach, "peak": pk, "unit": "TFLOP/s",
                "frac": ach / pk,
                "peak_source": ("measured bf16_tflops / 3 (three fp16 products per useful product)" if tensor else
                                "derived: 152 SMs x 128 FP32 lanes x 2 flops x 2.07 GHz")}}
    plan.set_multipole(-1)
    return res


def matmul_peaks(torch, reps=5):
    """Dense matmul peaks of this GPU that the float64 and float32 legs are
    measured against: torch.matmul (cuBLAS) in float64 (4096^3) and in float32
    with TF32 allowed (8192^3), best of `reps` under CUDA events after a
    warm-up.  A benchmark of the library GEMMs, not a GPU setting."""
    res = {}
    for name, dtype, n, tf32 in (("fp64", torch.float64, 4096, False), ("tf32", torch.float32, 8192, True)):
        prev = torch.backends.cuda.matmul.allow_tf32
        torch.backends.cuda.matmul.allow_tf32 = tf32
        try:
            a = torch.randn(n, n, dtype=dtype, device="cuda")
            b = torch.randn(n, n, dtype=dtype, device="cuda")
            c = torch.matmul(a, b)
            torch.cuda.synchronize()
            best = 1e30
            for _ in range(reps):
                e0 = torch.cuda.Event(enable_timing=True)
                e1 = torch.cuda.Event(enable_timing=True)
                e0.record()
                torch.matmul(a, b, out=c)
                e1.record()
                torch.cuda.synchronize()
                best = min(best, e0.elapsed_time(e1))
            res[name + "_tflops"] = 2.0 * n ** 3 / (best / 1e3) / 1e12
            res[name + "_shape"] = f"{n}x{n}x{n}"
            del a, b, c
        finally:
            torch.backends.cuda.matmul.allow_tf32 = prev
    res["how"] = "torch.matmul best of %d (CUDA events); fp64 plain, fp32 with allow_tf32" % reps
    return res


def c1_leg(kx, torch, stream, fp64_peak, reps=5):
    """Config 1 in full on the float64 plan: 32^3 isolated box, h = 0.5, 4
    orbitals.  The configuration counts the 16 ordered pairs; the library
    solves the 10 unordered ones (the ordered and symmetric sums agree).  Time
    per apply (best and median of `reps`), its float64 roofline fraction, and
    the error against the oracle over all 16 ordered pairs."""
    import oracle
    sysd = workloads.C1
    psi_h = workloads.make_orbitals(sysd)
    psi = torch.from_numpy(np.ascontiguousarray(psi_h.T)).cuda()
    plan = kx.Plan.for_system(sysd, precision=kx.KX_FP64)
    vx = torch.empty_like(psi)
    ex = torch.empty(1, dtype=torch.float64, device="cuda")
    kx.kx_vx_apply(plan, psi, out=vx, e_x=ex, stream=stream)
    torch.cuda.synchronize()
    times = []
    for _ in range(reps):
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        kx.kx_vx_apply(plan, psi, out=vx, e_x=ex, stream=stream)
        e1.record(stream)
        torch.cuda.synchronize()
        times.append(e0.elapsed_time(e1))
    op = oracle.Plan(sysd.n, sysd.h, sysd.bc, sysd.kernel, sysd.omega)
    t0 = time.perf_counter()
    vx_ref, ex_ref = oracle.vx_apply(op, psi_h, ordered=True)
    dt_o = time.perf_counter() - t0
    P_sym = sysd.n_orb * (sysd.n_orb + 1) // 2
    useful = workloads.useful_flops_per_pair(sysd.n) * P_sym
    best = min(times)
    ach = 0.5 * useful / (best / 1e3) / 1e12  # products by eigenvector parity: half the dense form's
    return {"ms_per_apply_best": best, "ms_per_apply_median": statistics.median(times), "repeats": reps,
            "ordered_pairs": sysd.n_orb ** 2, "solves": P_sym,
            "vx_psi_maxrel_vs_oracle": float(np.max(np.abs(vx.cpu().numpy().T - vx_ref)) / np.max(np.abs(vx_ref))),
            "e_x_rel_vs_oracle": abs(ex.item() - ex_ref) / abs(ex_ref), "e_x": ex.item(),
            "oracle_s": dt_o, "status": plan.status(),
            "roofline": {"bound": "fp64", "achieved": ach, "peak": fp64_peak, "unit": "TFLOP/s",
                         "frac": ach / fp64_peak,
                         "note": "launch-bound at this size (1.0e8 flops); peak = measured torch.matmul float64"}}


def c5_leg(kx, torch, stream):
    """Config 5: E_x of the 80^3 periodic screened 256-orbital system through
    the autograd function (forward kx_energy: forward products and the
    Parseval sum; backward kx_energy_gradient: pair products recomputed, Vx psi,
    2 dV g Vx psi), split-precision forward, float64 energy sums.  Forward and
    backward times (CUDA events), and the gradient and energy against the
    float64 plan's kx_energy_gradient on the same orbitals."""
    sysd = workloads.C5
    psi = torch.from_numpy(np.ascontiguousarray(workloads.make_orbitals(sysd).T)).cuda()
    plan = kx.Plan.for_system(sysd, precision=kx.KX_F16X3)
    P = sysd.n_orb * (sysd.n_orb + 1) // 2
    x = psi.clone().requires_grad_(True)
    kx.exchange_energy(x, plan).backward()  # warm-up (sizes the workspaces)
    torch.cuda.synchronize()
    fw, bw = [], []
    for _ in range(3):
        x.grad = None
        e0, e1, e2 = (torch.cuda.Event(enable_timing=True) for _ in range(3))
        e0.record(stream)
        E = kx.exchange_energy(x, plan)
        e1.record(stream)
        E.backward()
        e2.record(stream)
        torch.cuda.synchronize()
        fw.append(e0.elapsed_time(e1))
        bw.append(e1.elapsed_time(e2))
    g = x.grad.detach()
    e_split = E.item()
    del x
    plan64 = kx.Plan.for_system(sysd, precision=kx.KX_FP64)
    t0 = time.perf_counter()
    g64, e64 = kx.kx_energy_gradient(plan64, psi)
    torch.cuda.synchronize()
    dt64 = time.perf_counter() - t0
    res = {"forward_ms": min(fw), "backward_ms": min(bw), "repeats": 3, "pairs": P,
           "forward_pair_solves_per_s": P / (min(fw) / 1e3), "backward_pair_solves_per_s": P / (min(bw) / 1e3),
           "grad_maxrel_vs_fp64_plan": float((g - g64).abs().max() / g64.abs().max()),
           "e_x_rel_vs_fp64_plan": abs(e_split - e64.item()) / abs(e64.item()), "e_x": e_split,
           "fp64_gradient_s": dt64, "status": plan.status(),
           "targets": {"grad": 1e-5, "e_x": 1e-6}}
    del g, g64, psi, plan, plan64
    return res


def issued_tensor_flops_per_pair(n, fused=True):
    """Tensor-core flops the split path issues per pair: three fp16 products per
    mode product, M padded to 128-row tiles, K and N padded to multiples of 16."""
    n1, n2, n3 = n
    npad = [((x + 15) // 16) * 16 for x in n]
    np1, np2, np3 = npad
    f = 3 * 2 * 2 * (n1 * n2) * np3 * np3            # X3F and X3I: rows = positions
    if fused:
        f += n3 * 3 * 2 * 128 * (2 * np2 * np2 + 2 * np1 * np1)   # slab: M1, M4 (x2) and M2, M3 (x1)
    else:
        f += 3 * 2 * 2 * (n3 * n1) * np2 * np2 + 3 * 2 * 2 * (n3 * n2) * np1 * np1
    return float(f)


def main():
    args = parse()
    if args.profile_case:
        return run_profile_case(args.profile_case)
    if args.impl == "reference":
        return run_reference(args)
    import torch
    import paper_2406_16998_gb300 as kx
    from paper_2406_16998_gb300 import build
    world, rank, local = dist_setup(args.gpus)
    if rank == 0:
        build.build()
    barrier(world)
    hbm, bf16, bf16_sus, peak_src = peaks()

    psi_h = workloads.make_orbitals(SYS)                  # (N, n_orb) float64
    psi_t = np.ascontiguousarray(psi_h.T)                 # (n_orb, N): orbital-major, x1 fastest
    psi = torch.from_numpy(psi_t).cuda()
    n_orb, N = psi.shape
    P = n_orb * (n_orb + 1) // 2
    plan = kx.Plan.for_system(SYS, precision=kx.KX_F16X3)
    vx = torch.empty_like(psi)
    ex = torch.empty(1, dtype=torch.float64, device="cuda")
    stream = torch.cuda.current_stream()
    # launch shapes chosen by the library's tuner for this grid and orbital count
    t0 = time.perf_counter()
    if not args.no_tune:
        kx.kx_autotune(plan, n_orb, 6000)
    tune_s = time.perf_counter() - t0
    tuning = dict(plan.tuning(), tune_s=tune_s, tuned=not args.no_tune)

    for _ in range(max(3, args.warmup)):
        kx.kx_vx_apply(plan, psi, out=vx, e_x=ex)
    torch.cuda.synchronize()
    assert plan.status() == kx.KX_OK

    clocks = ClockSampler(local)
    clocks.start()
    barrier(world)
    torch.cuda.synchronize()
    plan.profile(True)
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(args.steps):
        kx.kx_vx_apply(plan, psi, out=vx, e_x=ex)
    e1.record(stream)
    torch.cuda.synchronize()
    barrier(world)
    ms_total = e0.elapsed_time(e1)
    clk = clocks.stop()
    prof = plan.profile_read()
    plan.profile(False)
    ms_total = max_over_ranks(ms_total, world)
    ms_step = ms_total / args.steps
    value = world * P * args.steps / (ms_total / 1e3)
    gpu_launches = sum(v[1] for v in prof.values())

    if rank != 0:
        barrier(world)
        return

    # roofline of the dominant kernel (largest share of timed device time)
    model = pass_model(SYS.n)
    kinds = {k: prof[k] for k in model}
    dom = max(kinds, key=lambda k: kinds[k][0])
    dom_ms, dom_launches = kinds[dom]
    avg_ms = dom_ms / max(1, dom_launches)
    items_per_launch = P * args.steps / max(1, dom_launches)
    flops, bytes_ = model[dom]
    t_tensor = flops * 3 / (bf16 * 1e12)
    t_hbm = bytes_ / (hbm * 1e9)
    if t_hbm >= t_tensor:
        ach = bytes_ * items_per_launch / (avg_ms / 1e3) / 1e9
        roof = {"bound": "hbm", "achieved": ach, "peak": hbm, "unit": "GB/s", "frac": ach / hbm,
                "traffic": None, "kernel": dom, "peak_source": f"{peak_src} hbm_gbs (copy)"}
    else:
        ach = flops * items_per_launch / (avg_ms / 1e3) / 1e12
        pk = bf16 / 3.0
        roof = {"bound": "tensor", "achieved": ach, "peak": pk, "unit": "TFLOP/s", "frac": ach / pk,
                "traffic": None, "kernel": dom,
                "peak_source": f"{peak_src} bf16_tflops / 3 (three fp16 products per useful product)"}
    roof["traffic"], roof["traffic_source"] = measured_traffic(dom, SYS.n[2] * items_per_launch)
    roof["avg_launch_ms"] = avg_ms
    if roof["traffic"] is not None:  # DRAM bytes per launch / launch time, against the measured copy peak
        roof["dram_gbs"] = roof["traffic"] / (avg_ms / 1e3) / 1e9
        roof["dram_frac_of_hbm_peak"] = roof["dram_gbs"] / hbm
    roof["items_per_launch"] = items_per_launch
    kern = {k: {"ms_total": v[0], "launches": v[1], "share": v[0] / max(1e-9, sum(x[0] for x in prof.values()))}
            for k, v in prof.items() if v[1] > 0}

    out = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
           "warmup": args.warmup, "ms_per_step": ms_step, "higher_is_better": True, "scaling": "weak",
           "vs_baseline": None, "dtype": "f16x3", "data": DATA,
           "config": {"workload": WORKLOAD, "grid": list(SYS.n), "h_bohr": SYS.h[0], "bc": "dirichlet",
                      "kernel": "unscreened", "fd_order": SYS.fd_order, "n_orb": n_orb, "pairs_per_step": P,
                      "precision": "f16x3: fp16 hi/lo split of both operands, 3 tcgen05 products, fp32 accumulate",
                      "l2": "inputs larger than L2 (psi 453 MB float64, fp32 scratch > 1 GB per chunk)",
                      "tuning": tuning},
           "vx_psi_ms": ms_step, "roofline": roof, "kernels": kern, "gpu_launches": gpu_launches,
           "clocks": clk}
    n1, n2, n3 = SYS.n
    useful = 4.0 * n1 * n2 * n3 * (n1 + n2 + n3)
    fused = prof.get("slab", (0.0, 0))[1] > 0
    out["flops"] = {"useful_per_pair": useful,
                    "useful_tflops": P * useful / (ms_step / 1e3) / 1e12,
                    "issued_tensor_tflops": P * issued_tensor_flops_per_pair(SYS.n, fused) / (ms_step / 1e3) / 1e12,
                    "split_tensor_bound_ms": 3 * P * useful / (bf16_sus * 1e12) * 1e3,
                    "peak_bf16_tflops": bf16, "peak_bf16_sustained_tflops": bf16_sus}

    if not args.no_extras:
        vx_split = vx.clone()
        ex_split = ex.item()
        # end to end through the C ABI with host buffers (pinned), copies inside the timed region;
        # measured right after the headline steps, before the long float64 leg heats the part
        psi_pin = torch.from_numpy(psi_t).pin_memory()
        vx_pin = torch.empty_like(psi_pin).pin_memory()
        kx.kx_vx_apply_host(plan, psi_pin, out=vx_pin)
        k_e2e = max(3, min(args.steps, 10))
        t_steps = []
        t0 = time.perf_counter()
        for _ in range(k_e2e):
            ts = time.perf_counter()
            kx.kx_vx_apply_host(plan, psi_pin, out=vx_pin)
            t_steps.append(1e3 * (time.perf_counter() - ts))
        dt = time.perf_counter() - t0
        # the host link's rates in the same process (one pinned copy each way), beside the end-to-end number
        c0, c1, c2 = (torch.cuda.Event(enable_timing=True) for _ in range(3))
        c0.record(stream)
        vx.copy_(psi_pin, non_blocking=True)
        c1.record(stream)
        vx_pin.copy_(vx, non_blocking=True)
        c2.record(stream)
        torch.cuda.synchronize()
        nb = psi_pin.numel() * 8
        out["e2e"] = {"value": P * k_e2e / dt, "unit": UNIT, "h2d_bytes_per_step": psi_pin.numel() * 8,
                      "d2h_bytes_per_step": vx_pin.numel() * 8 + 8, "ms_per_step": 1e3 * dt / k_e2e,
                      "ms_each": [round(t, 3) for t in t_steps],
                      "link_gbs": {"h2d": nb / c0.elapsed_time(c1) / 1e6, "d2h": nb / c1.elapsed_time(c2) / 1e6}}

        # float64 GPU path on the same inputs: the speed-up denominator and the full-size error reference
        plan64 = kx.Plan.for_system(SYS, precision=kx.KX_FP64)
        vx64 = torch.empty_like(psi)
        ex64 = torch.empty(1, dtype=torch.float64, device="cuda")
        kx.kx_vx_apply(plan64, psi, out=vx64, e_x=ex64)
        torch.cuda.synchronize()
        t64 = []
        for _ in range(3):
            f0 = torch.cuda.Event(enable_timing=True)
            f1 = torch.cuda.Event(enable_timing=True)
            f0.record(stream)
            kx.kx_vx_apply(plan64, psi, out=vx64, e_x=ex64)
            f1.record(stream)
            torch.cuda.synchronize()
            t64.append(f0.elapsed_time(f1))
        ms64 = statistics.median(t64)
        err_vx = float((vx_split - vx64).abs().max() / vx64.abs().max())
        err_ex = abs(ex_split - ex64.item()) / abs(ex64.item())
        mm = matmul_peaks(torch)
        out["measured_matmul_peaks"] = mm
        ach64 = 0.5 * P * useful / (ms64 / 1e3) / 1e12  # products by eigenvector parity: half the dense form's
        out["fp64_gpu"] = {"ms_per_step": ms64, "ms_per_step_all": t64, "pair_solves_per_s": P / (ms64 / 1e3),
                           "speedup_split_vs_fp64": ms64 / ms_step,
                           "roofline": {"bound": "fp64", "achieved": ach64, "peak": mm["fp64_tflops"],
                                        "unit": "TFLOP/s", "frac": ach64 / mm["fp64_tflops"],
                                        "peak_source": "measured torch.matmul float64 4096^3 (cuBLAS DGEMM)"}}
        out["c1_fp64_32cube_4orb"] = c1_leg(kx, torch, stream, mm["fp64_tflops"])
        out["error"] = {"vx_psi_maxrel_vs_fp64_gpu": err_vx, "e_x_rel_vs_fp64_gpu": err_ex,
                        "targets": {"vx_psi": 1e-5, "e_x": 1e-6}, "e_x": ex_split}
        del plan64, vx64
        out["ace"] = ace_legs(kx, torch, stream, plan, psi, vx_split, hbm)
        out["multipole"] = multipole_legs(kx, torch, stream, plan, psi, ms_step, bf16)
        out["multipole"]["e_x_zero_boundary"] = ex_split
        out["other_workloads"] = other_workloads(kx, torch, stream, hbm, bf16)
        out["c5_autograd_80cube_256orb"] = c5_leg(kx, torch, stream)
        line, done, vx_ref, ex_ref = cpu_baseline(psi_h)
        out["cpu_baseline"] = line
        # the split path over the same first pairs of the list, against the oracle
        vx_part, ex_part = kx.kx_vx_apply_pairs(plan, psi, 0, done)
        vx_part = vx_part.cpu().numpy().T
        out["error"]["vs_oracle_sampled"] = {
            "pairs": done,
            "vx_psi_maxrel": float(np.max(np.abs(vx_part - vx_ref)) / np.max(np.abs(vx_ref))),
            "e_x_rel": abs(ex_part.item() - ex_ref) / abs(ex_ref)}
    print(json.dumps(out), flush=True)
    barrier(world)


if __name__ == "__main__":
    main()
