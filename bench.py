#!/usr/bin/env python3
"""Benchmark: density-matrix solves/s of the sparse Chebyshev (FOE) method on GB300.

One step = one complete density-matrix solve of a synthetic atom-centred system
(10,000 atoms x 4 basis functions = 40,000 rows, 10 bohr block cutoff, 4 bohr
output buffer, kT = 0.005 Ha, N_e = 20,000) for a new Hamiltonian: H' =
S^-1/2 H S^-1/2, Lanczos bounds, coefficients and degree, the half-length
moment pass with the penalty check, the bisection that brackets mu*, the
accumulation pass with 4 simultaneous mu (FP32 block products, double-float
accumulators returned in FP64) that also collects every moment, the exact
bisection, interpolation at mu*, post-processing and Tr(FS).  The overlap
matrix is fixed across steps (as in a self-consistent-field loop): block
patterns, plans, gather plans, S^-1/2 and the trace functional are built once
per geometry before the timed region (their time is reported as setup_s), and
every step solves H_k = H + eps_k S (eps_k = 1e-4 k Ha), a new Hamiltonian
whose levels are those of H shifted by eps_k.

Usage: python bench.py [--gpus N] [--steps K] [--warmup W] [--impl cheb|reference]
N > 1 runs under torchrun: each rank solves its own system (seed = rank), no
collective on the data path (weak scaling); timing is the max over ranks.
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

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

METRIC = "density-matrix solves/s at <=1e-6 vs FP64 plain; masked SpGEMM HBM GB/s"
UNIT = "solves/s"
FALLBACK_HBM_GBS = 6800.0
# DRAM bytes (dram__bytes_read.sum + dram__bytes_write.sum) per step of the
# column-order kernel, from one ncu capture of every k_colstep launch of a
# 4-mu solve on 3,000 atoms (12,000 rows, r_c 10, r_out 14 bohr: 1,183,812
# P_out blocks; kT 0.05 Ha, 960 terms: 478 pass-1 launches with moments only,
# 958 pass-2 launches with four accumulators; grouped steps included; atoms in
# Hilbert order, as the 4-mu workloads run), GB300.  Per-launch traffic scales with the P_out blocks (the
# operator has the same share of them).  Valid only for the kernel source it was
# measured on: the sha256 of colstep.cu's text before its host-builder section
# (the kernels and their launch code); after any change there the bench reports
# traffic null.
COL_KERNEL_END = "// Host: the column kernel's panels and work streams"
COL_TRAFFIC = {"colstep_sha256": "154741e02d152208e90026c68cebafde56a0824781690b584981970ab666ee15",
               "blocks_P_out": 1183812, "pass1_bytes": 453.7e6, "pass2_4acc_bytes": 857.9e6, "order": "hilbert"}
SMS, FP32_LANES, MAX_SM_MHZ = 152, 128, 2070.0
# Dense f16 mma.sync rate measured with a register-only kernel (GB300, 2,070 MHz), and the
# digit products that make one product of the column kernel.
MMA_F16_TFLOPS = 604.0
DIGIT_PRODUCTS = {"float": 6, "double": 26}

WORKLOADS = {
    # The mixed-precision density matrix: 10,000 atoms x 4, 10 bohr cutoff,
    # 4 simultaneous mu (the bracket of a half-length moment pass).
    # The atoms are relabelled along a Hilbert curve inside the solve (inputs and
    # F stay in the generator's labelling).
    "foe_mixed_40k": dict(n_atoms=10000, r_c=10.0, r_buf=4.0, kT=0.005, N_e=20000.0, tol=1e-7, tol_S=1e-10,
                          precision="f32", n_mu=4, form="mu4", order="hilbert"),
    # The same solve as moment pass + bisection + accumulation pass at mu*.
    "foe_mixed_40k_twopass": dict(n_atoms=10000, r_c=10.0, r_buf=4.0, kT=0.005, N_e=20000.0, tol=1e-7,
                                  tol_S=1e-10, precision="f32", n_mu=1, form="twopass"),
    # The same solve in one pass: the learned mu proposal (weights trained by
    # paper_1704_00512_gb300/train_mu.py) brackets mu*, 8 accumulators at
    # Chebyshev nodes of the bracket, bisection on the same pass judges, a
    # second pass only if mu* falls outside the bracket.
    "foe_mixed_40k_learned": dict(n_atoms=10000, r_c=10.0, r_buf=4.0, kT=0.005, N_e=20000.0, tol=1e-7,
                                  tol_S=1e-10, precision="f32", n_mu=8, form="learned", max_half_kT=1.0),
    # The learned proposal deployed on 25,000 atoms x 4 (100,000 rows), 10 bohr
    # cutoff, kT = 0.005 Ha, N_e = rows/2; with the same system solved by the
    # plain moment pass + bisection + accumulation pass for comparison.
    "foe_learned_100k": dict(n_atoms=25000, r_c=10.0, r_buf=4.0, kT=0.005, N_e=50000.0, tol=1e-7, tol_S=1e-10,
                             precision="f32", n_mu=8, form="learned", max_half_kT=1.0),
    "foe_mixed_100k_twopass": dict(n_atoms=25000, r_c=10.0, r_buf=4.0, kT=0.005, N_e=50000.0, tol=1e-7,
                                   tol_S=1e-10, precision="f32", n_mu=1, form="twopass"),
    # The same solve on 3,000 atoms (12,000 rows): profiling stand-in for the launch list.
    "foe_mixed_12k": dict(n_atoms=3000, r_c=10.0, r_buf=4.0, kT=0.005, N_e=6000.0, tol=1e-7, tol_S=1e-10,
                          precision="f32", n_mu=4, form="mu4", order="hilbert"),
    # Same 12,000-row system at kT = 0.05 (about 10x fewer terms): keeps a per-launch
    # profiler capture of a whole solve short.
    "foe_mixed_12k_kT05": dict(n_atoms=3000, r_c=10.0, r_buf=4.0, kT=0.05, N_e=6000.0, tol=1e-7, tol_S=1e-10,
                               precision="f32", n_mu=4, form="mu4", order="hilbert"),
    # The smearing chosen on the fly on the 12,000-row system: two-pass solves
    # from kT = 0.04 Ha, halved until E = Tr(K H) and E' of the same polynomials
    # at 1.25 kT differ by at most dE_tol (0.2 Ha, 6.7e-5 Ha per atom).
    "foe_mixed_12k_autokT": dict(n_atoms=3000, r_c=10.0, r_buf=4.0, kT=0.04, N_e=6000.0, tol=1e-7, tol_S=1e-10,
                                 precision="f32", n_mu=1, form="autokT", dE_tol=0.2, widen=1.25, shrink=0.5),
    # The plain FP64 density matrix: 200 atoms x 4, 8 bohr cutoff, kT = 0.01, N_e = 400.
    "foe_fp64_800": dict(n_atoms=200, r_c=8.0, r_buf=4.0, kT=0.01, N_e=400.0, tol=1e-10, tol_S=1e-10,
                         precision="f64", n_mu=1, form="twopass"),
    # Matrix powers S^-1, S^1/2, S^-1/2 from one shared FP64 recursion: 3,000
    # atoms x 4 (12,000 rows), 10 bohr cutoff, 4 bohr output buffer.
    "powers_fp64_12k": dict(powers=True, n_atoms=3000, r_c=10.0, r_buf=4.0, tol=1e-10, precision="f64", n_mu=3,
                            exponents=(-1.0, 0.5, -0.5)),
    # The same powers with FP64-accurate double-float products on the FP32 pipe
    # (CHEB_F64X), timed against the FP64 expansion in the same run.
    "powers_f64x_12k": dict(powers=True, n_atoms=3000, r_c=10.0, r_buf=4.0, tol=1e-10, precision="f64x", n_mu=3,
                            exponents=(-1.0, 0.5, -0.5)),
    # Batched: 64 independent systems of U{125..1500} atoms (seeds 0..63), 8 bohr
    # cutoff, each with its own bounds, degree and mu; both passes one launch
    # each, captured in CUDA graphs; autotuned tile shapes.
    "foe_batched_64": dict(batched=True, n_sys=64, atoms_lo=125, atoms_hi=1500, r_c=8.0, r_buf=4.0, kT=0.01,
                           tol=1e-7, tol_S=1e-10, precision="f32", n_mu=1),
}
DEFAULT_WORKLOAD = "foe_mixed_40k"


def log(*a):
    print(*a, file=sys.stderr, flush=True)


# --------------------------------------------------------------------------
# clocks sampled during the timed region
# --------------------------------------------------------------------------

class ClockSampler:
    FIELDS = ("clocks.sm,clocks.max.sm,clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")
    NAMES = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]

    def __init__(self, gpu_index: int, enabled: bool = True):
        self.idx = gpu_index
        self.enabled = enabled
        self.proc = None
        self.lines: list[str] = []
        self.th = None

    def start(self):
        if not self.enabled:
            return
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.idx), f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
            return
        self.th = threading.Thread(target=self._read, daemon=True)
        self.th.start()

    def _read(self):
        for ln in self.proc.stdout:
            self.lines.append(ln.strip())

    def stop(self) -> dict:
        if self.proc is None:
            why = "not sampled (--no-clocks)" if not self.enabled else "nvidia-smi unavailable"
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": [why]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        if self.th:
            self.th.join(timeout=5)
        sm, smax, reasons = [], [], set()
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 6:
                continue
            try:
                sm.append(float(parts[0]))
                smax.append(float(parts[1]))
            except ValueError:
                continue
            for name, v in zip(self.NAMES, parts[2:6]):
                if v.lower().startswith("active"):
                    reasons.add(name)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(smax) if smax else None,
                "reasons": sorted(reasons), "samples": len(sm)}


# --------------------------------------------------------------------------
# algorithmic accounting of the recursion step
# --------------------------------------------------------------------------

def count_triples(row_ptr_H, col_idx_H, row_ptr_O, col_idx_O) -> int:
    """Number of (I,K,J) with (I,K) in P_H, (K,J) in P_out and (I,J) in P_out."""
    import scipy.sparse as sp
    n = len(row_ptr_H) - 1
    A = sp.csr_matrix((np.ones(len(col_idx_H), np.float64), col_idx_H, row_ptr_H), shape=(n, n))
    B = sp.csr_matrix((np.ones(len(col_idx_O), np.float64), col_idx_O, row_ptr_O), shape=(n, n))
    return int(round((A @ B).multiply(B).sum()))


def measured_hbm_peak() -> tuple[float, str]:
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(p) as f:
            d = json.load(f)
        for k in ("hbm_gbs", "hbm_GBps", "hbm"):
            if k in d:
                return float(d[k]), "measured"
    except (OSError, ValueError):
        pass
    return FALLBACK_HBM_GBS, "fallback"


# --------------------------------------------------------------------------
# ranks: each rank solves its own seeded system (no data-path collective); the
# timed region is bracketed by barriers and the job time is the max over ranks
# --------------------------------------------------------------------------

def rank_env() -> tuple[int, int, int]:
    """(rank, world size, local rank) from the torchrun environment (1 process by default)."""
    return (int(os.environ.get("RANK", "0")), int(os.environ.get("WORLD_SIZE", "1")),
            int(os.environ.get("LOCAL_RANK", "0")))


def system_seed(rank: int) -> int:
    """Seed of the system a rank solves: independent systems, weak scaling."""
    return rank


def max_over_ranks(x: float, world: int, device) -> float:
    """The largest value of x over all ranks (x itself for one rank)."""
    if world <= 1:
        return float(x)
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_throughput(steps: int, world: int, t_ms: float) -> float:
    """Whole-job solves/s: every rank solved `steps` systems within the max time t_ms."""
    return steps * world / (t_ms / 1e3)


# --------------------------------------------------------------------------
# the CUDA arm
# --------------------------------------------------------------------------

def col_step_bytes(nnz_out: int, nnz_H: int, n_acc: int, with_G: bool) -> int:
    """Algorithmic bytes of one FP32 step of the column-order kernel: T_k, T_{k-1}
    read and T_{k+1} written (FP32), the operator (FP32) once, 8 bytes per element
    read and written for each accumulator (double-float pairs, as many bytes as
    FP64), 8 bytes per element of G read."""
    b = nnz_out * 16 * 4 * 3 + nnz_H * 16 * 4 + nnz_out * 16 * 8 * 2 * n_acc
    if with_G:
        b += nnz_out * 16 * 8
    return b


def fp64_plain_step_ms(pb, Hpt, n_steps: int = 12) -> float:
    """Time of one step of the plain FP64 GPU form (FP64 products, one FP64
    accumulator) on the same operator: n_steps steps of the FP64 per-step kernel."""
    import torch
    import paper_1704_00512_gb300 as cg
    c = torch.ones((1, n_steps + 2), dtype=torch.float64, device=pb.device) * 1e-3
    acc = [pb.zeros_out()]
    cg.expand(pb.plan64, Hpt, 3, c, acc, precision=cg.F64, stepwise=True)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    cg.expand(pb.plan64, Hpt, n_steps + 2, c, acc, precision=cg.F64, stepwise=True)
    e1.record()
    torch.cuda.synchronize()
    return e0.elapsed_time(e1) / n_steps


def run_cheb(args, rank: int, world: int, local: int):
    import torch
    import torch.distributed as dist

    import synth
    import paper_1704_00512_gb300 as cg
    from paper_1704_00512_gb300 import solve

    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if world > 1:
        dist.init_process_group("nccl", device_id=dev)
    cfg = WORKLOADS[args.workload]
    prec = cg.F32 if cfg["precision"] == "f32" else cg.F64
    t0 = time.time()
    sysm = synth.make_system(cfg["n_atoms"], cfg["r_c"], seed=system_seed(rank))
    log(f"[rank {rank}] generated {sysm.n_rows} rows, {sysm.nnzb} blocks in {time.time() - t0:.1f}s")
    # per-geometry setup: patterns, plans, gather plans, S^-1/2 and G
    torch.cuda.synchronize()
    ts = time.time()
    pb = solve.problem_from_system(sysm, cfg["r_buf"], dev, prec, order=cfg.get("order"))
    torch.cuda.synchronize()
    plans_s = time.time() - ts
    ov = solve.overlap_setup(pb, cfg["tol_S"])
    torch.cuda.synchronize()
    setup_s = time.time() - ts
    log(f"[rank {rank}] setup {setup_s:.2f}s (patterns, plans, S^-1/2 with {ov['n_S']} terms, G); "
        f"column kernel {cg.plan_col_info(pb.planX) if prec != cg.F64 else 'n/a'}")
    H0 = pb.H.vals.clone()
    S_vals = pb.S.vals
    form = cfg.get("form", "twopass")
    if form == "learned":
        from paper_1704_00512_gb300 import learned
        prop = learned.load_proposal(dev)
        kw = dict(kT=cfg["kT"], N_e=cfg["N_e"], tol=cfg["tol"], n_mu=cfg["n_mu"], max_half_kT=cfg["max_half_kT"])

        def solve_once(timings=None):
            A, G = ov["A"], ov["G"]
            Hp = solve.orthogonalise(pb, A)
            e0, e1, _ = cg.bounds(Hp, 40)
            prepared = (A, Hp.with_vals(cg.scale(Hp, e0, e1)), (e0, e1), G, Hp)
            return learned.foe_learned(pb, prop, prepared=prepared, timings=timings, **kw)
    elif form == "autokT":
        def solve_once(timings=None):
            return solve.foe_auto_kT(pb, cfg["kT"], cfg["N_e"], cfg["dE_tol"], cfg["widen"], cfg["shrink"],
                                     tol=cfg["tol"], overlap=ov, timings=timings)
    else:
        kw = dict(kT=cfg["kT"], N_e=cfg["N_e"], tol=cfg["tol"], n_mu=cfg["n_mu"], form=form)

        def solve_once(timings=None):
            return solve.foe(pb, overlap=ov, timings=timings, **kw)

    def step(k, timings=None):
        # the step's Hamiltonian H_k = H + eps_k S: levels of H shifted by eps_k
        torch.add(H0, S_vals, alpha=1e-4 * k, out=pb.H.vals)
        return solve_once(timings)

    k_step = 0
    for i in range(args.warmup):
        tw = time.time()
        out = step(k_step)
        k_step += 1
        torch.cuda.synchronize()
        log(f"[rank {rank}] warmup {i}: {time.time() - tw:.2f}s n_terms={out['n_terms']} mu={out['mu']:.6f} "
            f"passes={out['passes']} TrFS={out['trace_FS'].item():.6f}")

    # ---- device-resident timed region
    clk = ClockSampler(local, enabled=not args.no_clocks)
    pass_ev = []
    outs = []
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    l0 = cg.launch_count()
    clk.start()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(args.steps):
        tm = {}
        out = step(k_step, tm)
        k_step += 1
        pass_ev.append(tm["events"])
        outs.append(out)
    e1.record()
    torch.cuda.synchronize()
    clocks = clk.stop()
    launches = cg.launch_count() - l0
    if world > 1:
        dist.barrier()
    t_ms = e0.elapsed_time(e1)
    t_ms = max_over_ranks(t_ms, world, dev)
    value = job_throughput(args.steps, world, t_ms)
    n_terms = out["n_terms"]
    nnz_out, nnz_H = pb.P_out.nnzb, pb.P_H.nnzb

    # ---- end-to-end through the same API: H from pinned host memory, F and
    # Tr(FS) back to the host, every step
    h_H = [torch.from_numpy(np.ascontiguousarray(sysm.H) + 1e-4 * (k_step + j) * np.ascontiguousarray(sysm.S))
           .pin_memory() for j in range(args.e2e_steps)]
    h_F = torch.empty((nnz_out, 4, 4), dtype=torch.float64).pin_memory()
    h_tr = torch.empty(1, dtype=torch.float64).pin_memory()
    h2d = sysm.H.size * 8
    d2h = h_F.numel() * 8 + 8
    d_H = torch.empty_like(pb.H.vals)  # the host H lands here, then moves to the solve's labelling
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    f0, f1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    f0.record()
    for j in range(args.e2e_steps):
        d_H.copy_(h_H[j], non_blocking=True)
        pb.set_H(d_H)
        o = solve_once()
        h_F.copy_(pb.to_caller_out(o["F"]), non_blocking=True)
        h_tr.copy_(o["trace_FS"], non_blocking=True)
    f1.record()
    torch.cuda.synchronize()
    te_ms = max_over_ranks(f0.elapsed_time(f1), world, dev)
    e2e_value = job_throughput(args.e2e_steps, world, te_ms) if args.e2e_steps > 0 else None

    # ---- roofline of the dominant kernel (the fused recursion step)
    triples = count_triples(pb.P_H.row_ptr.cpu().numpy(), pb.P_H.col_idx.cpu().numpy(),
                            pb.P_out.row_ptr.cpu().numpy(), pb.P_out.col_idx.cpu().numpy())
    flops = 2.0 * 64.0 * triples
    if prec == cg.F32 and form == "mu4":
        m = out["n_pass1"]
        launches_pass = [m - 2, n_terms - 2]
        bytes_pass = [col_step_bytes(nnz_out, nnz_H, 0, True), col_step_bytes(nnz_out, nnz_H, cfg["n_mu"], True)]
        p_ms = [statistics.mean(ev[0].elapsed_time(ev[1]) for ev in pass_ev),
                statistics.mean(ev[2].elapsed_time(ev[3]) for ev in pass_ev)]
    elif prec == cg.F32 and form in ("twopass", "autokT"):
        # (the smearing loop: the passes of its accepted round, whose second
        # pass also collects the energy moments)
        launches_pass = [n_terms - 2, n_terms - 2]
        bytes_pass = [col_step_bytes(nnz_out, nnz_H, 0, True),
                      col_step_bytes(nnz_out, nnz_H, 1, form == "autokT")]
        p_ms = [statistics.mean(ev[0].elapsed_time(ev[1]) for ev in pass_ev),
                statistics.mean(ev[2].elapsed_time(ev[3]) for ev in pass_ev)]
    else:
        launches_pass, bytes_pass, p_ms = [], [], []
    roof = None
    if launches_pass:
        n_launch = sum(launches_pass)
        avg_ms = sum(p_ms) / n_launch
        alg_bytes = sum(b * l for b, l in zip(bytes_pass, launches_pass)) / n_launch
        tflops = flops / (avg_ms / 1e3) / 1e12
        gbs = alg_bytes / (avg_ms / 1e3) / 1e9
        hbm_peak, hbm_src = measured_hbm_peak()
        traffic = col_traffic_per_launch(form, cfg["n_mu"], launches_pass, nnz_out, order=cfg.get("order"))
        roof = {**step_roof(tflops, "f32", True), "traffic": traffic, "algorithmic_flops_per_step": flops,
                "algorithmic_bytes_per_step": int(alg_bytes), "avg_step_ms": round(avg_ms, 5),
                "hbm_gbs": round(gbs, 1), "hbm_frac": round(gbs / hbm_peak, 4),
                "hbm_peak": hbm_peak, "hbm_peak_source": f"{hbm_src} copy bandwidth"}
    # ---- the plain FP64 GPU form on the same operator (time-to-solution)
    vs64 = None
    if prec == cg.F32 and not args.no_fp64_compare:
        A = ov["A"]
        Hp = solve.orthogonalise(pb, A)
        be0, be1 = out["bounds_H"]
        t64 = fp64_plain_step_ms(pb, Hp.with_vals(cg.scale(Hp, be0, be1)))
        other_s = t_ms / args.steps / 1e3 - sum(p_ms) / 1e3 if p_ms else 0.0
        t_plain = 2 * (n_terms - 2) * t64 / 1e3 + other_s
        vs64 = {"fp64_step_ms": round(t64, 3), "fp64_plain_solve_s": round(t_plain, 1),
                "extrapolated": True, "how": f"12 timed FP64 steps x 2 passes x {n_terms - 2} steps + the "
                                             f"solve's other work", "solve_s": round(t_ms / args.steps / 1e3, 2),
                "speedup": round(t_plain / (t_ms / args.steps / 1e3), 2)}
    res = {
        "metric": METRIC, "value": round(value, 5), "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": round(t_ms / args.steps, 2), "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32" if prec == cg.F32 else "f64",
        "data": "synthetic (seeded atom-centred S/H generator; paper's BigDFT matrices unavailable)",
        "config": {"workload": args.workload, "form": form, "atoms_per_gpu": cfg["n_atoms"],
                   "rows": 4 * cfg["n_atoms"], "r_c": cfg["r_c"], "r_buf": cfg["r_buf"], "kT": cfg["kT"],
                   "N_e": cfg["N_e"], "fit_tol": cfg["tol"], "n_mu": cfg["n_mu"], "n_terms": n_terms,
                   "n_S": ov["n_S"], "blocks_P_H": nnz_H, "blocks_P_out": nnz_out, "triples": triples,
                   "products": "fp32" if prec == cg.F32 else "fp64",
                   "accumulators": "double-float pairs (FP32 pipe), returned as FP64" if prec == cg.F32 else "fp64",
                   "per_step_input": "H_k = H + 1e-4 k S (new Hamiltonian each step)",
                   "setup_outside_timed_region": "patterns, plans, gather plans, S^-1/2, G (fixed overlap)",
                   "setup_s": round(setup_s, 2), "patterns_and_plans_s": round(plans_s, 2),
                   "parallelism": f"replicas x{world}",
                   "atom_order": cfg.get("order") or "generator's (Morton)",
                   "l2": "inputs larger than L2 (no flush)"},
        "pass_ms": [round(x, 1) for x in p_ms],
        "roofline": roof,
        "e2e": None if e2e_value is None else {"value": round(e2e_value, 5), "unit": UNIT, "h2d_bytes_per_step": int(h2d),
                "d2h_bytes_per_step": int(d2h)},
        "gpu_launches": int(launches),
        "clocks": clocks,
        "vs_fp64_plain": vs64,
        "check": {"trace_FS_minus_N_e": float(out["trace_FS"].item()) - cfg["N_e"], "mu": out["mu"],
                  "passes": [o["passes"] for o in outs],
                  **({"mu_half_minus_mu_kT": (out["mu_half"]["mu"] - out["mu"]) / cfg["kT"]}
                     if form == "mu4" else {}),
                  **({"rounds_kT_n_E_Eprime_ok": out["rounds"], "dE_tol": cfg["dE_tol"]}
                     if form == "autokT" else {}),
                  **({"mu_hat": out["mu_hat"], "half_kT": out["half"] / cfg["kT"]} if form == "learned" else {})},
    }
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        res["cpu_baseline"] = cpu_baseline(sysm, cfg, n_terms, out.get("n_pass1", n_terms),
                                           [r[1] for r in out.get("rounds", [])[:-1]])
    if world > 1:
        dist.destroy_process_group()
    if rank == 0:
        print(json.dumps(res), flush=True)


# GB300 FP64: 304 DFMA lanes per cycle (152 SMs x 2, ncu peak_sustained) x 2 flops x 2070 MHz
FP64_NOMINAL_TFLOPS = 1.26


def step_roof(tflops: float, precision: str, column: bool) -> dict:
    """Roofline of the recursion for tflops of useful block-triple FLOPs: of the f16 digit
    products where the column kernel runs it, else of the FMA units (FP32 ones for the
    double-floats of f64x).  The ratio to the FMA unit of the precision stands beside it."""
    elem = "float" if precision == "f32" else "double"
    fp32 = SMS * FP32_LANES * 2 * MAX_SM_MHZ * 1e6 / 1e12
    unit = fp32 if precision == "f32" else FP64_NOMINAL_TFLOPS
    if column:
        n = DIGIT_PRODUCTS[elem]
        bound, peak, kernel = "tensor", MMA_F16_TFLOPS / n, f"k_colstep<{elem}>"
        src = f"f16 mma.sync, {MMA_F16_TFLOPS:.0f} TFLOP/s measured, over {n} digit products per product"
    else:
        bound, kernel = "alu", {"f32": "k_resident<float>", "f64": "k_step<double>", "f64x": "k_step<dfl>"}[precision]
        peak = FP64_NOMINAL_TFLOPS if precision == "f64" else fp32
        src = ("FP64 unit count: 304 DFMA lanes per cycle x 2 flops x 2070 MHz" if precision == "f64" else
               "FP32 FMA unit count: 152 SMs x 128 lanes x 2 flops x 2070 MHz")
    return {"bound": bound, "achieved": round(tflops, 3), "peak": round(peak, 3), "unit": "TFLOP/s",
            "frac": round(tflops / peak, 4), "kernel": kernel, "peak_source": src,
            f"vs_fp{32 if precision == 'f32' else 64}_unit_peak": round(tflops / unit, 4)}


def run_powers(args, rank: int, world: int, local: int):
    """Matrix powers: one step = S^a for every exponent from one FP64 recursion
    (bounds, degree, coefficients and the expansion)."""
    import torch
    import torch.distributed as dist

    import synth
    import paper_1704_00512_gb300 as cg
    from paper_1704_00512_gb300 import solve

    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if world > 1:
        dist.init_process_group("nccl", device_id=dev)
    cfg = WORKLOADS[args.workload]
    prec = cg.F64X if cfg["precision"] == "f64x" else cg.F64
    sysm = synth.make_system(cfg["n_atoms"], cfg["r_c"], seed=system_seed(rank))
    pb = solve.problem_from_system(sysm, cfg["r_buf"], dev, prec)

    def step(precision=prec):
        pb.build_patterns()
        return solve.powers(pb, exponents=cfg["exponents"], tol=cfg["tol"], n_max=512, precision=precision)

    for i in range(args.warmup):
        out = step()
        torch.cuda.synchronize()
        log(f"[rank {rank}] warmup {i}: n_terms={out['n_terms']} bounds={out['bounds']}")
    clk = ClockSampler(local, enabled=not args.no_clocks)
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    l0 = cg.launch_count()
    clk.start()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(args.steps):
        out = step()
    e1.record()
    torch.cuda.synchronize()
    clocks = clk.stop()
    launches = cg.launch_count() - l0
    t_ms = max_over_ranks(e0.elapsed_time(e1), world, dev)
    value = job_throughput(args.steps, world, t_ms)
    h_S = torch.from_numpy(np.ascontiguousarray(sysm.S)).pin_memory()
    h_out = [torch.empty(tuple(a.shape), dtype=torch.float64).pin_memory() for a in out["acc"]]
    torch.cuda.synchronize()
    f0, f1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    f0.record()
    for _ in range(args.e2e_steps):
        pb.S.vals.copy_(h_S, non_blocking=True)
        o = step()
        for h, a in zip(h_out, o["acc"]):
            h.copy_(a, non_blocking=True)
    f1.record()
    torch.cuda.synchronize()
    te_ms = max_over_ranks(f0.elapsed_time(f1), world, dev)
    n_terms = out["n_terms"]
    triples = count_triples(pb.P_H.row_ptr.cpu().numpy(), pb.P_H.col_idx.cpu().numpy(),
                            pb.P_out.row_ptr.cpu().numpy(), pb.P_out.col_idx.cpu().numpy())
    # FLOPs of the n-2 recursion steps over the whole step time (bounds and
    # coefficients included, so a lower bound on the kernel's rate)
    tflops = 2.0 * 64.0 * triples * (n_terms - 2) / (t_ms / args.steps / 1e3) / 1e12
    if prec == cg.F64X:
        # the same step in FP64 mode, timed here, and the distance between the two
        # results
        torch.cuda.synchronize()
        d0, d1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        d0.record()
        o64 = step(cg.F64)
        d1.record()
        torch.cuda.synchronize()
        ms64 = d0.elapsed_time(d1)
        rel = max(float(torch.linalg.norm(a - b) / torch.linalg.norm(b)) for a, b in zip(out["acc"], o64["acc"]))
        vs_f64 = {"f64_step_ms": round(ms64, 2), "f64x_step_ms": round(t_ms / args.steps, 2),
                  "speedup": round(ms64 / (t_ms / args.steps), 3), "max_relF_vs_fp64": rel}
    else:
        vs_f64 = None
    plan = pb.plan64 if prec == cg.F64 else pb.planX
    column = cg.plan_col_info(plan)[0] > 0 and plan._op_pattern[0] is pb.S.row_ptr
    roof = {**step_roof(tflops, cfg["precision"], column), "traffic": None}
    res = {
        "metric": METRIC, "value": round(value, 4), "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": round(t_ms / args.steps, 2), "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f64" if prec == cg.F64 else "f64x (FP64-accurate)",
        "data": "synthetic",
        "config": {"workload": args.workload, "atoms_per_gpu": cfg["n_atoms"], "rows": 4 * cfg["n_atoms"],
                   "r_c": cfg["r_c"], "r_buf": cfg["r_buf"], "exponents": list(cfg["exponents"]), "n_terms": n_terms,
                   "fit_tol": cfg["tol"], "blocks_P_H": pb.P_H.nnzb, "blocks_P_out": pb.P_out.nnzb,
                   "triples": triples, "l2": "inputs larger than L2 (no flush)"},
        "roofline": roof,
        "vs_f64": vs_f64,
        "e2e": None if args.e2e_steps == 0 else {
            "value": round(job_throughput(args.e2e_steps, world, te_ms), 4), "unit": UNIT,
            "h2d_bytes_per_step": int(h_S.numel() * 8), "d2h_bytes_per_step": int(sum(h.numel() for h in h_out) * 8)},
        "gpu_launches": int(launches), "clocks": clocks,
    }
    if world > 1:
        dist.destroy_process_group()
    if rank == 0:
        print(json.dumps(res), flush=True)


def batched_sizes(cfg) -> list[int]:
    rng = np.random.default_rng(0)
    return [int(x) for x in rng.integers(cfg["atoms_lo"], cfg["atoms_hi"] + 1, cfg["n_sys"])]


def run_batched(args, rank: int, world: int, local: int):
    """The batched workload: one step = the density matrices of all systems of the batch."""
    import torch
    import torch.distributed as dist

    import synth
    import paper_1704_00512_gb300 as cg
    from paper_1704_00512_gb300 import batched

    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if world > 1:
        dist.init_process_group("nccl", device_id=dev)
    cfg = WORKLOADS[args.workload]
    prec = cg.F32 if cfg["precision"] == "f32" else cg.F64
    t0 = time.time()
    sizes = batched_sizes(cfg)
    systems = [synth.make_system(n, cfg["r_c"], seed=system_seed(rank) * 1000 + i) for i, n in enumerate(sizes)]
    log(f"[rank {rank}] generated {len(systems)} systems, {sum(sizes)} atoms in {time.time() - t0:.1f}s")
    bp = batched.BatchedProblem(systems, cfg["r_buf"], dev, precision=prec, log=log)
    N_e = [2.0 * n for n in sizes]
    kw = dict(tol=cfg["tol"], tol_S=cfg["tol_S"])
    for i in range(args.warmup):
        tw = time.time()
        out = batched.foe_batched(bp, cfg["kT"], N_e, **kw)
        log(f"[rank {rank}] warmup {i}: {time.time() - tw:.2f}s captured={out['captured']} "
            f"n_terms {min(out['n_terms'])}..{max(out['n_terms'])} tiles={out['tiles']}")
    clk = ClockSampler(local, enabled=not args.no_clocks)
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    l0 = cg.launch_count()
    clk.start()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    passes = []
    e0.record()
    for _ in range(args.steps):
        tm = {}
        out = batched.foe_batched(bp, cfg["kT"], N_e, timings=tm, **kw)
        passes.append(tm["pass1_ms"] + tm["pass2_ms"])
    e1.record()
    torch.cuda.synchronize()
    clocks = clk.stop()
    launches = cg.launch_count() - l0
    t_ms = max_over_ranks(e0.elapsed_time(e1), world, dev)
    value = job_throughput(args.steps * len(systems), world, t_ms)
    # end to end: H values from pinned host memory, F and the traces back
    h_H = torch.from_numpy(np.concatenate([s.H for s in systems])).pin_memory()
    h_F = torch.empty(tuple(out["F"].shape), dtype=torch.float64).pin_memory()
    torch.cuda.synchronize()
    f0, f1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    f0.record()
    for _ in range(args.e2e_steps):
        bp.H.vals.copy_(h_H, non_blocking=True)
        o = batched.foe_batched(bp, cfg["kT"], N_e, **kw)
        h_F.copy_(o["F"], non_blocking=True)
    f1.record()
    torch.cuda.synchronize()
    te_ms = max_over_ranks(f0.elapsed_time(f1), world, dev)
    e2e_value = job_throughput(args.e2e_steps * len(systems), world, te_ms)
    # roofline of the batched launches: block triples of every system x terms
    triples = [count_triples(bp.PH[i].row_ptr.cpu().numpy(), bp.PH[i].col_idx.cpu().numpy(),
                             bp.Pout[i].row_ptr.cpu().numpy(), bp.Pout[i].col_idx.cpu().numpy())
               for i in range(len(systems))]
    flops = sum(2.0 * 64.0 * t * 2 * (n - 2) for t, n in zip(triples, out["n_terms"]))
    # (a batch runs on the column kernel from 48 operator blocks per block row on)
    column = bp.P_H.nnzb >= 48 * bp.P_H.nbr
    pass_s = statistics.mean(passes) / 1e3
    tflops = flops / pass_s / 1e12
    res = {
        "metric": METRIC, "value": round(value, 4), "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": round(t_ms / args.steps, 2), "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": cfg["precision"], "data": "synthetic",
        "config": {"workload": args.workload, "systems": len(systems), "atoms": sum(sizes),
                   "atoms_range": [min(sizes), max(sizes)], "r_c": cfg["r_c"], "r_buf": cfg["r_buf"],
                   "kT": cfg["kT"], "n_terms_range": [min(out["n_terms"]), max(out["n_terms"])],
                   "blocks_P_out": bp.P_out.nnzb, "blocks_P_H": bp.P_H.nnzb, "tiles": out["tiles"],
                   "graphs": "expansions, post-processing and traces captured and replayed; bisections eager", "l2": "inputs larger than L2 (no flush)"},
        "roofline": {**step_roof(tflops, cfg["precision"], column), "traffic": None},
        "pass_ms": round(statistics.mean(passes), 1),
        "e2e": {"value": round(e2e_value, 4), "unit": UNIT, "h2d_bytes_per_step": int(h_H.numel() * 8),
                "d2h_bytes_per_step": int(h_F.numel() * 8)},
        "gpu_launches": int(launches), "clocks": clocks,
        "check": {"max_abs_trace_error": float(np.max(np.abs(out["trace_FS"] - np.array(N_e))))},
    }
    if world > 1:
        dist.destroy_process_group()
    if rank == 0:
        print(json.dumps(res), flush=True)


# --------------------------------------------------------------------------
# the CPU oracle: baseline leg and reference arm
# --------------------------------------------------------------------------

def oracle_sample(sysm, cfg, n_products: int = 1):
    """Time n_products steps of the oracle's masked recursion on this system."""
    from oracle import ref
    S = ref.Bsr(sysm.row_ptr, sysm.col_idx, sysm.S)
    H = ref.Bsr(sysm.row_ptr, sysm.col_idx, sysm.H)
    rp, ci = ref.pattern(sysm.xyz, sysm.L, cfg["r_c"] + cfg["r_buf"])
    P_out = ref.Bsr(rp, ci, None)
    Ht = ref.scale(H, -10.0, 10.0)
    coeffs = np.ones((cfg["n_mu"], n_products + 2))
    t0 = time.perf_counter()
    ref.chebyshev_expand(Ht, P_out, coeffs, G=ref.identity(P_out) if cfg["n_mu"] == 1 else None)
    dt = time.perf_counter() - t0
    del S
    return dt / n_products, len(ci)


def oracle_threads() -> int:
    """Threads the oracle's OpenMP loops use (OMP_NUM_THREADS, else one per host core)."""
    try:
        return max(1, int(os.environ["OMP_NUM_THREADS"]))
    except (KeyError, ValueError):
        return os.cpu_count() or 1


def col_kernel_measured(text: str | None = None) -> bool:
    """Whether the column kernel's source (colstep.cu before its host section)
    is the one COL_TRAFFIC was measured on."""
    import hashlib
    if text is None:
        with open(os.path.join(ROOT, "paper_1704_00512_gb300", "csrc", "colstep.cu"), encoding="utf-8") as f:
            text = f.read()
    if COL_KERNEL_END not in text:
        return False
    kernel = text[:text.index(COL_KERNEL_END)]
    return hashlib.sha256(kernel.encode()).hexdigest() == COL_TRAFFIC["colstep_sha256"]


def col_traffic_per_launch(form: str, n_mu: int, launches_pass, nnz_out: int, measured: bool | None = None,
                           order: str | None = None):
    """Measured DRAM bytes per k_colstep launch of a 4-mu solve, scaled to this
    system's P_out blocks and averaged over the solve's two passes; None for
    other forms, another atom order, or when the kernel source differs from
    the measured one."""
    if form != "mu4" or n_mu != 4 or len(launches_pass) != 2 or order != COL_TRAFFIC["order"]:
        return None
    if not (col_kernel_measured() if measured is None else measured):
        return None
    scale = nnz_out / COL_TRAFFIC["blocks_P_out"]
    per = [COL_TRAFFIC["pass1_bytes"], COL_TRAFFIC["pass2_4acc_bytes"]]
    return int(scale * sum(b * n for b, n in zip(per, launches_pass)) / sum(launches_pass))


def solve_step_equivalents(n_terms: int, n_pass1: int, nnz_out: int, nnz_H: int) -> float:
    """Recursion-step equivalents of one solve for a new H: the moment pass of
    n_pass1 terms and the accumulation pass of n_terms, plus the four P_out x
    P_out products of the orthogonalisation and the post-processing, each
    nnz_out/nnz_H times a step (S^-1/2 and G belong to the fixed overlap)."""
    return (n_pass1 - 2) + (n_terms - 2) + 4 * nnz_out / nnz_H


def cpu_baseline(sysm, cfg, n_terms, n_pass1, earlier_solves=()) -> dict:
    """earlier_solves: term counts of two-pass solves that preceded the accepted
    one (the smearing loop), each counted as a whole solve."""
    t_step, nnz_out = oracle_sample(sysm, cfg, 1)
    eq = solve_step_equivalents(n_terms, n_pass1, nnz_out, sysm.nnzb)
    eq += sum(solve_step_equivalents(n, n, nnz_out, sysm.nnzb) for n in earlier_solves)
    return {"value": 1.0 / (t_step * eq), "unit": UNIT, "cores": oracle_threads(), "kind": "oracle",
            "extrapolated": True,
            "sample": f"1 FP64 oracle recursion step of the same system timed ({t_step:.2f}s), extrapolated by "
                      f"{eq:.0f} step-equivalents per solve"}


def run_reference_batched(args, cfg):
    """Reference arm of the batched workload: the oracle's step time on the
    median-size system, scaled per system by its blocks and step-equivalents."""
    import synth
    from oracle import ref
    sizes = batched_sizes(cfg)
    med = sorted(sizes)[len(sizes) // 2]
    sysm = synth.make_system(med, cfg["r_c"], seed=0)
    n_terms = ref.choose_degree(ref.Func(ref.KIND_FERMI, mu=0.0, kT=cfg["kT"]), -8.6, 8.6, cfg["tol"], 16384)
    n_S = ref.choose_degree(ref.Func(ref.KIND_POWER, a=-0.5), 0.03, 3.1, cfg["tol_S"], 512, rel=True)
    times = []
    for i in range(args.warmup + args.steps):
        t_step, nnz_out = oracle_sample(sysm, cfg, 1)
        if i >= args.warmup:
            times.append(t_step)
    # the batched solve expands S^-1/2 and runs two full passes for every system
    eq = 2 * (n_terms - 2) + (n_S - 2) + 6 * nnz_out / sysm.nnzb
    # work per system ~ its P_out blocks: n_atoms x min(n_atoms, neighbours within r_c + r_buf)
    rho = 200.0 / 18.0 ** 3
    nb = lambda n: n * min(n, 1 + rho * 4.0 / 3.0 * np.pi * (cfg["r_c"] + cfg["r_buf"]) ** 3)
    t_batch = statistics.mean(times) * eq * sum(nb(n) for n in sizes) / nb(med)
    value = len(sizes) / t_batch
    return value, t_batch, {"workload": args.workload, "systems": len(sizes), "atoms": sum(sizes),
                            "sample_atoms": med, "n_terms": n_terms, "n_S": n_S}, (
        f"per bench step one FP64 oracle recursion step of the median ({med}-atom) system, scaled by "
        f"{eq:.0f} step-equivalents and by the batch's P_out blocks")


def run_reference(args, rank: int, world: int):
    if rank != 0:
        return
    import synth
    cfg = WORKLOADS[args.workload]
    if cfg.get("powers"):
        from oracle import ref
        sysm = synth.make_system(cfg["n_atoms"], cfg["r_c"], seed=0)
        n_terms = max(ref.choose_degree(ref.Func(ref.KIND_POWER, a=a), 0.03, 3.1, cfg["tol"], 512, rel=True)
                      for a in cfg["exponents"])
        times = []
        for i in range(args.warmup + args.steps):
            t_step, _ = oracle_sample(sysm, cfg, 1)
            if i >= args.warmup:
                times.append(t_step)
        t_solve = statistics.mean(times) * (n_terms - 2)
        value = 1.0 / t_solve
        conf = {"workload": args.workload, "atoms_per_gpu": cfg["n_atoms"], "rows": 4 * cfg["n_atoms"],
                "n_terms": n_terms}
        sample = (f"per bench step one FP64 oracle recursion step of the same system with {len(cfg['exponents'])} "
                  f"accumulators, scaled by {n_terms - 2} steps")
        res = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
               "steps": args.steps, "warmup": args.warmup, "ms_per_step": t_solve * 1e3, "higher_is_better": True,
               "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic", "config": conf,
               "extrapolated": True,
               "cpu_baseline": {"value": value, "unit": UNIT, "cores": oracle_threads(), "kind": "oracle",
                                "sample": sample},
               "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
        print(json.dumps(res), flush=True)
        return
    if cfg.get("batched"):
        value, t_solve, conf, sample = run_reference_batched(args, cfg)
        res = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
               "steps": args.steps, "warmup": args.warmup, "ms_per_step": t_solve * 1e3, "higher_is_better": True,
               "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic", "config": conf,
               "extrapolated": True,
               "cpu_baseline": {"value": value, "unit": UNIT, "cores": oracle_threads(), "kind": "oracle",
                                "sample": sample},
               "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
        print(json.dumps(res), flush=True)
        return
    sysm = synth.make_system(cfg["n_atoms"], cfg["r_c"], seed=0)
    # term counts of the solve come from the oracle's own degree rule on a
    # representative interval; the sample times one recursion step per bench step
    from oracle import ref
    n_terms = ref.choose_degree(ref.Func(ref.KIND_FERMI, mu=0.0, kT=cfg["kT"]), -8.6, 8.6, cfg["tol"], 16384)
    n_pass1 = n_terms // 2 if cfg.get("form") == "mu4" else n_terms
    times = []
    for i in range(args.warmup + args.steps):
        t_step, nnz_out = oracle_sample(sysm, cfg, 1)
        if i >= args.warmup:
            times.append(t_step)
    eq = solve_step_equivalents(n_terms, n_pass1, nnz_out, sysm.nnzb)
    t_solve = statistics.mean(times) * eq
    value = 1.0 / t_solve
    res = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
           "steps": args.steps, "warmup": args.warmup, "ms_per_step": t_solve * 1e3, "higher_is_better": True,
           "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
           "extrapolated": True,
           "config": {"workload": args.workload, "atoms_per_gpu": cfg["n_atoms"], "rows": 4 * cfg["n_atoms"],
                      "n_terms": n_terms, "n_pass1": n_pass1,
                      "timing": "extrapolated: one timed oracle step per bench step x step-equivalents per solve"},
           "cpu_baseline": {"value": value, "unit": UNIT, "cores": oracle_threads(), "kind": "oracle",
                            "extrapolated": True,
                            "sample": f"per bench step one FP64 oracle recursion step of the same system, "
                                      f"extrapolated by {eq:.0f} step-equivalents per solve"},
           "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(res), flush=True)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=1)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["cheb", "reference"], default="cheb")
    ap.add_argument("--workload", choices=sorted(WORKLOADS), default=DEFAULT_WORKLOAD)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--e2e-steps", type=int, default=1, help="solves in the end-to-end (host buffers) loop")
    ap.add_argument("--no-clocks", action="store_true", help="do not sample nvidia-smi (e.g. under a profiler)")
    ap.add_argument("--no-fp64-compare", action="store_true", help="skip the timed FP64 steps of the plain form")
    args = ap.parse_args()
    if args.warmup < 3:
        log("note: fewer than 3 warm-up steps")
    rank, world, local = rank_env()
    if args.impl == "reference":
        run_reference(args, rank, world)
    elif WORKLOADS[args.workload].get("batched"):
        run_batched(args, rank, world, local)
    elif WORKLOADS[args.workload].get("powers"):
        run_powers(args, rank, world, local)
    else:
        run_cheb(args, rank, world, local)


if __name__ == "__main__":
    main()
