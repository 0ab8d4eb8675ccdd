#!/usr/bin/env python
"""Throughput of the GW+C core-level hot path on GB300: Sigma_c(w) points/s + chi0 TFLOP/s.

Default workload: the pentacene-sized synthetic molecule (1300 states, 73 occupied incl. twenty-two
1s cores, 4500 auxiliary functions, N_ov = 89 571) in the precision form (split-BF16 chi0 on the
tensor cores, FP32-accurate 3xTF32 factorisation of eps; FP64 residues, assembly, QP and cumulant).
One step is one pass of the whole path over a fixed, stated subset of that workload:
  - residency: the inputs reloaded into the resident context (precision copies of O, Sigma^x);
  - the imaginary-axis W table (33 real builds, factorisations and 28 600 contractions);
  - the decoupled Im Sigma of all 22 cores on the 800-point relative grid (one residue build per
    grid point with a residue, shared by the cores) and the cumulant spectrum of every core;
  - the G_dH W0 QP energies (Hedin shift) of cores 0, 11 and 21;
  - the full contour-deformation Sigma^c (-I + R) of all 22 cores at 4 of the 800 grid points.
Points per step = the (core, w) self-energy values the step produces (decoupled Im Sigma points,
full Sigma^c points, one Sigma^c(eps_n) per QP core), broken down in the JSON line.
--workload benzene runs the whole benzene-sized job per step (all cores on the full grid).

  python bench.py [--gpus N] [--steps K] [--warmup W] [--prec bf16x3|bf16x3f64|fp32|fp64|bf16]
  python bench.py --impl reference     # the FP64 CPU oracle on a bounded sample, same metric

Under torchrun every rank runs an independent replica on its own GPU (the path needs no
exchange between GPUs); value = points of all ranks / max-over-ranks time.
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "core Sigma_c(w) points/s (whole GW+C step) + chi0 TFLOP/s"
UNIT = "points/s"
HARTREE_EV = 27.211386245988


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="gwc", choices=["gwc", "reference"])
    ap.add_argument("--prec", default="bf16x3", choices=["bf16x3", "bf16x3f64", "bf16", "fp32", "fp64"])
    ap.add_argument("--workload", default="pentacene",
                    choices=["pentacene", "benzene", "tiny", "pentacene-forms", "batch", "serve"])
    ap.add_argument("--no-fp64-path", action="store_true", help="pentacene: skip the FP64 GPU path sample")
    ap.add_argument("--molecules", type=int, default=48, help="batched form: molecules in the graph")
    ap.add_argument("--omega-points", type=int, default=800, help="batched/serving/pentacene: grid points")
    ap.add_argument("--requests", type=int, default=2000, help="serving form: requests in the stream")
    ap.add_argument("--rate", type=float, default=20.0, help="serving form: mean arrival rate (1/s)")
    ap.add_argument("--slots", type=int, default=8, help="serving form: requests in flight at most")
    ap.add_argument("--time-limit", type=float, default=900.0, help="serving form: stop after this many seconds")
    ap.add_argument("--fp64-points", type=int, default=1,
                    help="pentacene form: grid points for the FP64 path (0: mixed path only)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-fp64-check", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--batch", type=int, default=0, help="frequencies per internal batch (0: from free memory)")
    return ap.parse_args()


def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def make_workload(name):
    from paper_2412_17132_gb300 import synth

    return synth.benzene() if name == "benzene" else synth.tiny()


def describe(mol):
    return (f"{mol.name}-sized synthetic molecule: N_states={mol.n_states}, N_occ={mol.n_occ}, N_core={mol.n_core}, "
            f"N_aux={mol.n_aux}, N_ov={mol.n_occ * mol.n_virt}, {mol.omega.size} real omega over 30 eV, "
            f"{mol.n_im} imaginary nodes, eta={mol.eta} Ha, cumulant n_t={mol.n_t}, t_max={mol.t_max}")


# ------------------------------------------------------------------------------------------
# clocks sampled during the timed region
# ------------------------------------------------------------------------------------------
class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
              "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
              "clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.gpu = gpu_index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--id={self.gpu}", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except Exception:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        rows = [l.split(",") for l in self.lines if l]
        sm, smax, reasons = [], 0.0, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for r in rows:
            try:
                sm.append(float(r[1]))
                smax = max(smax, float(r[2]))
                for nm, v in zip(names, r[5:9]):
                    if v.strip().lower() == "active":
                        reasons.add(nm)
            except Exception:
                continue
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": smax, "reasons": sorted(reasons), "samples": len(sm)}


# ------------------------------------------------------------------------------------------
# CPU oracle timing (cpu_baseline leg and --impl reference)
# ------------------------------------------------------------------------------------------
def oracle_sample(mol, n_points=2, qp_builds=0):
    """Time the FP64 oracle on a bounded sample and extrapolate to the whole step.

    Sample: the imaginary-axis W table (n_im + 1 real builds, all states x cores) plus the
    self-energy of all cores at n_points grid frequencies. The full step is extrapolated as
    T_table + T_build * (residue builds of the grid + of the QP), where T_build is the measured
    time per residue build (chi0 + LU solve with N_core right-hand sides).
    """
    import numpy as np

    from oracle import gwc_oracle as G

    s = G.System.from_molecule(mol)
    t0 = time.perf_counter()
    s.w_imag_table()
    t_table = time.perf_counter() - t0
    idx = np.linspace(0, mol.omega.size - 1, n_points).round().astype(int)
    builds = 0
    t1 = time.perf_counter()
    for j in idx:
        w = float(mol.omega[j])
        builds += sum(1 for m in range(mol.n_states) if G.residue_prefactor(mol.eps[m], w, s.eps_f) != 0.0)
        s.sigma_c(w)
    t_pts = time.perf_counter() - t1
    t_build = t_pts / max(1, builds)
    grid_builds = sum(
        1 for w in mol.omega for m in range(mol.n_states) if G.residue_prefactor(mol.eps[m], float(w), s.eps_f) != 0.0)
    t_full = t_table + t_build * (grid_builds + qp_builds)
    points = mol.n_core * mol.omega.size
    return {
        "value": points / t_full,
        "t_full_s": t_full,
        "t_table_s": t_table,
        "t_build_s": t_build,
        "measured_s": t_table + t_pts,
        "sample": (f"FP64 oracle: imaginary-axis W table ({mol.n_im}+1 nodes) + Sigma of all {mol.n_core} cores at "
                   f"{n_points} of {mol.omega.size} grid points ({builds} residue builds); extrapolated to the whole step "
                   f"({grid_builds} grid + {qp_builds} QP residue builds) as T_table + builds * T_build"),
    }


def cpu_threads():
    """Threads the oracle's BLAS runs on: threadpoolctl's answer, else the thread-count variables
    the BLAS libraries honour, else every host core."""
    try:
        from threadpoolctl import threadpool_info

        n = [d.get("num_threads") for d in threadpool_info() if d.get("user_api") == "blas"]
        if n and n[0]:
            return int(n[0])
    except Exception:
        pass
    env = [int(os.environ[k]) for k in ("OPENBLAS_NUM_THREADS", "OMP_NUM_THREADS", "MKL_NUM_THREADS")
           if os.environ.get(k, "").isdigit() and int(os.environ[k]) > 0]
    return min(env) if env else os.cpu_count()


def run_reference(args):
    ws, rank, _ = dist_env()
    if rank != 0:
        return 0
    if args.workload == "pentacene":
        print(json.dumps(run_reference_pentacene(args)), flush=True)
        return 0
    mol = make_workload(args.workload)
    for _ in range(args.warmup):
        oracle_sample(mol, n_points=1)
    vals, times = [], []
    for _ in range(args.steps):
        t0 = time.perf_counter()
        r = oracle_sample(mol, n_points=1)
        times.append(time.perf_counter() - t0)
        vals.append(r["value"])
    value = statistics.mean(vals)
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": 1e3 * statistics.mean(times), "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": describe(mol), "implementation": "FP64 CPU oracle (numpy/LAPACK), bounded sample per step"},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": cpu_threads(), "kind": "oracle", "sample": r["sample"]},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


# ------------------------------------------------------------------------------------------
# GPU arm
# ------------------------------------------------------------------------------------------
def load_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        return d, "measured"
    return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0, "sm_max_mhz": 2070.0}, "fallback"


def load_traffic(kernel, workload, units_per_launch):
    """DRAM bytes per launch from the committed ncu capture, scaled to this run's units per launch
    (traffic of these kernels grows in proportion to the matrices / frequencies a launch processes)."""
    p = os.path.join(ROOT, "profiles", "traffic.json")
    if not os.path.exists(p) or not units_per_launch:
        return None
    with open(p) as f:
        d = json.load(f)
    e = d.get(kernel)
    if e and e.get("workload") == workload and e.get("source_unchanged", True):
        return e["bytes_per_unit"] * units_per_launch
    return None


def chi0_kernel_info(n_aux, n_ov):
    """The tensor-core chi0 kernel the library runs (CTA pairs unless GWC_CHI0_KERNEL=single): its name and the
    ratio of the MMA work of a lower triangle covered by 256-row blocks from row 0 (the one-CTA kernel: 128 x 128
    tiles) to the algorithmic N_aux (N_aux + 1) N_ov per part. The pair kernel's launch is chi0_executed_ratio."""
    n_aux_pad = -(-n_aux // 128) * 128
    n_ov_pad = -(-n_ov // 64) * 64
    nqb = n_aux_pad // 128
    if os.environ.get("GWC_CHI0_KERNEL", "") == "single":
        tiles, name = nqb * (nqb + 1) / 2, "chi0_tc_kernel"
    else:
        npb = -(-n_aux_pad // 256)
        tiles, name = 2 * (npb * (npb - 1) + min(2 * npb, nqb)), "chi0_pair_kernel"
    return name, tiles * 128 * 128 * 2 * n_ov_pad / (n_aux * (n_aux + 1.0) * n_ov)


def chi0_executed_ratio(n_aux, n_ov):
    """Executed MMA work of the chi0 kernel the library runs, over the algorithmic N_aux (N_aux + 1) N_ov per part: the
    pair kernel's 256 x 128 tiles start at any 128-row block, so the Q block q of n takes (n - q + 1) // 2 of them."""
    nqb = -(-n_aux // 128)
    if chi0_kernel_info(n_aux, n_ov)[0] != "chi0_pair_kernel":
        return chi0_kernel_info(n_aux, n_ov)[1]
    tiles = 2 * sum((nqb - q + 1) // 2 for q in range(nqb))
    return tiles * 128 * 128 * 2 * (-(-n_ov // 64) * 64) / (n_aux * (n_aux + 1.0) * n_ov)


def job_throughput(local_ms, local_units, pg=None, device=None):
    """Whole-job aggregate over the ranks of a replica run: the slowest rank's time (max over ranks)
    and the units all ranks processed; value = units / slowest time (units/s). Each rank's units
    are its own (no data exchange), so the sum is the job's work. pg: torch.distributed or None."""
    if pg is None:
        return float(local_ms), float(local_units), local_units / (local_ms * 1e-3)
    import torch

    t = torch.tensor([float(local_ms)], dtype=torch.float64, device=device)
    u = torch.tensor([float(local_units)], dtype=torch.float64, device=device)
    pg.all_reduce(t, op=pg.ReduceOp.MAX)
    pg.all_reduce(u, op=pg.ReduceOp.SUM)
    ms, units = float(t.item()), float(u.item())
    return ms, units, units / (ms * 1e-3)


def run_gpu(args):
    import numpy as np
    import torch

    from paper_2412_17132_gb300 import gwc

    ws, rank, local = dist_env()
    torch.cuda.set_device(local)
    pg = None
    if ws > 1:
        import torch.distributed as dist

        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
        pg = dist
    mol = make_workload(args.workload)
    nc, nw = mol.n_core, mol.omega.size
    dev = torch.device("cuda", local)
    eps_d = torch.as_tensor(mol.eps, device=dev)
    oov_d = torch.as_tensor(mol.o_ov, device=dev)
    ocore_d = torch.as_tensor(mol.o_core, device=dev)
    eps_h = torch.as_tensor(mol.eps).pin_memory()
    oov_h = torch.as_tensor(mol.o_ov).pin_memory()
    ocore_h = torch.as_tensor(mol.o_core).pin_memory()
    w_rel = torch.as_tensor(mol.omega[None, :] - mol.eps[mol.core_idx][:, None], device=dev).contiguous()
    ctx = gwc.Context(eps_d, mol.n_occ, mol.core_idx, oov_d, ocore_d, prec=args.prec, eta=mol.eta, n_im=mol.n_im,
                      xi0=mol.xi0, n_t=mol.n_t, t_max=mol.t_max, batch=args.batch, profile=True)
    sig = torch.empty((nc, nw, 2), dtype=torch.float64, device=dev)
    dec = torch.empty((nc, nw), dtype=torch.float64, device=dev)
    sx = torch.empty((nc,), dtype=torch.float64, device=dev)
    eqp = torch.empty((nc,), dtype=torch.float64, device=dev)
    dh = torch.empty_like(eqp)
    its = torch.empty((nc,), dtype=torch.int32, device=dev)
    a = torch.empty((nc, mol.n_t), dtype=torch.float64, device=dev)
    nu = torch.empty((mol.n_t,), dtype=torch.float64, device=dev)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)  # 256 MB > L2 (129 MB)
    sig_h = torch.empty(sig.shape, dtype=sig.dtype).pin_memory()
    eqp_h = torch.empty(eqp.shape, dtype=eqp.dtype).pin_memory()
    a_h = torch.empty(a.shape, dtype=a.dtype).pin_memory()

    def step(host=False):
        if host:
            ctx.load(eps_h.numpy(), oov_h.numpy(), ocore_h.numpy(), core_idx=mol.core_idx)
        else:
            ctx.load(eps_d, oov_d, ocore_d, core_idx=mol.core_idx)
        ctx.sigma_core(mol.omega, out=(sig, dec, sx))
        ctx.qp_solve(out=(eqp, dh, its))
        ctx.cumulant_spectrum(w_rel, dec, out=(a, nu))
        if host:  # results back through the C ABI (gwc_copy_out)
            ctx.copy_out(sig_h, sig)
            ctx.copy_out(eqp_h, eqp)
            ctx.copy_out(a_h, a)

    stream = torch.cuda.current_stream()
    for _ in range(max(3, args.warmup)):
        step()
    ctx.sync()

    def barrier():
        torch.cuda.synchronize()
        if pg is not None:
            pg.barrier()

    # ---- timed region: device-resident inputs -------------------------------------------------
    ctx.reset_stats()
    clocks = ClockSampler(local)
    barrier()
    clocks.start()
    times = []
    for _ in range(args.steps):
        flush.zero_()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        step()
        e1.record(stream)
        e1.synchronize()
        times.append(e0.elapsed_time(e1))
    barrier()
    clk = clocks.stop()
    ctx.sync()
    st = ctx.stats()
    total_ms, points, value = job_throughput(sum(times), nc * nw * args.steps, pg, dev)

    # ---- e2e: host buffers through the C ABI, copies inside the timed region ---------------
    e2e = None
    if not args.no_e2e:
        barrier()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(args.steps):
            step(host=True)
        e1.record(stream)
        e1.synchronize()
        _, _, e2e_value = job_throughput(e0.elapsed_time(e1), nc * nw * args.steps, pg, dev)
        h2d = mol.eps.nbytes + mol.o_ov.nbytes + mol.o_core.nbytes
        d2h = sig.numel() * 8 + eqp.numel() * 8 + a.numel() * 8
        e2e = {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": int(h2d),
               "d2h_bytes_per_step": int(d2h)}

    out = None
    if rank == 0:
        peaks, src = load_peaks()
        chi0_t = st["chi0_ms"] * 1e-3
        fac_t = st["factor_ms"] * 1e-3
        chi0_alg = st["chi0_flop"] / chi0_t if chi0_t > 0 else 0.0
        # executed tensor-core work per algorithmic flop: the kernel's whole tiles of the padded lower
        # triangle over the padded contraction (64-wide chunks), times the products per split (3 for bf16x3)
        n_ov = mol.n_occ * mol.n_virt
        kname, tile_ratio = chi0_kernel_info(mol.n_aux, n_ov)[0], chi0_executed_ratio(mol.n_aux, n_ov)
        mma_mult = {"bf16x3": 3.0, "bf16": 1.0}.get(args.prec, 0.0) * tile_ratio
        if chi0_t >= fac_t and args.prec in ("bf16x3", "bf16"):
            peak = peaks.get("bf16_tflops_sustained", peaks.get("bf16_tflops"))
            roof = {"kernel": kname + " (tcgen05 " + args.prec + ")", "bound": "tensor", "achieved": chi0_alg / 1e12,
                    "peak": peak, "unit": "TFLOP/s", "frac": chi0_alg / 1e12 / peak,
                    "traffic": load_traffic(kname, mol.name, st["chi0_builds"] / max(1, st["chi0_launches"])),
                    "mma_frac": mma_mult * chi0_alg / 1e12 / peak,
                    "peak_source": f"{src} bf16 sustained (kernel timed inside a long step)",
                    "share_of_step": chi0_t / (total_ms * 1e-3)}
        else:
            clk_mhz = peaks.get("sm_max_mhz", 2070.0)
            fp32_peak = 152 * 128 * 2 * clk_mhz * 1e6 / 1e12
            fac_alg = st["factor_flop"] / fac_t if fac_t > 0 else 0.0
            units = st["factorizations"] / max(1, st["factor_launches"])
            tc_factor = args.prec in ("bf16x3", "bf16") and os.environ.get("GWC_FACTOR", "") != "simt"
            if tc_factor:
                # trailing updates on the tensor cores in 3xTF32: three TF32 products per FP32-accurate one
                tf32 = peaks.get("bf16_tflops_sustained", peaks.get("bf16_tflops")) * 1.1 / 2.25
                peak = tf32 / 3.0
                split = os.environ.get("GWC_FACTOR", "") != "tc"
                roof = {"kernel": ("ldlt_update_kernel + ldlt_diag_kernel + ldlt_rows_kernel (complex-symmetric LDL^T per 64-column "
                                   "panel over the batch: tcgen05 3xTF32 updates + SIMT panels)") if split else
                                  ("ldlt_tc_kernel (batched complex-symmetric LDL^T, FP32: tcgen05 3xTF32 trailing "
                                   "updates + SIMT panels)"),
                        "bound": "tensor", "achieved": fac_alg / 1e12, "peak": peak, "unit": "TFLOP/s",
                        "frac": fac_alg / 1e12 / peak, "alu_frac": fac_alg / 1e12 / fp32_peak,
                        "traffic": None if split else load_traffic("ldlt_tc_kernel", mol.name, units),
                        "peak_source": f"{src} bf16 sustained x 1.1/2.25 (nominal TF32/BF16 dense) / 3 (3xTF32)",
                        "share_of_step": fac_t / (total_ms * 1e-3)}
            else:
                peak = fp32_peak if args.prec != "fp64" else 1.2
                roof = {"kernel": "ldlt_kernel (batched complex-symmetric LDL^T, " +
                                  ("FP64" if args.prec == "fp64" else "FP32") + ")",
                        "bound": "alu", "achieved": fac_alg / 1e12, "peak": peak, "unit": "TFLOP/s",
                        "frac": fac_alg / 1e12 / peak,
                        "traffic": load_traffic("ldlt_kernel", mol.name, units),
                        "peak_source": ("FP32 ALU: 152 SMs x 128 lanes x 2 flop x max SM clock" if args.prec != "fp64"
                                        else "FP64 FMA loop measured on this GB300 (1.20 TFLOP/s)"),
                        "share_of_step": fac_t / (total_ms * 1e-3)}
        lat = sorted(times)
        out = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": total_ms / args.steps, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": {"bf16x3": "bf16x3+f32+f64", "bf16": "bf16+f32+f64", "fp32": "f32+f64", "fp64": "f64"}[args.prec],
            "data": "synthetic",
            "config": {"workload": describe(mol), "precision": args.prec, "parallelism": f"replicas x{ws}",
                       "l2": "256 MB written between timed steps (L2 flushed)", "full_sigma": "all cores, all grid points",
                       "qp": "G_dH W0 secant on device", "spectrum": "decoupled, one per core"},
            "roofline": roof,
            "chi0_tflops": {"algorithmic": chi0_alg / 1e12, "gemm_equivalent": 2 * chi0_alg / 1e12,
                            "mma_executed": mma_mult * chi0_alg / 1e12 if mma_mult else None,
                            "note": "algorithmic = lower triangle, N_aux(N_aux+1) N_ov flop per real part"},
            "latency_ms": {"p50": lat[len(lat) // 2], "p99": lat[min(len(lat) - 1, int(math.ceil(0.99 * len(lat))) - 1)],
                           "per_step": times},
            "kernel_time_share": {"chi0": st["chi0_ms"] / total_ms, "factor": st["factor_ms"] / total_ms,
                                  "solve": st["solve_ms"] / total_ms},
            "gpu_launches": int(st["kernel_launches"]),
            "clocks": clk,
            "e2e": e2e,
            "qp": {"eps_qp_Ha": eqp.cpu().tolist(), "dH_Ha": dh.cpu().tolist(), "iters": its.cpu().tolist()},
        }
    # ---- CD-WAC beside CD (the paper's analytic continuation of W; one call, not the metric) ------
    if rank == 0:
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        wsig, wdec = ctx.sigma_core_wac(mol.omega)
        torch.cuda.synchronize()
        t_wac = time.perf_counter() - t0
        d = (wsig - sig).abs().amax(dim=2)  # [n_core][n_w]
        near = torch.as_tensor(np.abs(mol.omega - mol.eps[mol.core_idx].mean()) * HARTREE_EV < 2.0, device=dev)
        out["cdwac"] = {"seconds": t_wac, "points_per_s": nc * nw / t_wac,
                        "max_dev_from_cd_Ha_within_2eV_of_core": float(d[:, near].max()),
                        "max_dev_from_cd_Ha_all": float(d.max()),
                        "reference_points": "100 core-region (0-40 eV) + 100 valence-region real points + imaginary nodes"}
    ctx.close()

    # ---- accuracy vs the plain FP64 GPU path (QP) and its points/s on a subset -------------------
    if rank == 0 and not args.no_fp64_check and args.prec != "fp64":
        c64 = gwc.Context(eps_d, mol.n_occ, mol.core_idx, oov_d, ocore_d, prec="fp64", eta=mol.eta, n_im=mol.n_im,
                          xi0=mol.xi0, n_t=mol.n_t, t_max=mol.t_max)
        e64, dh64, _ = c64.qp_solve()
        sub = mol.omega[np.linspace(0, nw - 1, 8).round().astype(int)]
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        s64, _, _ = c64.sigma_core(sub)
        c64.sync()
        t64 = time.perf_counter() - t0
        sig_sub = sig[:, np.linspace(0, nw - 1, 8).round().astype(int), :]
        out["vs_fp64_gpu"] = {
            "qp_max_abs_err_eV": float((eqp - e64).abs().max()) * HARTREE_EV,
            "sigma_max_abs_err_Ha_at_8_points": float((sig_sub - s64).abs().max()),
            "fp64_path_points_per_s": nc * sub.size / t64,
            "fp64_path_sample": f"Sigma of all cores at 8 grid points (W table cached), FP64 chi0 + FP64 LDL^T",
        }
        c64.close()

    if rank == 0 and ws == 1 and not args.no_cpu_baseline:
        qp_builds = int(sum(int(i) + 1 for i in out["qp"]["iters"])) * mol.n_occ
        r = oracle_sample(mol, n_points=6, qp_builds=qp_builds)  # ~10 s of CPU work on 16 host cores
        out["cpu_baseline"] = {"value": r["value"], "unit": UNIT, "cores": cpu_threads(), "kind": "oracle",
                               "sample": r["sample"], "measured_s": r["measured_s"]}
    if rank == 0:
        print(json.dumps(out), flush=True)
    if pg is not None:
        pg.barrier()
        pg.destroy_process_group()
    return 0


# ------------------------------------------------------------------------------------------
# Default workload: the pentacene-sized precision form, a fixed subset of the job per step
# ------------------------------------------------------------------------------------------
PENT_SIGMA_IDX = [100, 300, 500, 700]  # grid points of the full Sigma^c (100 and 700 are in the oracle file)
PENT_QP_CORES = [0, 11, 21]  # cores whose QP energy the step computes (the oracle file's)
PENT_N_OMEGA = 800


def pent_grid_rel():
    import numpy as np

    return np.linspace(-25.0 / HARTREE_EV, 5.0 / HARTREE_EV, PENT_N_OMEGA)


def pentacene_mol(device):
    from paper_2412_17132_gb300 import synth

    return synth.pentacene_device() if device else synth.pentacene()


def pent_step_builds(eps, n_occ, core_idx, omega):
    """Residue builds one pentacene step does, by phase (bookkeeping for the extrapolations of the
    FP64 GPU path and the CPU oracle): a build per residue pair with a nonzero prefactor f_m, Theta(0) = 1/2."""
    import numpy as np

    ef = 0.5 * (eps[n_occ - 1] + eps[n_occ])

    def nz(m, w):
        th = lambda x: 1.0 if x > 0 else (0.0 if x < 0 else 0.5)  # noqa: E731
        return -th(ef - eps[m]) * th(eps[m] - w) + th(eps[m] - ef) * th(w - eps[m]) != 0.0

    dec = int(np.sum(pent_grid_rel() <= 0.0))  # occupied cores: a residue for w - eps_c <= 0
    qp = sum(1 for c in PENT_QP_CORES for m in range(eps.size) if nz(m, float(eps[core_idx[c]])))
    sig = sum(1 for j in PENT_SIGMA_IDX for m in range(eps.size) if nz(m, float(omega[j])))
    return {"table": 33, "decoupled": dec, "qp": qp, "sigma": sig}


def pent_points(n_core):
    full = n_core * len(PENT_SIGMA_IDX)
    return {"decoupled_im_sigma": n_core * PENT_N_OMEGA, "full_sigma": full, "qp_sigma": len(PENT_QP_CORES),
            "total": n_core * PENT_N_OMEGA + full + len(PENT_QP_CORES)}


def pent_oracle_sample(mol_host, builds, t_node=None):
    """FP64 oracle on the pentacene-sized system: one residue build (chi0 at x + i eta, LU solve with the
    22 core right-hand sides) and, unless t_node is given, one imaginary-axis node (real chi0, LU solve
    with all 28 600 right-hand sides of the W table), timed; the step extrapolated as
    33 T_node + residue builds x T_build."""
    from oracle import gwc_oracle as G

    s = G.System.from_molecule(mol_host)
    t0 = time.perf_counter()
    s.w_residue(30, abs(float(mol_host.eps[30]) - float(mol_host.omega[PENT_SIGMA_IDX[0]])))
    t_build = time.perf_counter() - t0
    measured = t_build
    if t_node is None:
        rhs = s.o_core.reshape(s.n_states * s.n_core, -1).T
        t1 = time.perf_counter()
        G.screened_wc(G.chi0(s.o_ov, s.delta, 1j * float(s.xi[0])).real, rhs)
        t_node = time.perf_counter() - t1
        measured += t_node
    n_res = builds["decoupled"] + builds["qp"] + builds["sigma"]
    t_step = builds["table"] * t_node + n_res * t_build
    pts = pent_points(mol_host.n_core)["total"]
    return {"value": pts / t_step, "t_step_s": t_step, "t_build_s": t_build, "t_node_s": t_node,
            "measured_s": measured,
            "sample": (f"FP64 oracle on the pentacene-sized system: one residue build (chi0 + LU, 22 right-hand sides) "
                       f"and one imaginary-axis node (chi0 + LU, {s.n_states * s.n_core} right-hand sides) timed; the step "
                       f"extrapolated as {builds['table']} nodes + {n_res} residue builds")}


def host_copy(mol):
    """The device-generated molecule with its arrays on the host (numpy), for the CPU oracle."""
    import copy

    h = copy.copy(mol)
    h.o_ov = mol.o_ov.cpu().numpy()
    h.o_core = mol.o_core.cpu().numpy()
    return h


def run_reference_pentacene(args):
    import torch

    dev = torch.cuda.is_available()
    mol = pentacene_mol(dev)
    mh = host_copy(mol) if dev else mol
    del mol
    builds = pent_step_builds(mh.eps, mh.n_occ, mh.core_idx, mh.omega)
    # the imaginary-axis node once (in the first warm-up step), then one residue build per step
    t_node = pent_oracle_sample(mh, builds)["t_node_s"]
    for _ in range(max(0, args.warmup - 1)):
        pent_oracle_sample(mh, builds, t_node)
    vals, times = [], []
    for _ in range(args.steps):
        t0 = time.perf_counter()
        r = pent_oracle_sample(mh, builds, t_node)
        times.append(time.perf_counter() - t0)
        vals.append(r["value"])
    value = statistics.mean(vals)
    return {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": 1e3 * statistics.mean(times), "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": describe_pent(mh), "implementation": "FP64 CPU oracle (numpy/LAPACK), bounded sample per step",
                   "step": pent_step_text(), "residue_builds_per_step": builds},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": cpu_threads(), "kind": "oracle", "sample": r["sample"]},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }


def describe_pent(mol):
    return (f"pentacene-sized synthetic molecule: N_states={mol.n_states}, N_occ={mol.n_occ}, N_core={mol.n_core}, "
            f"N_aux={mol.n_aux}, N_ov={mol.n_occ * mol.n_virt}, {PENT_N_OMEGA} real omega over 30 eV, {mol.n_im} imaginary "
            f"nodes, eta={mol.eta} Ha, cumulant n_t={mol.n_t}, t_max={mol.t_max}")


def pent_step_text():
    return ("reload of the inputs; imaginary-axis W table; decoupled Im Sigma of all cores on the 800-point relative grid "
            "and their cumulant spectra; G_dH W0 QP (Hedin shift) of cores " + ", ".join(map(str, PENT_QP_CORES)) +
            "; full CD Sigma^c of all cores at grid points " + ", ".join(map(str, PENT_SIGMA_IDX)))


def run_pentacene_headline(args):
    import numpy as np
    import torch

    from paper_2412_17132_gb300 import gwc

    ws, rank, local = dist_env()
    torch.cuda.set_device(local)
    pg = None
    if ws > 1:
        import torch.distributed as dist

        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
        pg = dist
    dev = torch.device("cuda", local)
    mol = pentacene_mol(True)
    nc, nt = mol.n_core, mol.n_t
    eps_d = torch.as_tensor(mol.eps, device=dev)
    oov_d, ocore_d = mol.o_ov, mol.o_core
    grid_rel = pent_grid_rel()
    pts = mol.omega[PENT_SIGMA_IDX]
    builds = pent_step_builds(mol.eps, mol.n_occ, mol.core_idx, mol.omega)
    npts = pent_points(nc)
    ctx = gwc.Context(eps_d, mol.n_occ, mol.core_idx, oov_d, ocore_d, prec=args.prec, qp_mode="hedin", eta=mol.eta,
                      n_im=mol.n_im, xi0=mol.xi0, n_t=nt, t_max=mol.t_max, batch=args.batch, profile=True)
    ctx.request_plan(grid_rel)
    ctx.set_qp_cores(PENT_QP_CORES)
    sig = torch.empty((nc, len(pts), 2), dtype=torch.float64, device=dev)
    sx = torch.empty((nc,), dtype=torch.float64, device=dev)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)  # 256 MB > L2 (129 MB)
    # e2e buffers: inputs and results in pinned host memory
    eps_h = torch.as_tensor(mol.eps).pin_memory()
    oov_h = torch.empty(oov_d.shape, dtype=torch.float64).pin_memory()
    ocore_h = torch.empty(ocore_d.shape, dtype=torch.float64).pin_memory()
    oov_h.copy_(oov_d)
    ocore_h.copy_(ocore_d)
    res_h = [torch.empty(nc, dtype=torch.float64).pin_memory(), torch.empty(nc, dtype=torch.float64).pin_memory(),
             torch.empty(nc, dtype=torch.int32).pin_memory(),
             torch.empty((nc, PENT_N_OMEGA), dtype=torch.float64).pin_memory(),
             torch.empty((nc, nt), dtype=torch.float64).pin_memory(), torch.empty(nt, dtype=torch.float64).pin_memory()]
    sig_h = torch.empty(sig.shape, dtype=torch.float64).pin_memory()

    def step(host=False):
        if host:
            ctx.load(eps_h.numpy(), oov_h.numpy(), ocore_h.numpy(), core_idx=mol.core_idx)
        else:
            ctx.load(eps_d, oov_d, ocore_d, core_idx=mol.core_idx)
        ctx.request_step()  # table, QP of the selected cores, decoupled residues, spectra
        ctx.sigma_core(pts, want_dec=False, out=(sig, None, sx))  # full Sigma^c (the table is reused)
        if host:  # results back through the C ABI
            ctx.request_results(out=res_h)
            ctx.copy_out(sig_h, sig)

    stream = torch.cuda.current_stream()
    for _ in range(max(3, args.warmup)):
        step()
    ctx.sync()

    def barrier():
        torch.cuda.synchronize()
        if pg is not None:
            pg.barrier()

    ctx.reset_stats()
    clocks = ClockSampler(local)
    barrier()
    clocks.start()
    times = []
    for _ in range(args.steps):
        flush.zero_()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        step()
        e1.record(stream)
        e1.synchronize()
        times.append(e0.elapsed_time(e1))
    barrier()
    clk = clocks.stop()
    ctx.sync()
    st = ctx.stats()
    total_ms, units, value = job_throughput(sum(times), npts["total"] * args.steps, pg, dev)
    res_d = ctx.request_results()  # device copies of the last step's results
    eqp, dh = res_d[0].cpu().numpy(), res_d[1].cpu().numpy()
    im_dec = res_d[3]
    a_spec = res_d[4]
    sig_last = sig.cpu().numpy()

    e2e = None
    if not args.no_e2e:
        k = min(2, args.steps)
        barrier()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(k):
            step(host=True)
        e1.record(stream)
        e1.synchronize()
        _, _, e2e_value = job_throughput(e0.elapsed_time(e1), npts["total"] * k, pg, dev)
        h2d = mol.eps.nbytes + oov_h.numel() * 8 + ocore_h.numel() * 8
        d2h = sum(t.numel() * t.element_size() for t in res_h) + sig_h.numel() * 8
        e2e = {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": int(h2d), "d2h_bytes_per_step": int(d2h),
               "steps": k, "path": "gwc_load from pinned host memory, gwc_request_copy_results and gwc_copy_out to pinned host"}

    out = None
    if rank == 0:
        peaks, src = load_peaks()
        chi0_t, fac_t = st["chi0_ms"] * 1e-3, st["factor_ms"] * 1e-3
        chi0_alg = st["chi0_flop"] / chi0_t if chi0_t > 0 else 0.0
        n_ov = mol.n_occ * mol.n_virt
        kname, tile_ratio = chi0_kernel_info(mol.n_aux, n_ov)[0], chi0_executed_ratio(mol.n_aux, n_ov)
        mma_mult = {"bf16x3": 3.0, "bf16x3f64": 3.0, "bf16": 1.0}.get(args.prec, 0.0) * tile_ratio
        peak = peaks.get("bf16_tflops_sustained", peaks.get("bf16_tflops"))
        per_launch = st["chi0_builds"] / max(1, st["chi0_launches"])
        roof = {"kernel": f"{kname} (tcgen05 {args.prec})", "bound": "tensor", "achieved": chi0_alg / 1e12,
                "peak": peak, "unit": "TFLOP/s", "frac": chi0_alg / 1e12 / peak,
                "traffic": load_traffic(kname, "pentacene", per_launch),
                "traffic_unit": f"DRAM bytes per launch ({per_launch:.1f} frequencies) from the committed ncu capture, "
                                "scaled to N_ov = 89 571 and to the frequencies per launch",
                "mma_frac": mma_mult * chi0_alg / 1e12 / peak,
                "peak_source": f"{src} bf16 sustained (kernel timed inside a long step)",
                "share_of_step": chi0_t / (total_ms * 1e-3),
                "work": "algorithmic flop of the builds done: N_aux(N_aux+1) N_ov per real part, 2 parts at complex z"}
        lat = sorted(times)
        out = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": total_ms / args.steps, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": {"bf16x3": "bf16x3+f32+f64", "bf16x3f64": "bf16x3+f64", "bf16": "bf16+f32+f64", "fp32": "f32+f64",
                      "fp64": "f64"}[args.prec],
            "data": "synthetic",
            "config": {"workload": describe_pent(mol), "precision": args.prec,
                       "factorisation": {"bf16x3": "FP32-accurate (tcgen05 3xTF32 trailing updates, FP32 panels)",
                                         "bf16": "FP32-accurate (tcgen05 3xTF32)", "bf16x3f64": "FP64 (SIMT)",
                                         "fp32": "FP32 (SIMT)", "fp64": "FP64 (SIMT)"}[args.prec],
                       "step": pent_step_text(), "points_per_step": npts, "residue_builds_per_step": builds,
                       "parallelism": f"replicas x{ws}", "l2": "256 MB written between timed steps (L2 flushed)",
                       "qp": "G_dH W0, eps_n + dH_n (exact fixed point of the QP equation)"},
            "roofline": roof,
            "chi0_tflops": {"algorithmic": chi0_alg / 1e12, "gemm_equivalent": 2 * chi0_alg / 1e12,
                            "mma_executed": mma_mult * chi0_alg / 1e12 if mma_mult else None},
            "latency_ms": {"p50": lat[len(lat) // 2], "p99": lat[min(len(lat) - 1, int(math.ceil(0.99 * len(lat))) - 1)],
                           "per_step": times},
            "kernel_time_share": {"chi0": st["chi0_ms"] / total_ms, "factor": st["factor_ms"] / total_ms,
                                  "solve": st["solve_ms"] / total_ms},
            "builds_done": st["chi0_builds"] / args.steps,
            "gpu_launches": int(st["kernel_launches"]),
            "clocks": clk,
            "e2e": e2e,
            "spectra_per_s": nc / (total_ms * 1e-3 / args.steps),
            "qp": {"cores": PENT_QP_CORES, "eps_qp_Ha": [float(eqp[c]) for c in PENT_QP_CORES],
                   "dH_Ha": [float(dh[c]) for c in PENT_QP_CORES]},
        }
        out["vs_oracle"] = pent_vs_oracle(dh, sig_last, im_dec.cpu().numpy(), grid_rel)
    # residue contractions at 8 frequencies, compared with the FP64 GPU path below
    z8, rhs8 = pent_fp64_sample_inputs(mol, dev)
    w_mixed = ctx.screen(z8, rhs8).cpu().numpy()
    ctx.sync()
    ctx.close()
    del flush

    if rank == 0 and not args.no_fp64_path and args.prec != "fp64":
        out["fp64_path"], w64 = pent_fp64_path(gwc, mol, eps_d, builds, npts, dev)
        out["fp64_path"]["w_mixed_vs_fp64_max_rel"] = float(np.max(np.abs(w_mixed - w64)) / np.max(np.abs(w64)))
        if out["fp64_path"].get("value"):
            out["mixed_over_fp64_path"] = value / out["fp64_path"]["value"]
    if rank == 0 and ws == 1 and not args.no_cpu_baseline:
        r = pent_oracle_sample(host_copy(mol), builds)
        out["cpu_baseline"] = {"value": r["value"], "unit": UNIT, "cores": cpu_threads(), "kind": "oracle",
                               "sample": r["sample"], "measured_s": r["measured_s"]}
    if rank == 0:
        print(json.dumps(out), flush=True)
    if pg is not None:
        pg.barrier()
        pg.destroy_process_group()
    return 0


def pent_vs_oracle(dh, sig, im_dec, grid_rel):
    """Errors against the FP64 oracle values in tests/golden/pentacene_oracle.json, per core."""
    import numpy as np

    p = os.path.join(ROOT, "tests", "golden", "pentacene_oracle.json")
    if not os.path.exists(p):
        return None
    with open(p) as f:
        gold = json.load(f)
    out = {"dH_err_eV": {}, "sigma_err_Ha": {}, "im_sigma_dec_err_Ha": {}}
    for k, c in enumerate(gold["cores"]):
        if c in PENT_QP_CORES:
            out["dH_err_eV"][str(c)] = float((dh[c] - gold["dH"][k]) * HARTREE_EV)
    for j, gi in enumerate(PENT_SIGMA_IDX):
        if gi in gold.get("omega_idx", []):
            ref = np.array([complex(*v) for v in gold["points"][gold["omega_idx"].index(gi)]["sigma_c"]])
            got = sig[:, j, 0] + 1j * sig[:, j, 1]
            out["sigma_err_Ha"][str(gi)] = {"max_abs": float(np.max(np.abs(got - ref))),
                                            "max_rel": float(np.max(np.abs(got - ref) / np.abs(ref)))}
    d = gold.get("dec_rel")
    if d:
        for k, c in enumerate(d["cores"][: len(d["values"])]):
            got = im_dec[c, d["nu_idx"]]
            out["im_sigma_dec_err_Ha"][str(c)] = float(np.max(np.abs(got - np.array(d["values"][k]))))
    return out


def pent_fp64_path(gwc, mol, eps_d, builds, npts, dev):
    """The plain FP64 GPU path (FP64 chi0, FP64 LDL^T) on a measured sample: its imaginary-axis W table and
    one factorisation wave of 8 residue builds (22 right-hand sides each); the step's time extrapolated as
    T_table + residue builds x T_chi0 + factorisation waves x T_wave (waves of `batch` matrices per phase)."""
    import numpy as np
    import torch

    batch = 73  # FP64 complex 4500 x 4500 matrices fitting the 24 GB workspace
    z, rhs = pent_fp64_sample_inputs(mol, dev)
    c64 = gwc.Context(eps_d, mol.n_occ, mol.core_idx, mol.o_ov, mol.o_core, prec="fp64", eta=mol.eta, n_im=mol.n_im,
                      xi0=mol.xi0, n_t=mol.n_t, t_max=mol.t_max, batch=batch, profile=True)
    ef = 0.5 * (mol.eps[mol.n_occ - 1] + mol.eps[mol.n_occ])
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    c64.sigma_core(np.array([ef]), want_dec=False)  # between HOMO and LUMO: no residues, the table alone
    c64.sync()
    t_table = time.perf_counter() - t0
    c64.reset_stats()
    w64 = c64.screen(z, rhs)
    c64.sync()
    st = c64.stats()
    c64.close()
    t_chi0 = st["chi0_ms"] * 1e-3 / 8
    t_wave = st["factor_ms"] * 1e-3
    waves = sum(-(-builds[k] // batch) for k in ("decoupled", "qp", "sigma"))
    n_res = builds["decoupled"] + builds["qp"] + builds["sigma"]
    t_step = t_table + n_res * t_chi0 + waves * t_wave
    return {"value": npts["total"] / t_step, "unit": UNIT, "extrapolated": True, "t_step_s": t_step,
            "t_table_s": t_table, "t_chi0_per_build_s": t_chi0, "t_factor_wave_s": t_wave, "waves": waves,
            "sample": ("FP64 GPU path measured: its imaginary-axis W table, and 8 residue builds (FP64 chi0, one "
                       "FP64 LDL^T wave, 22 right-hand sides); the same step extrapolated from these")}, w64.cpu().numpy()


def pent_fp64_sample_inputs(mol, dev):
    """8 residue frequencies near the valence residue of grid point 100 and the 22 core right-hand sides."""
    import torch

    z = torch.tensor([[abs(mol.eps[30] - mol.omega[PENT_SIGMA_IDX[0]]) + 0.01 * k, mol.eta] for k in range(8)],
                     dtype=torch.float64, device=dev)
    return z, mol.o_core[30].unsqueeze(0).expand(8, -1, -1).contiguous()


# ------------------------------------------------------------------------------------------
# Precision form at the pentacene size, batched form, serving form
# ------------------------------------------------------------------------------------------
def _events():
    import torch

    return torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)


def run_pentacene(args):
    """Pentacene-sized molecule (1300 states, 73 occupied, 22 cores, 4500 aux): Hedin shifts of all
    cores and Sigma^c of all cores at a subset of grid points, mixed path vs the plain FP64 GPU path,
    errors per core against the FP64 oracle values of tests/golden/pentacene_oracle.json."""
    import numpy as np
    import torch

    from paper_2412_17132_gb300 import gwc, synth

    mol = synth.pentacene_device()
    pts_idx = [100, 700][: max(1, min(2, args.omega_points))]
    out = {"metric": "pentacene-sized: Sigma_c points/s, mixed vs FP64 GPU path", "unit": UNIT, "n_gpus": 1,
           "data": "synthetic", "config": {"workload": describe(mol), "grid_points": pts_idx}}
    res = {}
    for prec in (args.prec, "fp64") if args.fp64_points > 0 else (args.prec,):
        ctx = gwc.Context(torch.as_tensor(mol.eps, device="cuda"), mol.n_occ, mol.core_idx, mol.o_ov, mol.o_core,
                          prec=prec, qp_mode="hedin", batch=args.batch or 64, eta=mol.eta, n_im=mol.n_im, profile=True)
        torch.cuda.synchronize()
        t_qp, dh = None, None
        if prec != "fp64":  # FP64 Hedin shifts of all 22 cores would take ~1.5 h at 1.2 TFLOP/s FP64
            e0, e1 = _events()
            e0.record()
            e, dh, it = ctx.qp_solve()
            e1.record()
            e1.synchronize()
            t_qp = e0.elapsed_time(e1) / 1e3
            dh = dh.cpu().numpy()
        pts = mol.omega[pts_idx[: (args.fp64_points if prec == "fp64" else len(pts_idx))]]
        e0, e1 = _events()
        e0.record()
        sig, dec, sx = ctx.sigma_core(pts)
        e1.record()
        e1.synchronize()
        t_sig = e0.elapsed_time(e1) / 1e3
        ctx.sync()
        res[prec] = {"dh": dh, "sig": sig.cpu().numpy(), "t_qp": t_qp, "t_sig": t_sig,
                     "points": mol.n_core * len(pts), "stats": ctx.stats()}
        ctx.close()
    m, f = res[args.prec], res.get("fp64")
    out["value"] = m["points"] / m["t_sig"]
    out["hedin_shift_seconds_all_cores"] = m["t_qp"]
    if f is not None:
        out["fp64_path"] = {"value": f["points"] / f["t_sig"], "points": f["points"], "seconds": f["t_sig"]}
        out["mixed_over_fp64"] = out["value"] / out["fp64_path"]["value"]
        out["sigma_mixed_minus_fp64_Ha_max"] = float(np.max(np.abs(m["sig"][:, : f["sig"].shape[1]] - f["sig"])))
    gold_p = os.path.join(ROOT, "tests", "golden", "pentacene_oracle.json")
    if os.path.exists(gold_p):
        with open(gold_p) as fh:
            gold = json.load(fh)
        out["vs_oracle"] = {
            "cores": gold["cores"],
            "dH_err_eV": {p: [float((res[p]["dh"][c] - gold["dH"][k]) * HARTREE_EV) for k, c in enumerate(gold["cores"])]
                          for p in res if res[p]["dh"] is not None},
        }
        # Sigma at the grid points both the run and the oracle file have (matched by grid index)
        errs = {}
        for p in res:
            e = []
            for j, gi in enumerate(pts_idx[: res[p]["sig"].shape[1]]):
                if gi in gold.get("omega_idx", []):
                    ref = np.array([complex(*v) for v in gold["points"][gold["omega_idx"].index(gi)]["sigma_c"]])
                    e.append(float(np.max(np.abs(res[p]["sig"][:, j, 0] + 1j * res[p]["sig"][:, j, 1] - ref))))
            if e:
                errs[p] = max(e)
        out["vs_oracle"]["sigma_err_Ha_max"] = errs
    print(json.dumps(out), flush=True)
    return 0


def run_batch(args):
    """Batched form: molecules j = 0..M-1 (N_states ~ U{100..1300}, seed 1000 + j) generated on the GPU,
    each a request (decoupled spectra of all cores on the relative grid + Hedin QP), all captured into
    one CUDA graph after autotuning the frequency batch and the chi0 tile and launch shapes per shape bucket."""
    import numpy as np
    import torch

    from paper_2412_17132_gb300 import gwc, synth

    grid = np.linspace(-25.0 / HARTREE_EV, 5.0 / HARTREE_EV, args.omega_points)
    ctxs, sizes, tuned, ctas_chosen, tiles_chosen = [], [], [], [], []
    t_setup = time.perf_counter()
    for j in range(args.molecules):
        mol = synth.batch_member_device(j)
        c = gwc.Context(torch.as_tensor(mol.eps, device="cuda"), mol.n_occ, mol.core_idx, mol.o_ov, mol.o_core,
                        prec=args.prec, qp_mode="hedin", batch=args.batch or 32, eta=mol.eta, n_im=mol.n_im)
        del mol
        c.request_plan(grid)
        tuned.append(c.autotune())
        ctas_chosen.append(c.chi0_ctas())
        tiles_chosen.append(c.chi0_tile())
        ctxs.append(c)
        sizes.append((c.n_states, c.n_aux, c.n_core))
        torch.cuda.empty_cache()
    t_setup = time.perf_counter() - t_setup
    t_cap = time.perf_counter()
    batch = gwc.Batch(ctxs)
    t_cap = time.perf_counter() - t_cap
    times = []
    clocks = ClockSampler(0)
    torch.cuda.synchronize()
    clocks.start()
    for _ in range(args.steps):
        e0, e1 = _events()
        e0.record()
        batch.launch()
        e1.record()
        e1.synchronize()
        times.append(e0.elapsed_time(e1) / 1e3)
    clk = clocks.stop()
    points = sum(nc for _, _, nc in sizes) * args.omega_points
    out = {"metric": "batched form: decoupled Sigma points/s (+ Hedin QP + spectra) in one graph launch", "unit": UNIT,
           "value": points / statistics.mean(times), "n_gpus": 1, "steps": args.steps, "data": "synthetic",
           "ms_per_step": 1e3 * statistics.mean(times), "dtype": args.prec,
           "config": {"workload": f"{args.molecules} molecules, N_states ~ U{{100..1300}} (seed 1000+j), N_aux = 3.5 N, "
                                  f"{args.omega_points}-point relative grid, cores = round(0.3 N_occ), QP = eps_n + dH_n",
                      "sizes_states_aux_cores": sizes, "autotuned_batch": tuned,
                      "autotuned_chi0_ctas": ctas_chosen,
                      "autotuned_chi0_tile": tiles_chosen,
                      "form": ("grouped: per residue chunk one grouped chi0 launch and one grouped LDL^T launch over "
                               "all molecules (" + batch.chi0_shape + "), in one CUDA graph")
                      if batch.grouped else "graph of per-molecule steps on forked streams",
                      "plans_timed_ms": dict(zip(["per_molecule", "grouped_sequential_persistent", "grouped_pipelined_per_item"],
                                                 batch.timings()))},
           "spectra_per_s": sum(nc for _, _, nc in sizes) / statistics.mean(times),
           "setup_s": t_setup, "capture_s": t_cap, "clocks": clk,
           "latency_ms": {"per_launch": [1e3 * t for t in times]}}
    batch.close()
    for c in ctxs:
        c.close()
    print(json.dumps(out), flush=True)
    return 0


def run_serve(args):
    """Serving form: Poisson arrivals of spectrum requests (N_states log-uniform on [100, 1500], inputs
    generated on the GPU from seed = request id), admitted by HBM footprint, continuous batching."""
    import numpy as np
    import torch

    from paper_2412_17132_gb300 import serve, synth

    grid = np.linspace(-25.0 / HARTREE_EV, 5.0 / HARTREE_EV, args.omega_points)
    arr = serve.poisson_arrivals(args.requests, args.rate, seed=0)
    reqs = [serve.Request(rid=i, arrival=float(arr[i]), make=(lambda i=i: synth.serving_request_device(i)),
                          n_states=serve.serving_size(i)) for i in range(args.requests)]
    free, _ = torch.cuda.mem_get_info()
    srv = serve.SpectrumServer(grid, budget_bytes=int(0.5 * free), slots=args.slots, prec=args.prec, qp_mode="hedin",
                               batch=args.batch or 64)
    clocks = ClockSampler(0)
    clocks.start()
    t0 = time.perf_counter()
    done = srv.run(reqs, time_limit=args.time_limit)
    makespan = time.perf_counter() - t0
    clk = clocks.stop()
    summ = serve.summarize(done, makespan)
    out = {"metric": "serving form: spectra/s and p50/p99 latency (arrival to results in host memory)", "unit": "requests/s",
           "value": summ["requests_per_s"], "n_gpus": 1, "data": "synthetic", "dtype": args.prec,
           "config": {"workload": f"{args.requests} requests offered at {args.rate}/s (Poisson, seed 0), N_states log-uniform "
                                  f"[100, 1500] from seed = request id, {args.omega_points}-point grid, QP = eps_n + dH_n",
                      "slots": args.slots, "budget_GB": 0.5 * free / 1e9, "time_limit_s": args.time_limit},
           "serving": summ, "makespan_s": makespan,
           "offered_requests": args.requests, "arrived_by_end": int(sum(1 for a in arr if a <= makespan)),
           "max_sustainable_requests_per_s": summ["requests_per_s"],
           "contexts": {"created": srv.created, "reused": srv.reused, "classes": list(serve.SIZE_CLASSES)},
           "sizes_served": [int(r.n_states) for r in done], "clocks": clk,
           "note": "completed/makespan under saturation is the sustainable rate; p50/p99 include queueing"}
    srv.close()
    print(json.dumps(out), flush=True)
    return 0


def main():
    args = parse()
    if args.impl == "reference":
        return run_reference(args)
    if args.workload == "pentacene":
        return run_pentacene_headline(args)
    if args.workload == "pentacene-forms":
        return run_pentacene(args)
    if args.workload == "batch":
        return run_batch(args)
    if args.workload == "serve":
        return run_serve(args)
    return run_gpu(args)


if __name__ == "__main__":
    sys.exit(main())
