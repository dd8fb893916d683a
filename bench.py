#!/usr/bin/env python3
"""Throughput of the batched recursive Green's function (RGF) hot path on GB300.

Workload: a block-tridiagonal device of N = 70 slabs x 400 x 400 complex blocks (40 atoms x
10 orbitals per slab, Si with 10% Ge as +0.2 eV on-site shifts), 512 energies in [-3, 3] eV x
8 transverse k-points = 4096 (E, k) points, eta = 1e-6, synthetic seeded Hamiltonians.
One step = one batch of points through the whole path: Sancho-Rubio lead self-energies,
forward and backward sweeps, density / bond current / transmission, and the FP64 energy
quadrature of the batch.  Inputs (8 k-point Hamiltonians, 2.9 GB) are resident in HBM; every
step streams 358 MB of Hamiltonian blocks, more than the 129 MB L2.

Prints one JSON line (metric energy-points/s).  --impl reference times the CPU oracle instead.
"""
from __future__ import annotations

import argparse
import json
import os
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

WORK = dict(N=70, b=400, n_E=512, n_k=8, ge_frac=0.1, eta=1e-6, seed=1001,
            name="ballistic RGF, N=70 slabs x 400x400 blocks, alloy p(Ge)=0.1, 512 E x 8 k")
METRIC = "RGF energy-points/s (leads + forward/backward sweeps + observables + FP64 quadrature)"
PEAKS_FALLBACK = dict(hbm_gbs=6800.0, bf16_tflops=1900.0, bf16_tflops_sustained=1700.0)
# DRAM bytes (read + write) of k_crt_gemm per 400 x 400 x 400 complex item from an ncu capture of
# a 64-item 48-bit launch (1015.4 MB read + 159.8 MB written), scaled by the items of a launch; None
# once the kernel has changed since the capture (the line then reports null).
TC_DRAM_BYTES_PER_ITEM_B400 = (1015.397e6 + 159.823e6) / 64
GOLDEN = os.path.join(ROOT, "tests", "golden", "c1_oracle.json")


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--precision", default="mixed", choices=["mixed", "mixed40", "mixed56", "fp64"],
                    help="tier of the sweeps: tensor cores with 48- (mixed), 40- or 56-bit "
                         "operand values, or FP64 on the CUDA cores; the lead decimation of the "
                         "mixed tiers runs at 56 bits")
    ap.add_argument("--points-per-step", type=int, default=256)
    ap.add_argument("--cpu-points", type=int, default=4)
    ap.add_argument("--fp64-points", type=int, default=64,
                    help="points of the FP64 GPU comparison batch (one batch; the FP64 form's "
                         "rate saturates near 64 points on this device)")
    ap.add_argument("--no-golden", action="store_true",
                    help="skip the accuracy check of a full k-slice against the stored oracle "
                         "values (tests/golden/c1_oracle.json)")
    ap.add_argument("--no-extras", action="store_true",
                    help="skip the CPU-oracle, FP64-GPU and end-to-end side measurements")
    ap.add_argument("--workload", default="rgf",
                    choices=["rgf", "scba", "adjoint", "ragged", "gemm", "iface", "zinv"],
                    help="rgf: the throughput line above; scba / adjoint / ragged / gemm: side "
                         "measurements of the Born loop (N=70, b=600), the adjoint sweep "
                         "(b=3430), ragged block sizes (b=200..800) and the batched tensor-core "
                         "complex GEMM alone (b x b x b, --gemm-batch items)")
    ap.add_argument("--scba-energies", type=int, default=128)
    ap.add_argument("--adj-slabs", type=int, default=20)
    ap.add_argument("--adj-segment", type=int, default=0,
                    help="--workload adjoint: slabs per checkpointed segment (0 = keep all)")
    ap.add_argument("--adj-ckpt", action="store_true",
                    help="--workload adjoint: time solve + adjoint with the solve's checkpoints "
                         "handed to the adjoint, beside solve + a recomputing adjoint")
    ap.add_argument("--adj-iface", type=int, default=0,
                    help="--workload adjoint: hoppings supported on the last r rows / first r "
                         "columns (the facing atoms), r orbitals; 0 = dense")
    ap.add_argument("--ragged-points", type=int, default=4,
                    help="energies per (sample, k) system of the ragged workload")
    ap.add_argument("--ragged-samples", type=int, default=16)
    ap.add_argument("--ragged-chunk", type=int, default=16,
                    help="points per launch chain in the ragged workload (bounds each group's "
                         "workspace)")
    ap.add_argument("--tc-config", type=int, default=None,
                    help="tensor-core GEMM configuration of calls of fewer than 12 points (default: "
                         "autotuned per block size and batch for the rgf workload, the library "
                         "default otherwise)")
    ap.add_argument("--scba-sigma", choices=["diag", "atom"], default="diag",
                    help="--workload scba: orbital-diagonal or atom-block (10 x 10) self-energies")
    ap.add_argument("--iface-orbitals", type=int, default=100,
                    help="rows and columns of the hopping support in --workload iface")
    ap.add_argument("--gemm-b", type=int, default=400)
    ap.add_argument("--gemm-batch", type=int, default=64)
    return ap.parse_args()


def peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as fh:
            d = json.load(fh)
        return d, "measured"
    return dict(PEAKS_FALLBACK), "fallback"


def build_hamiltonians():
    from workloads import make_device, hamiltonian_k, k_grid, energy_grid_linspace
    dev = make_device(WORK["N"], WORK["b"], WORK["seed"], ge_frac=WORK["ge_frac"], with_k=True)
    ks, wk = k_grid(WORK["n_k"])
    Hd = np.empty((WORK["n_k"], WORK["N"], WORK["b"], WORK["b"]), dtype=np.complex128)
    for i, k in enumerate(ks):
        Hd[i] = hamiltonian_k(dev, float(k))[0]
    Hu = np.broadcast_to(dev.T, (WORK["n_k"],) + dev.T.shape)
    E, wE = energy_grid_linspace(-3.0, 3.0, WORK["n_E"])
    return dev, Hd, Hu, ks, wk, E, wE


def point_index(n_pts_total, start, count):
    idx = (np.arange(count) + start) % n_pts_total
    return idx // WORK["n_E"], idx % WORK["n_E"]   # (k index, energy index)


def rank_points(step, rank, world, P):
    """(k index, energy index) of the P points that rank `rank` of `world` solves in `step`:
    consecutive blocks of P points of the (k, E) grid dealt out to the ranks in turn, so ranks
    solve disjoint points and `world` ranks solve `world` times the points of one (weak scaling,
    no data-path collective)."""
    n_tot = WORK["n_E"] * WORK["n_k"]
    return point_index(n_tot, (step * world + rank) * P, P)


def max_over_ranks(ms, dist, device):
    """Length of the timed region as the slowest rank measured it (every rank gets it)."""
    if dist is None:
        return ms
    import torch
    t = torch.tensor([ms], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    dist.barrier()
    return float(t.item())


def aggregate_rate(steps, P, world, ms):
    """Whole-job points per second: the points all ranks solved over the slowest rank's time."""
    return steps * P * world / (ms / 1e3)


class Clocks:
    """nvidia-smi sampling (read-only) while the timed region runs."""

    def __init__(self, gpu_index):
        self.samples = []
        self.proc = None
        self.gpu = gpu_index

    def __enter__(self):
        q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={q}", "--format=csv,noheader,nounits",
                                          "-i", str(self.gpu), "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except Exception:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.samples.append([x.strip() for x in line.split(",")])

    def __exit__(self, *a):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()

    def summary(self):
        if not self.samples:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        sm = [float(s[1]) for s in self.samples if len(s) > 2 and s[1].replace('.', '').isdigit()]
        mx = [float(s[2]) for s in self.samples if len(s) > 2 and s[2].replace('.', '').isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = set()
        for s in self.samples:
            for n, v in zip(names, s[5:9]):
                if v.strip().lower() == "active":
                    reasons.add(n)
        return {"sm_mhz": float(np.median(sm)) if sm else None,
                "sm_max_mhz": max(mx) if mx else None, "samples": len(self.samples),
                "reasons": sorted(reasons)}


def run_reference(args):
    """CPU oracle on the host cores: each step solves one point of the same workload."""
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    import oracle as O
    dev, Hd, Hu, ks, wk, E, wE = build_hamiltonians()
    n_tot = WORK["n_E"] * WORK["n_k"]
    for s in range(args.warmup):
        kk, ee = point_index(n_tot, 1000 + s * 97, 1)
        O.solve_point(Hd[kk[0]], dev.T, E[ee[0]], WORK["eta"], None)
    t0 = time.perf_counter()
    for s in range(args.steps):
        kk, ee = point_index(n_tot, s * 211, 1)
        O.solve_point(Hd[kk[0]], dev.T, E[ee[0]], WORK["eta"], None)
    dt = time.perf_counter() - t0
    v = args.steps / dt
    cores = _blas_threads()
    print(json.dumps({
        "impl": "reference", "metric": METRIC, "value": v, "unit": "points/s",
        "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": 1e3 * dt / args.steps, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "c128", "data": "synthetic",
        "config": {"workload": WORK["name"], "points_per_step": 1},
        "cpu_baseline": {"value": v, "unit": "points/s", "cores": cores, "kind": "oracle",
                         "blas": _blas_info(), "host_cores": os.cpu_count(),
                         "sample": f"{args.steps} points of the workload, one per step"},
        "e2e": {"value": v, "unit": "points/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }), flush=True)


_ONE_CORE = r"""
import sys, time
sys.path.insert(0, {root!r})
import oracle as O
from workloads import make_device, hamiltonian_k, k_grid, energy_grid_linspace
dev = make_device({N}, {b}, {seed}, ge_frac={ge}, with_k=True)
ks, _ = k_grid({n_k})
Hd = hamiltonian_k(dev, float(ks[{k}]))[0]
E, _ = energy_grid_linspace(-3.0, 3.0, {n_E})
t0 = time.perf_counter()
O.solve_point(Hd, dev.T, E[{e}], {eta}, None)
print(time.perf_counter() - t0)
"""


def _oracle_one_core(k, e):
    """Seconds of one oracle point of the workload with BLAS on one thread (a child process,
    so that the thread count is fixed before numpy loads); None if it could not run."""
    code = _ONE_CORE.format(root=ROOT, N=WORK["N"], b=WORK["b"], seed=WORK["seed"],
                            ge=WORK["ge_frac"], n_k=WORK["n_k"], k=int(k), n_E=WORK["n_E"],
                            e=int(e), eta=WORK["eta"])
    env = dict(os.environ, OPENBLAS_NUM_THREADS="1", OMP_NUM_THREADS="1", MKL_NUM_THREADS="1",
               CUDA_VISIBLE_DEVICES="")
    try:
        r = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True,
                           timeout=600)
        return float(r.stdout.strip().splitlines()[-1]) if r.returncode == 0 else None
    except Exception:
        return None


def _blas_info():
    """numpy's BLAS (name and version) for the CPU-baseline record."""
    try:
        d = np.show_config(mode="dicts")["Build Dependencies"]["blas"]
        return f"{d.get('name', '?')} {d.get('version', '')}".strip()
    except Exception:
        return "unknown"


def _blas_threads():
    try:
        from threadpoolctl import threadpool_info
        n = [i.get("num_threads", 0) for i in threadpool_info() if i.get("user_api") == "blas"]
        if n:
            return int(max(n))
    except Exception:
        pass
    return os.cpu_count()


def _timed(torch, fn, warmup, steps):
    for _ in range(warmup):
        fn()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(steps):
        out = fn()
    e1.record()
    torch.cuda.synchronize()
    return e0.elapsed_time(e1), out


def run_side(args):
    """Side measurements for the Born loop, the adjoint sweep and ragged block sizes."""
    import torch
    import paper_1510_04686_gb300 as negf
    from workloads import make_device, config_workload
    torch.cuda.set_device(0)
    negf._build.build()
    dvc = torch.device("cuda", 0)
    line = {"impl": "ours", "n_gpus": 1, "steps": args.steps, "warmup": args.warmup,
            "data": "synthetic", "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None}
    if args.workload == "scba":
        w = config_workload(3, n_E=args.scba_energies)
        dev, E, prm = w["device"], w["E"], w["params"]
        N, b, nE = dev.N, dev.b, E.size
        D = negf.Device(torch.as_tensor(dev.D[None], device=dvc), torch.as_tensor(dev.T[None], device=dvc))
        Et = torch.as_tensor(E, device=dvc)
        st = torch.zeros(nE, dtype=torch.int32, device=dvc)
        atom = args.scba_sigma == "atom"
        opt = negf.options(precision=negf.PREC_MIXED, chunk=min(nE, 128),
                           sigma_structure=negf.SIGMA_ATOM_BLOCK if atom else
                           negf.SIGMA_ORBITAL_DIAG, atom_orbitals=10)
        nS = N * b * negf.sigma_width(opt)  # entries of a self-energy row
        lead = negf.lead_selfenergy(D, Et, st, opt)
        sR = torch.zeros((nE, nS), dtype=torch.complex128, device=dvc)
        sL = torch.zeros_like(sR)
        wk = torch.ones(1, dtype=torch.float64, device=dvc)
        n0 = 1.0 / (np.exp(prm["hw"] / prm["kT"]) - 1.0)
        deltas = []

        def born():
            out = negf.rgf_solve(D, Et, st, lead["sigma_R"], lead["sigma_L"], opt, scat_R=sR,
                                 scat_L=sL, diag=True, outputs=("density", "current"))
            d = negf.scba_step(out["diagGR"].reshape(1, nE, nS), out["diagGL"].reshape(1, nE, nS),
                               wk, sR, sL, prm["D_ac"], prm["D_op"],
                               int(round(prm["hw"] / prm["dE"])), n0)
            deltas.append(d)
            return out
        ms, _ = _timed(torch, born, args.warmup, args.steps)
        line.update(metric="SCBA point-iterations/s (RGF with phonon self-energies + Born update)",
                    value=nE * args.steps / (ms / 1e3), unit="point-iterations/s",
                    ms_per_step=ms / args.steps, dtype="bf16-integers->fp32 (fp64 storage)",
                    config={"workload": f"SCBA N=70 b=600, energies 0..{nE - 1} of the 5 meV grid, "
                                        + ("atom-block (10 x 10) self-energies" if atom else
                                           "orbital-diagonal self-energies"),
                            "D_ac": 0.01, "D_op": 0.01, "hw_steps": 12,
                            "last_delta": float(deltas[-1].item())})
    elif args.workload == "adjoint":
        w = config_workload(4, N=args.adj_slabs, n_E=1)
        dev, V = w["device"], w["V"]
        N, b = dev.N, dev.b
        rng = np.random.default_rng(4)
        T = dev.T
        iface = None
        if args.adj_iface > 0:
            # hoppings only between the facing atoms: the last r rows and first r columns
            r = args.adj_iface
            T = T.copy()
            T[:, :b - r, :] = 0.0
            T[:, :, r:] = 0.0
            iface = (r, r)
        D = negf.Device(torch.as_tensor(dev.D[None], device=dvc), torch.as_tensor(T[None], device=dvc),
                        iface=iface)
        Et = torch.as_tensor(np.array([0.1]), device=dvc)
        st = torch.zeros(1, dtype=torch.int32, device=dvc)
        opt = negf.options(precision=negf.PREC_MIXED, chunk=1, adjoint_segment=args.adj_segment)
        lead = negf.lead_selfenergy(D, Et, st, opt)
        Vt = torch.as_tensor(V, device=dvc)
        c = torch.as_tensor(rng.normal(size=(1, N * b)), device=dvc)
        d = torch.as_tensor(rng.normal(size=(1, N - 1)), device=dvc)

        def adj():
            return negf.rgf_adjoint(D, Et, st, lead["sigma_R"], lead["sigma_L"], opt,
                                    density_bar=c, current_bar=d, V=Vt)
        extra = {}
        if args.adj_ckpt:
            # the autograd step: solve + adjoint, with the solve's sweep blocks handed to the
            # adjoint, against solve + an adjoint that recomputes them
            ck = negf.checkpoint_buffer(D, 1)

            def step_ck():
                negf.rgf_solve(D, Et, st, lead["sigma_R"], lead["sigma_L"], opt, V=Vt,
                               checkpoints=ck)
                return negf.rgf_adjoint(D, Et, st, lead["sigma_R"], lead["sigma_L"], opt,
                                        density_bar=c, current_bar=d, V=Vt, checkpoints=ck)

            def step_re():
                negf.rgf_solve(D, Et, st, lead["sigma_R"], lead["sigma_L"], opt, V=Vt)
                return adj()
            ms_re, _ = _timed(torch, step_re, args.warmup, args.steps)
            ms, _ = _timed(torch, step_ck, args.warmup, args.steps)
            extra = {"solve_plus_recomputing_adjoint_ms": ms_re / args.steps,
                     "speedup_of_checkpoint_handoff": ms_re / ms}
        else:
            ms, _ = _timed(torch, adj, args.warmup, args.steps)
        line.update(metric=("solve + adjoint points/s with the checkpoint hand-off (dL/dV)"
                            if args.adj_ckpt else
                            "adjoint points/s (forward sweep kept + reverse sweep, dL/dV)"),
                    value=args.steps / (ms / 1e3), unit="points/s", ms_per_step=ms / args.steps,
                    dtype="bf16-integers->fp32 (fp64 storage)",
                    config={"workload": f"adjoint, N={N} slabs x 3430 orbitals (343 atoms x 10),"
                                        " V ~ U(-0.3, 0.3) eV per atom, 1 point"
                                        + (f", hoppings on the {args.adj_iface} x "
                                           f"{args.adj_iface} facing-atom block"
                                           if args.adj_iface > 0 else ""),
                            "adjoint_segment": args.adj_segment, **extra})
    elif args.workload == "iface":
        # the benchmark device with interface couplings: every hopping block keeps only the
        # orbitals of the 10 facing atoms of each slab (its last 100 rows, first 100 columns)
        from workloads import hamiltonian_k, k_grid, energy_grid_linspace
        r = c = args.iface_orbitals
        dv = make_device(WORK["N"], WORK["b"], WORK["seed"], ge_frac=WORK["ge_frac"],
                         with_k=True, iface=(r, c))
        ks, _ = k_grid(WORK["n_k"])
        Hd = torch.as_tensor(np.stack([hamiltonian_k(dv, float(k))[0] for k in ks]), device=dvc)
        Hu = torch.as_tensor(np.ascontiguousarray(np.broadcast_to(dv.T, (WORK["n_k"],) + dv.T.shape)),
                             device=dvc)
        E_all, _ = energy_grid_linspace(-3.0, 3.0, WORK["n_E"])
        P = args.points_per_step
        Et = torch.as_tensor(E_all[(np.arange(P) * 7) % WORK["n_E"]], device=dvc)
        st = torch.as_tensor((np.arange(P) % WORK["n_k"]).astype(np.int32), device=dvc)
        opt = negf.options(precision=negf.PREC_MIXED, chunk=P)
        rates = {}
        for name, iface in (("interface", (r, c)), ("dense", None)):
            d = negf.Device(Hd, Hu, iface=iface)
            ms_l, lead = _timed(torch, lambda: negf.lead_selfenergy(d, Et, st, opt),
                                args.warmup, args.steps)

            def solve():
                return negf.rgf_solve(d, Et, st, lead["sigma_R"], lead["sigma_L"], opt)
            ms_s, out = _timed(torch, solve, args.warmup, args.steps)
            rates[name] = dict(step=P * args.steps / ((ms_l + ms_s) / 1e3),
                               leads=P * args.steps / (ms_l / 1e3),
                               sweeps=P * args.steps / (ms_s / 1e3),
                               ms=(ms_l + ms_s) / args.steps, out=out, lead=lead)
        it, dn_ = rates["interface"], rates["dense"]
        dn = (it["out"]["density"] - dn_["out"]["density"]).abs().max().item()
        ds = (it["lead"]["sigma_R"] - dn_["lead"]["sigma_R"]).abs().max().item()
        line.update(metric="energy-points/s with interface couplings (lead decimation + RGF "
                           "sweeps)",
                    unit="points/s", value=it["step"], ms_per_step=it["ms"],
                    dtype="bf16-integers->fp32 (fp64 storage)",
                    config={"workload": f"N=70 slabs x 400x400 blocks, hoppings between the "
                                        f"{r // 10} facing atoms of each slab ({r} x {c} support),"
                                        f" {P} points",
                            "leads_points_per_s": it["leads"],
                            "sweeps_points_per_s": it["sweeps"],
                            "dense_points_per_s": dn_["step"],
                            "dense_leads_points_per_s": dn_["leads"],
                            "dense_sweeps_points_per_s": dn_["sweeps"],
                            "speedup_vs_dense": it["step"] / dn_["step"],
                            "max_density_difference_vs_dense": dn,
                            "max_sigma_difference_vs_dense": ds})
    elif args.workload == "zinv":
        # the mixed block inverse alone (FP32 Gauss-Jordan start + Newton-Schulz refinement)
        b, nb = args.gemm_b, args.gemm_batch
        g = torch.Generator(device=dvc).manual_seed(2)
        M0 = torch.randn((nb, b, b), dtype=torch.complex128, device=dvc, generator=g) / b ** 0.5
        M0 += 4.0 * torch.eye(b, dtype=torch.complex128, device=dvc)
        M = torch.empty_like(M0)

        def inv():
            M.copy_(M0)  # the inverse consumes its input
            return negf.zinv(M, precision=negf.PREC_MIXED)
        ms, (X, st) = _timed(torch, inv, args.warmup, args.steps)
        res = (torch.eye(b, dtype=torch.complex128, device=dvc) - M0 @ X).abs().max().item()
        line.update(metric="batched block inverses/s (mixed: FP32 Gauss-Jordan + Newton-Schulz)",
                    value=nb * args.steps / (ms / 1e3), unit="inverses/s",
                    ms_per_step=ms / args.steps, dtype="fp32 elimination, bf16-integers->fp32 "
                    "refinement (fp64 in/out)",
                    config={"workload": f"{nb} items of {b} x {b} complex128",
                            "max_residual": res,
                            "status_ok": bool((st == 0).all().item())})
    elif args.workload == "gemm":
        b, nb = args.gemm_b, args.gemm_batch
        if args.tc_config is not None:
            negf.tc_config(args.tc_config)
        g = torch.Generator(device=dvc).manual_seed(1)
        A = torch.randn((nb, b, b), dtype=torch.complex128, device=dvc, generator=g)
        B = torch.randn((nb, b, b), dtype=torch.complex128, device=dvc, generator=g)
        C = torch.empty_like(A)
        negf.profile_reset()
        negf.profile(True)
        ms, _ = _timed(torch, lambda: negf.zgemm(A, B, C, precision=negf.PREC_MIXED),
                       args.warmup, args.steps)
        negf.profile(False)
        n_tc, tc_ms, alg, hw = negf.profile_read(negf.PROF_TC_GEMM)
        n_sl, sl_ms, _, _ = negf.profile_read(negf.PROF_SLICE)
        line.update(metric="batched complex GEMM, algorithmic TFLOP/s (8 b^3 per item)",
                    value=8.0 * b ** 3 * nb * args.steps / (ms / 1e3) / 1e12, unit="TFLOP/s",
                    ms_per_step=ms / args.steps, dtype="bf16-integers->fp32 (fp64 in/out)",
                    config={"workload": f"{nb} items of {b} x {b} x {b} complex128",
                            "tc_config": negf.tc_config(),
                            "tc_kernel_ms": tc_ms / max(n_tc, 1),
                            "slicing_ms": sl_ms / max(n_sl, 1),
                            "issued_bf16_tflops": hw / (tc_ms / 1e3) / 1e12 if tc_ms else None})
    else:
        # the batched uneven workload scaled down: samples of the 128-sample set (block sizes
        # drawn from {200, ..., 800} per sample as in the full set), 4 k-points each, a few
        # energies per (sample, k); every (sample, k) is one system of the ragged batch
        from workloads import hamiltonian_k, k_grid, energy_grid_linspace
        n_s, n_e = args.ragged_samples, args.ragged_points
        ks, _ = k_grid(4)
        E_all, _ = energy_grid_linspace(-3.0, 3.0, 256)
        systems, bs = [], []
        for s in range(n_s):
            w = config_workload(2, sample=s, n_E=256, n_k=4)
            dv = w["device"]
            for m, kval in enumerate(ks):
                Hd = hamiltonian_k(dv, float(kval))[0]
                e_idx = (np.arange(n_e) * 256 // n_e + 17 * s + 5 * m) % 256
                systems.append((torch.as_tensor(Hd, device=dvc), torch.as_tensor(dv.T, device=dvc),
                                torch.as_tensor(E_all[e_idx], device=dvc)))
                bs.append(dv.b)
        n_pts = sum(int(x[2].numel()) for x in systems)
        opt = negf.options(precision=negf.PREC_MIXED, chunk=args.ragged_chunk)
        rg = negf.RaggedGraph(systems, opt, sr_steps=48)
        ms, _ = _timed(torch, rg.replay, args.warmup, args.steps)
        # the same batch with the block-size groups one after another, eagerly (no graph, no
        # concurrent streams): what one launch chain per group gives without the overlap
        seq_opt = negf.options(precision=negf.PREC_MIXED, chunk=args.ragged_chunk,
                               sr_host_check=0, sr_max_iter=48)
        ms_seq, _ = _timed(torch, lambda: negf.solve_ragged(systems, seq_opt, concurrent=False),
                           0, 1)
        counts = {int(b): bs.count(b) for b in sorted(set(bs))}
        flops = sum(8.0 * b ** 3 * (18 * 70 + 2 * (7 * 28 + 2)) * int(x[2].numel())
                    for b, x in zip(bs, systems))
        line.update(metric="RGF energy-points/s over ragged block sizes (one CUDA graph)",
                    unit="points/s", value=n_pts * args.steps / (ms / 1e3),
                    ms_per_step=ms / args.steps, dtype="bf16-integers->fp32 (fp64 storage)",
                    config={"workload": f"{n_s} samples of the b = 200..800 alloy set (N = 70), "
                                        f"4 k-points x {n_e} energies each: {n_pts} points",
                            "systems_per_block_size": counts,
                            "grouping": "one batched launch chain per block size on its own "
                                        "stream, all captured in one CUDA graph",
                            "sequential_groups_ms": ms_seq,
                            "speedup_vs_sequential_groups": ms_seq / (ms / args.steps),
                            "algorithmic_tflops": flops * args.steps / (ms / 1e3) / 1e12})
    print(json.dumps(line), flush=True)


def main():
    args = parse()
    if args.impl == "reference":
        run_reference(args)
        return
    if args.workload != "rgf":
        run_side(args)
        return
    import torch
    import paper_1510_04686_gb300 as negf

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl")
    else:
        dist = None
        torch.cuda.set_device(0)
    negf._build.build()
    negf.library()
    dvc = torch.device("cuda", torch.cuda.current_device())

    dev_np, Hd, Hu, ks, wk, E, wE = build_hamiltonians()
    Hd_t = torch.as_tensor(Hd, device=dvc)
    Hu_t = torch.as_tensor(np.ascontiguousarray(Hu), device=dvc)
    device = negf.Device(Hd_t, Hu_t)
    prec = {"mixed": negf.PREC_MIXED, "mixed40": negf.PREC_MIXED_40,
            "mixed56": negf.PREC_MIXED_56, "fp64": negf.PREC_FP64}[args.precision]
    mixed = prec != negf.PREC_FP64
    P = args.points_per_step
    tuned = None
    if mixed:
        if args.tc_config is not None:
            tuned = negf.tc_config(args.tc_config)
        else:
            # pick the tensor-core GEMM configuration for this block size and batch (untimed; large
            # batches have none to pick)
            from paper_1510_04686_gb300 import autotune
            tuned = autotune.tune_tc(WORK["b"], P)["config"]
    opt = negf.options(precision=prec, chunk=P)
    total_steps = args.warmup + args.steps
    # per-step index tensors (ranks solve disjoint points)
    step_E, step_sys, step_w = [], [], []
    for s in range(total_steps):
        kk, ee = rank_points(s, rank, world, P)
        step_E.append(torch.as_tensor(E[ee], device=dvc))
        step_sys.append(torch.as_tensor(kk.astype(np.int32), device=dvc))
        step_w.append(torch.as_tensor(wE[ee] * wk[kk], device=dvc))
    NB = WORK["N"] * WORK["b"]
    n_int = torch.empty((total_steps, 1, NB), dtype=torch.float64, device=dvc)
    j_int = torch.empty((total_steps, 1, WORK["N"] - 1), dtype=torch.float64, device=dvc)

    def step(s):
        lead = negf.lead_selfenergy(device, step_E[s], step_sys[s], opt)
        out = negf.rgf_solve(device, step_E[s], step_sys[s], lead["sigma_R"], lead["sigma_L"], opt)
        lib = negf.library()
        st = torch.cuda.current_stream().cuda_stream
        import ctypes
        lib.negf_integrate(P, NB, 1, ctypes.c_void_p(step_w[s].data_ptr()), None,
                           ctypes.c_void_p(out["density"].data_ptr()),
                           ctypes.c_void_p(n_int[s].data_ptr()), ctypes.c_void_p(st))
        lib.negf_integrate(P, WORK["N"] - 1, 1, ctypes.c_void_p(step_w[s].data_ptr()), None,
                           ctypes.c_void_p(out["current"].data_ptr()),
                           ctypes.c_void_p(j_int[s].data_ptr()), ctypes.c_void_p(st))
        return out

    for s in range(args.warmup):
        step(s)
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    negf.profile_reset()
    negf.profile(True)
    l0 = negf.launch_count()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with Clocks(torch.cuda.current_device()) as clk:
        torch.cuda.synchronize()
        torch.cuda.nvtx.range_push("bench_timed")  # lets a profiler select the timed launches
        ev0.record()
        for s in range(args.warmup, total_steps):
            step(s)
        ev1.record()
        torch.cuda.synchronize()
        torch.cuda.nvtx.range_pop()
    launches = negf.launch_count() - l0
    negf.profile(False)
    ms = max_over_ranks(ev0.elapsed_time(ev1), dist, dvc)
    # one more step without the per-launch profiling events (instrumentation overhead check)
    torch.cuda.synchronize()
    ev2, ev3 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    ev2.record()
    step(args.warmup)
    ev3.record()
    torch.cuda.synchronize()
    ms_noprof = ev2.elapsed_time(ev3)
    n_launch, tc_ms, alg, hw = negf.profile_read(negf.PROF_TC_GEMM)
    sl_n, sl_ms, _, _ = negf.profile_read(negf.PROF_SLICE)
    inv_n, inv_ms, _, _ = negf.profile_read(negf.PROF_INV)
    pan_n, pan_ms, _, _ = negf.profile_read(negf.PROF_GJ_PANEL)
    value = aggregate_rate(args.steps, P, world, ms)

    pk, pk_kind = peaks()
    peak_bf16 = pk.get("bf16_tflops_sustained", PEAKS_FALLBACK["bf16_tflops_sustained"])
    achieved = (alg / (tc_ms / 1e3)) / 1e12 if tc_ms > 0 else None
    roofline = {
        "kernel": "k_crt_gemm (tcgen05 complex GEMM on BF16 residues)",
        "bound": "tensor", "unit": "TFLOP/s",
        "achieved": achieved, "peak": peak_bf16,
        "frac": (achieved / peak_bf16) if achieved else None,
        "peak_kind": f"bf16 dense sustained, {pk_kind}",
        "algorithmic_flops_per_launch": alg / max(n_launch, 1),
        "avg_launch_ms": tc_ms / max(n_launch, 1), "launches": n_launch,
        "issued_bf16_tflops": (hw / (tc_ms / 1e3)) / 1e12 if tc_ms > 0 else None,
        "issued_frac": ((hw / (tc_ms / 1e3)) / 1e12 / peak_bf16) if tc_ms > 0 else None,
        "share_of_step": tc_ms / ms if ms > 0 else None,
        "slicing_share_of_step": sl_ms / ms if ms > 0 else None,
        "inverse_elimination_share_of_step": inv_ms / ms if ms > 0 else None,
        "gj_panel_share_of_step": pan_ms / ms if ms > 0 else None,
        "traffic": (TC_DRAM_BYTES_PER_ITEM_B400 * (alg / max(n_launch, 1)) / (8.0 * WORK["b"] ** 3)
                    if TC_DRAM_BYTES_PER_ITEM_B400 and WORK["b"] == 400 and n_launch
                    and prec == negf.PREC_MIXED else None),
        "traffic_unit": "bytes per launch (DRAM read + write, ncu capture of 64 items scaled "
                        "to the launch's items)",
    }
    line = {
        "metric": METRIC, "value": value, "unit": "points/s", "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": (f"bf16-integers->fp32 (fp64 storage; sweeps {tier_bits(negf, prec)}-bit, "
                  "lead decimation 56/48/40-bit by doubling step)") if mixed else "f64",
        "data": "synthetic",
        "config": {"workload": WORK["name"], "points_per_step": P, "precision": args.precision,
                   "l2": "inputs > L2: each step streams 358 MB of H blocks",
                   "parallelism": f"points sharded over {world} rank(s), no data-path collective", "tc_config": tuned},
        "gpu_launches": int(launches), "clocks": clk.summary(), "roofline": roofline,
        "ms_per_step_profiling_off": ms_noprof,
    }
    if rank == 0 and not args.no_extras:
        line.update(extras(args, negf, torch, device, dvc, Hd, dev_np, E, wE, wk, prec))
        if "fp64_gpu" in line:
            line["speedup_vs_fp64_gpu"] = value / world / line["fp64_gpu"]["value"]
        if not args.no_golden and os.path.exists(GOLDEN):
            line["rel_err_vs_oracle_kslice"] = golden_check(negf, torch, device, dvc, E, wE,
                                                            prec, P)
    if rank == 0:
        print(json.dumps(line), flush=True)
    if dist:
        dist.destroy_process_group()


def extras(args, negf, torch, device, dvc, Hd, dev_np, E, wE, wk, prec):
    """Side measurements on rank 0: end-to-end with host buffers, FP64 GPU form, CPU oracle and
    the accuracy of this run's points against the oracle."""
    import oracle as O
    out = {}
    n_tot = WORK["n_E"] * WORK["n_k"]
    P = args.points_per_step
    NB = WORK["N"] * WORK["b"]
    # ---- end to end: pinned host inputs -> device -> solve -> host results, per step
    kk, ee = point_index(n_tot, 7 * P, P)
    k0 = int(kk[0])
    Hd_h = torch.as_tensor(Hd[k0][None]).pin_memory()
    Hu_h = torch.as_tensor(dev_np.T[None]).pin_memory()
    E_h = torch.as_tensor(E[ee]).pin_memory()
    sys_h = torch.zeros(P, dtype=torch.int32).pin_memory()
    dens_h = torch.empty((P, NB), dtype=torch.float64).pin_memory()
    cur_h = torch.empty((P, WORK["N"] - 1), dtype=torch.float64).pin_memory()
    tr_h = torch.empty((P,), dtype=torch.float64).pin_memory()
    opt = negf.options(precision=prec, chunk=P)
    e2e_steps = 2
    h2d = Hd_h.numel() * 16 + Hu_h.numel() * 16 + P * 8 + P * 4
    d2h = dens_h.numel() * 8 + cur_h.numel() * 8 + P * 8
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(e2e_steps):
        hd = Hd_h.to(dvc, non_blocking=True)
        hu = Hu_h.to(dvc, non_blocking=True)
        Et = E_h.to(dvc, non_blocking=True)
        st = sys_h.to(dvc, non_blocking=True)
        d1 = negf.Device(hd, hu)
        lead = negf.lead_selfenergy(d1, Et, st, opt)
        r = negf.rgf_solve(d1, Et, st, lead["sigma_R"], lead["sigma_L"], opt)
        dens_h.copy_(r["density"], non_blocking=True)
        cur_h.copy_(r["current"], non_blocking=True)
        tr_h.copy_(r["transmission"], non_blocking=True)
        torch.cuda.synchronize()
    dt = time.perf_counter() - t0
    out["e2e"] = {"value": e2e_steps * P / dt, "unit": "points/s", "h2d_bytes_per_step": int(h2d),
                  "d2h_bytes_per_step": int(d2h), "steps": e2e_steps}
    # ---- accuracy against the oracle and CPU baseline on a bounded sample
    cp = max(1, args.cpu_points)
    kk, ee = point_index(n_tot, 1234, cp)
    Et = torch.as_tensor(E[ee], device=dvc)
    st = torch.as_tensor(kk.astype(np.int32), device=dvc)
    lead = negf.lead_selfenergy(device, Et, st, negf.options(precision=prec))
    g = negf.rgf_solve(device, Et, st, lead["sigma_R"], lead["sigma_L"], negf.options(precision=prec))
    g = {k: v.cpu().numpy() for k, v in g.items() if v is not None}
    t0 = time.perf_counter()
    refs = [O.solve_point(Hd[kk[i]], dev_np.T, E[ee[i]], WORK["eta"], None) for i in range(cp)]
    dt = time.perf_counter() - t0
    out["cpu_baseline"] = {"value": cp / dt, "unit": "points/s", "cores": _blas_threads(),
                           "kind": "oracle", "blas": _blas_info(), "host_cores": os.cpu_count(),
                           "sample": f"{cp} (E,k) points of the workload, numpy complex128"}
    t1 = _oracle_one_core(kk[0], ee[0])
    if t1:
        out["cpu_baseline"]["single_core"] = {"value": 1.0 / t1, "unit": "points/s", "cores": 1,
                                              "sample": "the first of those points, BLAS on one "
                                                        "thread"}

    def rel(a, b):
        return float(np.abs(a - b).max() / max(np.abs(b).max(), 1e-300))
    d_ref = np.array([r_["density"] for r_ in refs])
    j_ref = np.array([r_["current"] for r_ in refs])
    T_ref = np.array([r_["transmission"] for r_ in refs])
    out["rel_err_vs_oracle"] = {
        "density_per_point": rel(g["density"], d_ref),
        "current_per_point": rel(g["current"], j_ref),
        "transmission": float(np.abs(g["transmission"] - T_ref).max() / max(1.0, np.abs(T_ref).max())),
        "points": cp, "norm": "inf-norm relative over the sample",
    }
    # ---- FP64 GPU form on a subset
    if prec != negf.PREC_FP64 and args.fp64_points > 0:
        fpn = args.fp64_points
        kk, ee = point_index(n_tot, 99, fpn)
        Et = torch.as_tensor(E[ee], device=dvc)
        st = torch.as_tensor(kk.astype(np.int32), device=dvc)
        o64 = negf.options(precision=negf.PREC_FP64, chunk=fpn)
        torch.cuda.synchronize()
        ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        ev0.record()
        lead = negf.lead_selfenergy(device, Et, st, o64)
        negf.rgf_solve(device, Et, st, lead["sigma_R"], lead["sigma_L"], o64)
        ev1.record()
        torch.cuda.synchronize()
        sec = ev0.elapsed_time(ev1) / 1e3
        v64 = fpn / sec
        # executed block work of the FP64 form (complex b^3 GEMM-equivalents, an inverse counted
        # as one): decimation steps per side as run, then the sweeps of negf_rgf_solve
        N, b = WORK["N"], WORK["b"]
        iters = float(lead["iters"].sum().item())
        eq = iters * 7 + fpn * (2 * 2 + 4) + fpn * (2 + 5 * (N - 2) + 7 + 2 + 6 * (N - 1) + N)
        flops64 = eq * 8.0 * b ** 3
        peak64 = fp64_peak(torch)
        out["fp64_gpu"] = {"value": v64, "unit": "points/s", "points": fpn,
                           "sample": f"{fpn} points of the workload in one batch (the FP64 "
                                     "form's rate saturates with the batch: 0.93 / 1.35 / 1.59 "
                                     "points/s at 4 / 16 / 64 points)",
                           "roofline": {"bound": "fp64", "unit": "TFLOP/s",
                                        "achieved": flops64 / sec / 1e12, "peak": peak64,
                                        "frac": flops64 / sec / 1e12 / peak64,
                                        "peak_kind": "cuBLAS DGEMM 8192^3 measured in this run",
                                        "executed_flops_per_point": flops64 / fpn}}
    return out


def fp64_peak(torch):
    """FP64 dense rate of this GPU: cuBLAS DGEMM of 8192^3 through torch, best of 3."""
    n = 8192
    a = torch.randn(n, n, dtype=torch.float64, device="cuda")
    b = torch.randn(n, n, dtype=torch.float64, device="cuda")
    a @ b
    torch.cuda.synchronize()
    best = 0.0
    for _ in range(3):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        a @ b
        e1.record()
        torch.cuda.synchronize()
        best = max(best, 2.0 * n ** 3 / (e0.elapsed_time(e1) / 1e3) / 1e12)
    del a, b
    return best


def tier_bits(negf, prec):
    return {negf.PREC_MIXED: 48, negf.PREC_MIXED_40: 40, negf.PREC_MIXED_56: 56}.get(prec, 64)


def golden_check(negf, torch, device, dvc, E, wE, prec, P):
    """Accuracy of this run's options against stored oracle values of the same device: every
    energy of one k-slice (energy integrals of the per-atom density and of the bond currents,
    T(E)) and per-point values at 64 stored points (48 on that slice, 16 on the -k slice)."""
    with open(GOLDEN) as fh:
        gd = json.load(fh)
    N, b = WORK["N"], WORK["b"]
    km, kp = gd["k_main"], gd["k_partner"]
    opt = negf.options(precision=prec, chunk=P)
    n_E = len(E)
    dens_int = torch.zeros((1, N * b), dtype=torch.float64, device=dvc)
    cur_int = torch.zeros((1, N - 1), dtype=torch.float64, device=dvc)
    T = np.empty(n_E)
    per = {}
    want = {(q["k_index"], q["energy_index"]) for q in gd["points"]}
    jobs = [(km, np.arange(s, min(s + P, n_E))) for s in range(0, n_E, P)]
    part = sorted(e for (k, e) in want if k == kp)
    if part:
        jobs.append((kp, np.array(part)))
    for k, idx in jobs:
        Et = torch.as_tensor(E[idx], device=dvc)
        st = torch.full((len(idx),), k, dtype=torch.int32, device=dvc)
        lead = negf.lead_selfenergy(device, Et, st, opt)
        r = negf.rgf_solve(device, Et, st, lead["sigma_R"], lead["sigma_L"], opt)
        if k == km:
            w = torch.as_tensor(wE[idx], device=dvc)
            dens_int += negf.integrate(r["density"], w)
            cur_int += negf.integrate(r["current"], w)
            T[idx] = r["transmission"].cpu().numpy()
        dn = r["density"].reshape(len(idx), N, b).sum(dim=2).cpu().numpy()
        cu = r["current"].cpu().numpy()
        tr = r["transmission"].cpu().numpy()
        for q, e in enumerate(idx):
            if (k, int(e)) in want:
                per[(k, int(e))] = (dn[q], cu[q], tr[q])
    atoms = dens_int.reshape(-1, 10).sum(dim=1).cpu().numpy()
    jint = cur_int.reshape(-1).cpu().numpy()

    def rel(a, ref):
        # a point with zero density (E above mu + 1 eV: f = 0 exactly) compares absolutely
        return float(np.abs(np.asarray(a) - np.asarray(ref)).max()
                     / max(np.abs(ref).max(), 1e-300))
    jscale = max(np.abs(q["current"]).max() for q in gd["points"] if q["k_index"] == km)
    pd, pj, pt = [], [], []
    for q in gd["points"]:
        dn, cu, tr = per[(q["k_index"], q["energy_index"])]
        pd.append(rel(dn, q["slab_density"]))
        pj.append(float(np.abs(cu - np.asarray(q["current"])).max() / jscale))
        pt.append(abs(tr - q["transmission"]) / max(1.0, abs(q["transmission"])))
    Tref = np.asarray(gd["transmission_main"])
    return {
        "integrated_density_per_atom": rel(atoms, gd["integrated_atom_density_main"]),
        "integrated_current": rel(jint, gd["integrated_current_main"]),
        "transmission_max": float(np.abs(T - Tref).max() / max(1.0, np.abs(Tref).max())),
        "points": len(pd), "slab_density_per_point_max": max(pd),
        "current_per_point_max": max(pj), "transmission_per_point_max": max(pt),
        "norm": ("inf-norm relative; per-point current relative to the largest stored current "
                 "of the slice (outside the bias window j(E) ~ (f_L - f_R) T vanishes)"),
        "sample": f"k-slice {km} (512 energies, trapezoid weights) + {len(part)} points of slice "
                  f"{kp}, stored oracle values",
    }


if __name__ == "__main__":
    main()
