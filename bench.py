"""Benchmark of the Kubo-transport hot path on GB300.

Default workload (one GPU): the FP64 honeycomb lattice of 4096 x 2048 cells
(N = 16,777,216 orbitals, t = -2.7 eV, Anderson disorder in [-1, 1] eV,
dE = 9.555 eV), one random-phase vector, M = 3000 Chebyshev moments, time step
dt = 2 hbar/|t| (N_p = 29 Bessel orders).  One step = one time step of the VAC
and MSD runs: the VAC row (velocity, M fused Chebyshev orders against V a) and
the U(-dt) evolution of (a, b); the MSD step (coupled [X,U] evolution of
(p, p_X)) and its row (M orders); and the kernel-polynomial reconstruction of
both rows on 1001 energies.  Metric: orbital-moments per second, N * 2M per
step.  ``--impl reference`` times the serial FP64 oracle on the host cores on
a bounded sample of the same workload (a few moments at full N).
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

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import gqt_synth as S  # noqa: E402

METRIC = "orbital-moments/s (H.phi products)"
UNIT = "orbital*moments/s"


def _dist():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


class Clocks:
    """nvidia-smi sampling of SM clocks and throttle reasons during the timed region."""

    Q = ("clocks.sm,clocks.max.sm,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.idx = gpu_index
        self.p = None

    def __enter__(self):
        try:
            self.p = subprocess.Popen(["nvidia-smi", "-i", str(self.idx), f"--query-gpu={self.Q}",
                                       "--format=csv,noheader,nounits", "-lms", "200"], stdout=subprocess.PIPE,
                                      stderr=subprocess.DEVNULL, text=True)
        except (OSError, FileNotFoundError):
            self.p = None
        return self

    def __exit__(self, *a):
        self.out = ""
        if self.p is not None:
            self.p.terminate()
            try:
                self.out, _ = self.p.communicate(timeout=5)
            except subprocess.TimeoutExpired:
                self.p.kill()
                self.out, _ = self.p.communicate()

    def summary(self):
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in (self.out or "").splitlines():
            f = [x.strip() for x in line.split(",")]
            if len(f) < 7:
                continue
            try:
                sm.append(float(f[0]))
                mx.append(float(f[1]))
            except ValueError:
                continue
            for n, v in zip(names, f[3:7]):
                if v.lower() == "active":
                    reasons.add(n)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unavailable"]}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
                "samples": len(sm)}


def _peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured"
    except (OSError, KeyError, ValueError):
        return 6800.0, "fallback"


def measured_traffic(family: str, n_orbitals: int):
    """Per-launch DRAM traffic of a moment-kernel family scaled to n_orbitals, from
    the committed ncu capture; None when any of its kernel sources changed since."""
    import hashlib
    try:
        with open(os.path.join(ROOT, "profiles", "traffic_moment_kernels.json")) as f:
            d = json.load(f)
        fam = d["families"][family]
        for src, sha in fam["kernel_sources"].items():
            with open(os.path.join(ROOT, src), "rb") as f:
                if hashlib.sha256(f.read()).hexdigest() != sha:
                    return None
        return (fam["dram_read_bytes"] + fam["dram_write_bytes"]) / fam["n_orbitals"] * n_orbitals
    except (OSError, KeyError, ValueError):
        return None


def workload(small: bool, cells: str | None = None, moments: int | None = None):
    """The honeycomb FP64 workload; ``cells`` ('L1xL2') and ``moments`` shrink it for
    profiling captures (the default is the full 4096 x 2048, M = 3000 case)."""
    w = S.config(1, small=small)
    if cells:
        L1, L2 = (int(x) for x in cells.lower().split("x"))
        w.lattice_args = dict(w.lattice_args, L1=L1, L2=L2)
        w.name = f"honeycomb{L1}x{L2}_fp64"
    if moments:
        w.M = int(moments)
    lat = S.build_lattice(w.lattice_args, w.seed)
    return w, lat


def bytes_per_orbital_cheb(K: int, fp64: bool, hop_real: bool, R: int) -> float:
    """Algorithmic bytes per orbital per Chebyshev order of the fused moment kernel:
    per vector element T_{m-1} (gather counted once), T_{m-2}, T_m, l (4 complex
    values); H~ once per site: K int32 indices, K hoppings, 1 diagonal."""
    v = 16 if fp64 else 8
    s = 8 if fp64 else 4
    hop = s if hop_real else 2 * s
    return 4 * v * R + K * (4 + hop) + s


def bytes_per_orbital_pair(K: int, hop_real: bool, R: int) -> float:
    """Algorithmic bytes per orbital per step of the two-recurrence kernel (FP64):
    per vector element A and B of orders k-1 (gather counted once), k-2 and k
    (6 complex values); H~ once per site."""
    return 6 * 16 * R + K * (4 + (8 if hop_real else 16)) + 8


def bytes_per_orbital_tiled(K: int, hop_real: bool, pair: bool, uniform: bool = False) -> float:
    """Algorithmic bytes per orbital per launch of the temporally blocked kernel
    (two orders): per chain T_m and T_{m-1} read and T_{m+1}, T_{m+2} written
    (4 complex FP64-sized values), H~ once per site (K hoppings and the
    diagonal as FP32 pairs, no index array; no hoppings either when they all
    hold one value)."""
    return (2 if pair else 1) * 4 * 16 + (0 if uniform else K * (8 if hop_real else 16)) + 8


def fp64_fma_per_orbital(K: int, hop_real: bool, dot: str) -> int:
    """Algorithmic FP64 fused multiply-adds per orbital per launch: the recurrence
    (diagonal 2, each neighbour 2 real or 4 complex) plus the moment dot products
    (Re <l|T_m>: 2; the l = r kernel's <u|u> and Re <u_m|u_m-1>: 4); the
    two-recurrence kernel runs two recurrences and two Re dots (4)."""
    rec = 2 + K * (2 if hop_real else 4)
    return {"re": rec + 2, "dbl": rec + 4, "pair": 2 * rec + 4}[dot]


def df_fp32_ops_per_orbital(K: int, hop_real: bool, kind: str, uniform: bool = False) -> int:
    """FP32-pipe instructions per orbital per launch of the paired-FP32 kernels: one
    pair multiply-accumulate (TwoProduct by FMA, three FMAs for the low parts, TwoSum
    and two adds) is 12; a recurrence takes 2 of them per real diagonal or
    neighbour term on each of Re, Im (4 for complex hoppings) and two 6-instruction
    renormalisations; each Re dot takes 2 (24 instructions).  With one common
    hopping a recurrence instead sums the K neighbour pairs (K - 1 pair additions
    of 8 on each of Re, Im) before two multiply-accumulates per part.  The l = r
    kernel runs one recurrence and two dots, the two-recurrence kernel two and two."""
    if uniform:
        rec = 2 * (8 * (K - 1) + 2 * 12) + 12
    else:
        rec = 12 * (2 + K * (2 if hop_real else 4)) + 12
    return {"dbl": rec + 48, "pair": 2 * rec + 48, "re": rec + 24}[kind]


def fp32_batched(args, g, torch):
    """Batched FP32 form vs plain FP64 on the simple-cubic Anderson model L = 256
    (N = 16,777,216, 6 neighbours, t = -1, W = 16.5): DOS moments for R = 32 FP32
    vectors in one launch sequence vs one FP64 vector, per orbital-moment."""
    w = S.config(2, small=args.small)
    L = args.fp32_L or w.lattice_args["L"]
    M = args.fp32_moments
    out = {"workload": f"cubic{L}_W16.5", "moments": M}
    res = {}
    for prec, R in ((g.GQT_FP32_ACC64, w.R), (g.GQT_FP64, 1)):
        ham = g.gqt_build_hamiltonian(None, w.energy_scale, prec, kind=g.GQT_LATTICE_CUBIC, L1=L, t=-1.0,
                                      W=16.5, seed=w.seed)
        cd = torch.complex64 if prec == g.GQT_FP32_ACC64 else torch.complex128
        phi = torch.empty((ham.n, R), dtype=cd, device="cuda")
        g.gqt_random_phase(ham, w.seed, R, phi)
        mu = torch.empty((1, R, M), dtype=torch.float64, device="cuda")
        g.gqt_dos_moments(ham, phi, R, M, mu)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(2):
            g.gqt_dos_moments(ham, phi, R, M, mu)
        e1.record()
        torch.cuda.synchronize()
        t = e0.elapsed_time(e1) / 2 * 1e-3
        res[prec] = (ham.n * R * M / t, mu[0, 0].cpu().numpy(), t, R, ham.n)
        del phi, ham
        torch.cuda.empty_cache()
    # ragged batch: 48 realisations, L ~ U{32..96}, one block-diagonal launch sequence
    if not args.small and not args.no_ragged:
        t0 = time.perf_counter()
        blk = S.ragged_cubic(48, 32, 96, -1.0, 16.5, w.seed)
        ham = g.gqt_build_hamiltonian(blk, w.energy_scale, g.GQT_FP32_ACC64)
        t_build = time.perf_counter() - t0
        phi = torch.empty((ham.n, 1), dtype=torch.complex64, device="cuda")
        g.gqt_random_phase(ham, w.seed, 1, phi)
        mu = torch.empty((ham.nseg, 1, M), dtype=torch.float64, device="cuda")
        g.gqt_dos_moments(ham, phi, 1, M, mu)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        g.gqt_dos_moments(ham, phi, 1, M, mu)
        e1.record()
        torch.cuda.synchronize()
        tr = e0.elapsed_time(e1) * 1e-3
        out["ragged"] = {"realisations": int(ham.nseg), "n_orbitals": int(ham.n), "moments": M,
                         "orbital_moments_per_s": ham.n * M / tr, "ms": tr * 1e3, "build_s": t_build,
                         "mu0_per_segment_max_dev": float((mu[:, 0, 0] - 1.0).abs().max())}
        del blk, ham, phi
        torch.cuda.empty_cache()
    v32, mu32, t32, R32, n = res[g.GQT_FP32_ACC64]
    v64, mu64, t64, _, _ = res[g.GQT_FP64]
    # FP32 storage reads 8 B per vector element (T_m-1, T_m-2, T_m) and H~ once for all R vectors
    bpo32 = (3 * 8 * R32 + 6 * (4 + 4) + 4) / R32
    hbm, _ = _peaks()
    out.update({"fp32_R": R32, "fp32_orbital_moments_per_s": v32, "fp64_orbital_moments_per_s": v64,
                "speedup": v32 / v64, "fp32_ms": t32 * 1e3, "fp64_ms": t64 * 1e3,
                "fp32_hbm_frac": v32 / 2 * bpo32 / 1e9 / hbm,
                "dos_moment_error_fp32_vs_fp64": float(np.max(np.abs(mu32 - mu64)) / np.max(np.abs(mu64)))})
    return out


def precision_table(args, g, torch):
    """Per-result error of the FP32-storage form against the FP64 path on the
    honeycomb 2048 x 2048 lattice with 1% vacancies (N = 8,388,608, W = 0.5 eV,
    R = 8, M = 4000, dt = 2 hbar/|t|): DOS moments and reconstructed DOS, VAC
    moments, rho*C_vv(E, t) and sigma_VAC(E, t) over Nt steps (default 200, the
    workload's count), MSD moments, rho*dX^2(E) and sigma_MSD over the first
    --precision-msd-steps steps.  The FP32 form runs all R vectors in one batched
    handle; the FP64 reference runs the first --precision-ref-vectors of the same
    random-phase vectors one at a time (R = 1 rows of an FP64 handle).  Errors are
    normalised L-infinity over n (moments) or E, per vector, maximised over the
    reference vectors and rows; the VAC row error is also reported per step."""
    w = S.config(3, small=args.small)
    L1 = args.precision_L or w.lattice_args["L1"]
    M, R, Nt = args.precision_moments or w.M, w.R, args.precision_steps
    nref = max(1, min(args.precision_ref_vectors, R))
    Nm = max(1, min(args.precision_msd_steps, Nt))
    dE = w.energy_scale
    E = torch.from_numpy(w.energies).cuda()
    dts = np.full(Nt, w.dt)

    def run(prec, R_, first):
        ham = g.gqt_build_hamiltonian(None, dE, prec, kind=g.GQT_LATTICE_HONEYCOMB, L1=L1, L2=L1, t=-2.7, W=0.5,
                                      vacancy_frac=0.01, seed=w.seed)
        g.gqt_set_temporal_blocking(ham, args.temporal_blocking)
        nO = ham.n / ham.volume
        cd = torch.complex128 if prec == g.GQT_FP64 else torch.complex64
        phi = torch.empty((ham.n, R_), dtype=cd, device="cuda")
        g.gqt_random_phase(ham, w.seed, R_, phi, first_vector=first)
        dos = torch.empty((1, R_, M), dtype=torch.float64, device="cuda")
        g.gqt_dos_moments(ham, phi, R_, M, dos)
        a, b = torch.empty_like(phi), torch.empty_like(phi)
        g.gqt_vac_init(ham, phi, a, b, R_)
        vac = torch.empty((Nt, 1, R_, M), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        g.gqt_vac_moments(ham, a, b, R_, dts, M, vac)
        torch.cuda.synchronize()
        t_vac = time.perf_counter() - t0
        p, px = torch.empty_like(phi), torch.empty_like(phi)
        g.gqt_msd_init(ham, phi, p, px, R_)
        msd = torch.empty((Nm, 1, R_, M), dtype=torch.float64, device="cuda")
        g.gqt_msd_moments(ham, p, px, R_, dts[:Nm], M, msd)
        out = {"dos_mu": dos[0].cpu().numpy(), "vac_mu": vac[:, 0].cpu().numpy(), "msd_mu": msd[:, 0].cpu().numpy(),
               "t_vac": t_vac, "n": ham.n}
        # reconstruction of every vector's rows, then sigma over time
        for key, rows in (("dos", dos[0]), ("vac", vac[:, 0].transpose(0, 1).reshape(R_ * Nt, M)),
                          ("msd", msd[:, 0].transpose(0, 1).reshape(R_ * Nm, M))):
            rec = torch.empty((rows.shape[0], E.numel()), dtype=torch.float64, device="cuda")
            g.gqt_kpm_reconstruct(rows.contiguous(), E, dE, nO, rec)
            out[key] = rec
        out["vac"] = out["vac"].view(R_, Nt, -1)
        out["msd"] = out["msd"].view(R_, Nm, -1)
        sv, sm = [], []
        for r in range(R_):
            s1 = torch.empty_like(out["vac"][r])
            g.gqt_sigma_vac(out["vac"][r].contiguous(), dts, s1)
            s2 = torch.empty_like(out["msd"][r])
            g.gqt_sigma_msd(out["msd"][r].contiguous(), dts[:Nm], s2)
            sv.append(s1)
            sm.append(s2)
        out["sigma_vac"], out["sigma_msd"] = torch.stack(sv), torch.stack(sm)
        for k in ("dos", "vac", "msd", "sigma_vac", "sigma_msd"):
            out[k] = out[k].cpu().numpy()
        del ham, phi, a, b, p, px
        torch.cuda.empty_cache()
        return out

    def nerr(x, y):
        return float(np.max(np.abs(x - y)) / max(np.max(np.abs(y)), 1e-300))

    r32 = run(g.GQT_FP32_ACC64, R, 0)
    refs = [run(g.GQT_FP64, 1, r) for r in range(nref)]
    tab = {}
    for key, axis_r in (("dos_mu", 0), ("dos", 0)):
        tab[key] = max(nerr(r32[key][r], refs[r][key][0]) for r in range(nref))
    for key in ("vac_mu", "msd_mu"):
        tab[key] = max(nerr(r32[key][k, r], refs[r][key][k, 0]) for r in range(nref) for k in range(r32[key].shape[0]))
    for key in ("vac", "msd", "sigma_vac", "sigma_msd"):
        tab[key] = max(nerr(r32[key][r], refs[r][key][0]) for r in range(nref))
    marks = sorted({k for k in (0, 1, 2, 5, 10, 20, 50, 100, 150, Nt - 1) if k < Nt})
    curve = {str(k): max(nerr(r32["vac_mu"][k, r], refs[r]["vac_mu"][k, 0]) for r in range(nref)) for k in marks}
    sig_curve = {str(k): max(nerr(r32["sigma_vac"][r][k], refs[r]["sigma_vac"][0][k]) for r in range(nref))
                 for k in marks if k > 0}
    n = r32["n"]
    v32 = n * R * M * Nt / r32["t_vac"]
    t64 = float(np.mean([x["t_vac"] for x in refs]))
    v64 = n * M * Nt / t64
    return {"workload": f"honeycomb{L1}x{L1}_vac1pct_R{R}_M{M}", "vac_steps": Nt, "msd_steps": Nm,
            "reference": f"FP64 handle, R = 1 rows (paired-FP32 moment arithmetic, FP64 evolution), vectors 0..{nref - 1}",
            "errors_fp32_vs_fp64": tab, "vac_row_error_by_step": curve, "sigma_vac_error_by_step": sig_curve,
            "vac_seconds_fp32_R%d" % R: r32["t_vac"], "vac_seconds_fp64_per_vector": t64,
            "vac_orbital_moments_per_s_fp32": v32, "vac_orbital_moments_per_s_fp64": v64,
            "vac_speedup_fp32": v32 / v64, "temporal_blocking": args.temporal_blocking}


def latency(args, g, torch):
    """Latency-bound workloads.  C1: honeycomb 32 x 32 (N = 2048) VAC + MSD, 10 steps
    of 1 hbar/|t|, M = 512, with CUDA graphs on and off (microseconds per moment).
    C5: honeycomb 256 x 256 (N = 131072), sigma_VAC(E, t_50) loss and its gradient
    with respect to N on-site energies and 3N/2 hoppings (M = 1024)."""
    from paper_1705_01387_gb300 import autograd as AG
    out = {}
    w = S.config(0)
    lat = S.build_lattice(w.lattice_args, w.seed)
    ham = g.gqt_build_hamiltonian(lat, w.energy_scale)
    phi = torch.empty((lat.n, 1), dtype=torch.complex128, device="cuda")
    g.gqt_random_phase(ham, w.seed, 1, phi)
    dts = np.full(w.n_steps, w.dt)
    mu = torch.empty((w.n_steps, 1, 1, w.M), dtype=torch.float64, device="cuda")
    a, b, p, px = (torch.empty_like(phi) for _ in range(4))
    for graphs in (True, False):
        g.gqt_set_graphs(ham, graphs)
        times = []
        for rep in range(4):
            g.gqt_vac_init(ham, phi, a, b, 1)
            g.gqt_msd_init(ham, phi, p, px, 1)
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            g.gqt_vac_moments(ham, a, b, 1, dts, w.M, mu)
            g.gqt_msd_moments(ham, p, px, 1, dts, w.M, mu)
            torch.cuda.synchronize()
            times.append(time.perf_counter() - t0)
        t = min(times[1:])
        out["c1_graphs" if graphs else "c1_direct"] = {"seconds": t,
                                                       "us_per_moment": t / (2 * w.n_steps * w.M) * 1e6}
    w5 = S.config(4)
    lat5 = S.build_lattice(w5.lattice_args, w5.seed)
    E = torch.from_numpy(w5.energies).cuda()
    wts = torch.exp(-E ** 2 / (2 * 0.5 ** 2))
    topo = AG.BondTopology.from_lattice(lat5)
    phi5 = torch.empty((lat5.n, 1), dtype=torch.complex128, device="cuda")
    ham5 = g.gqt_build_hamiltonian(lat5, w5.energy_scale)
    g.gqt_random_phase(ham5, w5.seed, 1, phi5)
    spec = AG.VacSigmaLossSpec(topo, w5.energy_scale, phi5, np.full(w5.n_steps - 1, w5.dt), w5.M, E, wts)
    onsite = torch.from_numpy(lat5.onsite.copy()).requires_grad_(True)
    hop = torch.full((topo.nbonds,), -2.7, dtype=torch.float64, requires_grad=True)
    times = []
    for rep in range(2):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        L = AG.GqtVacSigmaLoss.apply(onsite, hop, spec)
        L.backward()
        torch.cuda.synchronize()
        times.append(time.perf_counter() - t0)
    out["c5_loss_and_grad"] = {"seconds": min(times), "n_orbitals": lat5.n, "n_bonds": topo.nbonds,
                               "moments": w5.M, "rows": w5.n_steps}
    return out


def paper_examples(args, g, torch):
    """The paper's two examples (Sec. 5), end to end on one GPU, with the host
    post-processing of Sec. 2.3.  Ex. 1: square lattice 2000 x 2000, W = 4, hopping
    -1, dE = 6.1, N_m = 1000, one vector, 20 steps of 0.2, VAC and MSD, energies
    -6..6 step 0.02.  Ex. 2: chain of 4,000,000 sites, W = 4, dE = 4.1, N_m = 500,
    two vectors, MSD over the 30 non-uniform steps 0.1..1.0, 1..10, 10..100,
    energies -4..4 step 0.02.  The paper reports about 3 minutes for both on a
    Tesla K40 (context only)."""
    from paper_1705_01387_gb300 import analysis as A
    out = {}

    def recon(rows, E, dE, nO):
        r = torch.empty((rows.shape[0], E.numel()), dtype=torch.float64, device="cuda")
        g.gqt_kpm_reconstruct(rows.contiguous(), E, dE, nO, r)
        return r

    # Example 1 (diffusive, Fig. 1)
    t0 = time.perf_counter()
    ham = g.gqt_build_hamiltonian(None, 6.1, g.GQT_FP64, kind=g.GQT_LATTICE_SQUARE, L1=2000, L2=2000, t=-1.0, W=4.0,
                                  seed=S.BASE_SEED + 10)
    nO = ham.n / ham.volume
    phi = torch.empty((ham.n, 1), dtype=torch.complex128, device="cuda")
    g.gqt_random_phase(ham, S.BASE_SEED + 10, 1, phi)
    torch.cuda.synchronize()
    t1 = time.perf_counter()
    M, Nt = 1000, 20
    dts = np.full(Nt, 0.2)
    E = torch.arange(-300, 301, dtype=torch.float64, device="cuda") * 0.02
    dos = torch.empty((1, 1, M), dtype=torch.float64, device="cuda")
    g.gqt_dos_moments(ham, phi, 1, M, dos)
    a, b = torch.empty_like(phi), torch.empty_like(phi)
    g.gqt_vac_init(ham, phi, a, b, 1)
    vac = torch.empty((Nt, 1, 1, M), dtype=torch.float64, device="cuda")
    g.gqt_vac_moments(ham, a, b, 1, dts, M, vac)
    p, px = torch.empty_like(phi), torch.empty_like(phi)
    g.gqt_msd_init(ham, phi, p, px, 1)
    msd = torch.empty((Nt, 1, 1, M), dtype=torch.float64, device="cuda")
    g.gqt_msd_moments(ham, p, px, 1, dts, M, msd)
    rd, rv, rm = recon(dos[0], E, 6.1, nO), recon(vac.view(Nt, M), E, 6.1, nO), recon(msd.view(Nt, M), E, 6.1, nO)
    sv, sm = torch.empty_like(rv), torch.empty_like(rm)
    g.gqt_sigma_vac(rv, dts, sv)
    g.gqt_sigma_msd(rm, dts, sm)
    torch.cuda.synchronize()
    t2 = time.perf_counter()
    rd, rv, sv, sm = rd.cpu().numpy()[0], rv.cpu().numpy(), sv.cpu().numpy(), sm.cpu().numpy()
    e0 = 300
    sc = A.semiclassical(rd, rv, sv)
    # sigma_VAC at t_19 = 3.8 against sigma_MSD at the step midpoint 3.9 (Fig. 1d: equivalent)
    out["example1_square2000"] = {"build_s": t1 - t0, "compute_s": t2 - t1, "sigma_vac_E0_t3.8": float(sv[-1, e0]),
                                  "sigma_msd_E0_t3.9": float(sm[-1, e0]), "sigma_sc_E0": float(sc["sigma_sc"][e0]),
                                  "tau_E0": float(sc["tau"][e0]), "mfp_E0": float(sc["mfp"][e0]),
                                  "dos_E0": float(rd[e0])}
    del ham, phi, a, b, p, px
    torch.cuda.empty_cache()
    # Example 2 (localized, Fig. 2)
    t0 = time.perf_counter()
    ham = g.gqt_build_hamiltonian(None, 4.1, g.GQT_FP64, kind=g.GQT_LATTICE_CHAIN, L1=4_000_000, t=-1.0, W=4.0,
                                  seed=S.BASE_SEED + 11)
    nO = ham.n / ham.volume
    R = 2
    phi = torch.empty((ham.n, R), dtype=torch.complex128, device="cuda")
    g.gqt_random_phase(ham, S.BASE_SEED + 11, R, phi)
    torch.cuda.synchronize()
    t1 = time.perf_counter()
    M = 500
    dts = np.concatenate([np.arange(1, 11) * 0.1, np.arange(1, 11) * 1.0, np.arange(1, 11) * 10.0])
    Nt = dts.size
    E = torch.arange(-200, 201, dtype=torch.float64, device="cuda") * 0.02
    dos = torch.empty((1, R, M), dtype=torch.float64, device="cuda")
    g.gqt_dos_moments(ham, phi, R, M, dos)
    p, px = torch.empty_like(phi), torch.empty_like(phi)
    g.gqt_msd_init(ham, phi, p, px, R)
    msd = torch.empty((Nt, 1, R, M), dtype=torch.float64, device="cuda")
    g.gqt_msd_moments(ham, p, px, R, dts, M, msd)
    rd = recon(dos[0].mean(0, keepdim=True), E, 4.1, nO)
    rm = recon(msd[:, 0].mean(1), E, 4.1, nO)
    sm = torch.empty_like(rm)
    g.gqt_sigma_msd(rm, dts, sm)
    torch.cuda.synchronize()
    t2 = time.perf_counter()
    rd, rm, sm = rd.cpu().numpy()[0], rm.cpu().numpy(), sm.cpu().numpy()
    e0 = 200
    Lp = A.propagation_length(rd, rm)
    Lmid = 0.5 * (Lp[1:, e0] + Lp[:-1, e0])
    out["example2_chain4M"] = {"build_s": t1 - t0, "compute_s": t2 - t1, "xi_saturation_E0": float(A.xi_saturation(Lp)[e0]),
                               "xi_fit_E0": A.xi_fit(Lmid, sm[1:, e0]), "L_final_E0": float(Lp[-1, e0]),
                               "max_bessel_orders": int(g.gqt_np_rule(4.1 * 100.0, 4096))}
    out["total_compute_s"] = out["example1_square2000"]["compute_s"] + out["example2_chain4M"]["compute_s"]
    out["paper_k40_s_context"] = 180.0
    return out


def run_ours(args):
    import torch
    import paper_1705_01387_gb300 as g
    from paper_1705_01387_gb300.replicas import max_over_ranks, shard_vectors

    ws, rank, local = _dist()
    torch.cuda.set_device(local)
    if ws > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    w, lat = workload(args.small, args.cells, args.moments)
    dE = w.energy_scale
    ham = g.gqt_build_hamiltonian(lat, dE, g.GQT_FP64)
    g.gqt_set_fp64_arith(ham, args.fp64_arith)
    if args.small:  # the reduced lattice stands in for the large one: its kernels, not the on-chip rows
        g.gqt_set_cluster(ham, False)
    g.gqt_set_temporal_blocking(ham, args.temporal_blocking)
    N, M, R = lat.n, w.M, 1
    Np = g.gqt_np_rule(dE * w.dt, 64)
    del lat
    cd = torch.complex128
    phi = torch.empty((N, R), dtype=cd, device="cuda")
    first, _ = shard_vectors(ws * R, ws, rank)  # one independent random vector per rank
    g.gqt_random_phase(ham, w.seed, R, phi, first_vector=first)
    a, b, p, px = (torch.empty_like(phi) for _ in range(4))
    g.gqt_vac_init(ham, phi, a, b, R)
    g.gqt_msd_init(ham, phi, p, px, R)
    E = torch.from_numpy(w.energies).cuda()
    nO = N / ham.volume
    rows = torch.empty((2, M), dtype=torch.float64, device="cuda")
    recon = torch.empty((2, E.numel()), dtype=torch.float64, device="cuda")
    dts = np.array([w.dt])

    def step():
        g.gqt_vac_moments(ham, a, b, R, dts, M, rows[0], Np=[Np])
        g.gqt_msd_moments(ham, p, px, R, dts, M, rows[1], Np=[Np])
        g.gqt_kpm_reconstruct(rows, E, dE, nO, recon)

    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize()
    if ws > 1:
        torch.distributed.barrier()
    launches0 = g.gqt_launch_count()
    st = torch.cuda.current_stream()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with Clocks(local) as clk:
        torch.cuda.synchronize()
        g.gqt_profile_start()
        torch.cuda.nvtx.range_push("timed")  # lets ncu select exactly these launches (--nvtx-include timed/)
        e0.record(st)
        for _ in range(args.steps):
            step()
        e1.record(st)
        torch.cuda.nvtx.range_pop()
        torch.cuda.synchronize()
        prof_ms, prof_n = g.gqt_profile_stop(12)
    launches = g.gqt_launch_count() - launches0
    t_ms = e0.elapsed_time(e1)
    if ws > 1:
        t_ms = max_over_ranks(t_ms, device="cuda")
    units = float(N) * 2 * M * args.steps * ws
    value = units / (t_ms * 1e-3)

    # end to end through the C ABI with host buffers: every step hands the library
    # the four state vectors in pinned host memory; gqt_vac_moments and
    # gqt_msd_moments copy them to the device and back inside the call, and the
    # reconstructed rows (the step's result) come back to the host.
    hs = [torch.empty((N, R), dtype=cd, pin_memory=True) for _ in range(4 if not args.no_e2e else 0)]
    for h_, d_ in zip(hs, (a, b, p, px)):
        h_.copy_(d_)
    hrec = torch.empty((2, E.numel()), dtype=torch.float64, pin_memory=True)

    def e2e_step():
        g.gqt_vac_moments(ham, hs[0], hs[1], R, dts, M, rows[0], Np=[Np])
        g.gqt_msd_moments(ham, hs[2], hs[3], R, dts, M, rows[1], Np=[Np])
        g.gqt_kpm_reconstruct(rows, E, dE, nO, recon)
        hrec.copy_(recon)
        torch.cuda.synchronize()

    # warm-up as for the device-resident leg: the first host-buffer call stages the
    # vectors into the handle's own buffers and captures the graphs for them
    for _ in range(args.warmup if not args.no_e2e else 0):
        e2e_step()
    t0 = time.perf_counter()
    for _ in range(args.steps if not args.no_e2e else 0):
        e2e_step()
    t_e2e = max(time.perf_counter() - t0, 1e-9)
    vb = N * R * 16
    e2e = None if args.no_e2e else {"value": units / t_e2e, "unit": UNIT, "h2d_bytes_per_step": 4 * vb,
                                    "d2h_bytes_per_step": 4 * vb + hrec.numel() * 8,
                                    "path": "gqt_vac_moments + gqt_msd_moments on host state vectors (copied in "
                                            "and out inside the calls) + gqt_kpm_reconstruct, result read back"}

    # roofline of the dominant kernel family (largest share of the timed kernel time):
    # family 1 = VAC orders Re <l|T_m|r> by one recurrence (k_cheb_re), 5 = MSD orders
    # with l = r, two moments per step (k_cheb_dbl, no l read), 6 = VAC orders by two
    # recurrences, two moments per step (k_cheb_pair).  With paired-FP32 arithmetic
    # (mode 1) families 5 and 6 run k_cheb_dbl_df and k_cheb_pair_df, and on the
    # honeycomb layout the temporally blocked k_cheb2_honey_df runs two steps per
    # launch (10 = VAC rows, 11 = l = r rows).
    hbm, peak_kind = _peaks()
    df = args.fp64_arith == 1
    sfx = "_df" if df else ""
    uniform = bool(ham.forms & g.GQT_FORM_UNIFORM_HOP)
    # the single-order kernels read a row's class (2 bytes) instead of its indices and, in
    # paired arithmetic with one common hopping, no hoppings
    row = 0 if R > 1 else 2 - 3 * 4 - (3 * 8 if df and uniform else 0)
    fam = {1: ("k_cheb_re (VAC row: fused SpMV + three-term recurrence + Re <l|T_m|r>)",
               bytes_per_orbital_cheb(3, True, ham.hop_real, R) + row, "re", 1),
           5: (f"k_cheb_dbl{sfx} (MSD row: fused SpMV + recurrence + <u_n|u_n>, <u_n+1|u_n>)",
               bytes_per_orbital_cheb(3, True, ham.hop_real, R) - 16 * R + row, "dbl", 1),
           6: (f"k_cheb_pair{sfx} (VAC row: two fused SpMV + recurrences, T_k l and T_k r, + Re <A_k|B_k>, "
               "Re <A_k|B_k+1>)", bytes_per_orbital_pair(3, ham.hop_real, R) + row, "pair", 1),
           10: ("k_cheb2_honey_df_pair (VAC row, temporally blocked: two steps of both recurrences per launch, "
                "the second from the first's rows in shared memory" + (", one common hopping" if uniform else "") + ")",
                bytes_per_orbital_tiled(3, ham.hop_real, True, uniform), "pair", 2),
           11: ("k_cheb2_honey_df_dbl (MSD row, temporally blocked: two steps per launch"
                + (", one common hopping" if uniform else "") + ")",
                bytes_per_orbital_tiled(3, ham.hop_real, False, uniform), "dbl", 2)}
    total_prof = float(np.sum(prof_ms))
    dom = max(fam, key=lambda k: prof_ms[k])
    fams = {}
    for k, (name, bpo_k, _, _) in fam.items():
        nl = int(prof_n[k])
        avg = prof_ms[k] * 1e-3 / max(nl, 1)
        fams[name.split()[0]] = {"launches": nl, "avg_launch_us": avg * 1e6, "bytes_per_orbital": bpo_k,
                                 "achieved_gbs": N * bpo_k / avg / 1e9 if nl else None,
                                 "share_of_timed_kernels": prof_ms[k] / max(total_prof, 1e-12)}
    kname, bpo, fkind, nsteps = fam[dom]
    traffic = measured_traffic(kname.split()[0] + ("_uh" if uniform and nsteps == 2 else ""), N)
    n_launch = int(prof_n[dom])
    avg_s = prof_ms[dom] * 1e-3 / max(n_launch, 1)
    achieved = N * bpo / avg_s / 1e9
    hbm_frac = achieved / hbm
    clocks = clk.summary()
    hbm_obj = {"bound": "hbm", "achieved": achieved, "peak": hbm, "unit": "GB/s", "frac": hbm_frac,
               "traffic": traffic, "traffic_source": "profiles/traffic_moment_kernels.json (ncu at N = 4.2M, "
                                                     "scaled by N)",
               "kernel": kname, "bytes_per_orbital": bpo, "peak_source": peak_kind + " (MEASURED_PEAKS.json hbm_gbs)"}
    if df:
        # arithmetic roofline of the paired-FP32 kernel: FP32-pipe instructions per
        # orbital against SMs x 128 lanes x the SM clock sampled during the timed region
        ops = df_fp32_ops_per_orbital(3, ham.hop_real, fkind, uniform and nsteps == 2) * R * nsteps
        sms = torch.cuda.get_device_properties(local).multi_processor_count
        mhz = float(clocks.get("sm_mhz") or clocks.get("sm_max_mhz") or 2070.0)
        fp32_peak = sms * 128 * mhz * 1e6 / 1e9
        fp32_achieved = ops * N / avg_s / 1e9
        alu = {"achieved": fp32_achieved, "peak": fp32_peak, "unit": "G FP32-pipe instr/s",
               "frac": fp32_achieved / fp32_peak, "fp32_instr_per_orbital": ops,
               "peak_source": f"{sms} SMs x 128 FP32 lanes x {mhz:.0f} MHz (median SM clock under load)"}
        roof = dict(hbm_obj, fp32_pipe=alu) if hbm_frac >= alu["frac"] else \
            {"bound": "alu", **{k: alu[k] for k in ("achieved", "peak", "unit", "frac")}, "traffic": traffic,
             "kernel": kname, "hbm": {k: hbm_obj[k] for k in ("achieved", "peak", "unit", "frac")}}
        if nsteps == 2:
            # the two single-step launches this one replaces would move these bytes
            eq = 2 * (bytes_per_orbital_pair(3, ham.hop_real, R) if fkind == "pair"
                      else bytes_per_orbital_cheb(3, True, ham.hop_real, R) - 16 * R) + 2 * row
            roof["steps_per_launch"] = 2
            roof["single_step_equivalent"] = {"bytes_per_orbital": eq, "achieved": N * eq / avg_s / 1e9,
                                              "frac": N * eq / avg_s / 1e9 / hbm, "unit": "GB/s"}
    else:
        # FP64 arithmetic roofline of the same kernel against the measured FMA peak
        fp64_peak = g.gqt_probe_fp64()
        fma = fp64_fma_per_orbital(3, ham.hop_real, fkind) * R * nsteps
        fp64_achieved = 2.0 * fma * N / avg_s / 1e9
        alu_frac = fp64_achieved / fp64_peak
        roof = ({"bound": "alu", "achieved": fp64_achieved, "peak": fp64_peak, "unit": "GFLOP/s (FP64)",
                 "frac": alu_frac, "traffic": traffic, "kernel": kname, "fp64_fma_per_orbital": fma,
                 "peak_source": "measured FP64 FMA probe (gqt_probe_fp64)",
                 "hbm": {"achieved": achieved, "peak": hbm, "unit": "GB/s", "frac": hbm_frac,
                         "bytes_per_orbital": bpo}}
                if alu_frac > hbm_frac else
                dict(hbm_obj, fp64={"achieved": fp64_achieved, "peak": fp64_peak, "unit": "GFLOP/s",
                                    "frac": alu_frac, "fp64_fma_per_orbital": fma}))
    out = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": t_ms / args.steps, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f32x2" if df else "f64",
        "data": "synthetic (seeded Anderson honeycomb lattice and random-phase vectors)",
        "config": {"workload": w.name if not args.small else w.name + "_small", "n_orbitals": N, "moments": M,
                   "vectors_per_gpu": R, "bessel_orders": Np, "dt_hbar_per_eV": w.dt, "energies": int(E.numel()),
                   "step": "one VAC + MSD time step (2M moments, 2 evolutions) + KPM reconstruction",
                   "temporal_blocking": bool(args.temporal_blocking),
                   "hop_storage": ("real FP64" if ham.hop_real else "complex FP64")
                   + ("; one common hopping (blocked rows read no hop array)" if uniform else ""),
                   "arith": ("moment rows on pairs of FP32 numbers (double-float, ~48-bit significands; FP64 "
                             "storage, results within 1e-12 of the FP64 mode), evolution in FP64")
                   if df else "FP64 fused multiply-adds",
                   "l2": "inputs larger than L2 (H~ ELL %.2f GB + state vectors)" % (N * (3 * 12 + 8 + 24) / 1e9),
                   "parallelism": f"replicas x{ws} (independent random vectors)"},
        "gpu_launches": int(launches),
        "roofline": roof,
        "kernels": {"dominant": kname, "avg_launch_us": avg_s * 1e6, "launches": n_launch,
                    "share_of_timed_kernels": prof_ms[dom] / max(total_prof, 1e-12), "families": fams},
        "e2e": e2e,
        "clocks": clocks,
    }
    if rank == 0 and not args.no_fp32:
        out["fp32_batched"] = fp32_batched(args, g, torch)
    if rank == 0 and not args.no_cpu_baseline:
        out["cpu_baseline"] = cpu_baseline(args.small, budget_s=args.cpu_seconds)
    if rank == 0:
        print(json.dumps(out))
    if ws > 1:
        torch.distributed.destroy_process_group()


def _oracle_sample(small: bool):
    import oracle as O
    w, lat = workload(small)
    h = O.Hamiltonian(lat, w.energy_scale)
    phi = S.random_phase(lat.n, 1, seed=w.seed)[:, 0]
    return w, lat, h, phi


def hall(args, g, torch):
    """Hall conductivity (Kubo-Bastin; the paper's Sec. 6 outlook) of the
    disordered Haldane model: honeycomb 512 x 512 cells (N = 524,288), t1 = -1,
    t2 = 0.15, phi = pi/2, Anderson W = 1, one random-phase vector, M = 1024
    Kubo-Bastin moments, sigma_xy on 2001 energies.  Times gqt_kb_moments (the
    two chains plus the M x M complex contraction) in three forms -- FP32 storage
    with the split-TF32 tensor-core contraction, FP64 chains with it, and FP64
    throughout -- and gqt_kubo_bastin, with CUDA events; per-kernel times from the
    library's profiler (families 7-9)."""
    L = args.hall_L or (32 if args.small else 512)
    M = args.hall_moments or (128 if args.small else 1024)
    seed = 1705013875
    lat = S.haldane(L, L, -1.0, 0.15, math.pi / 2, 0.0, 1.0, seed=seed)
    dE = 1.05 * (3 + 6 * 0.15 + 0.5)
    ham = g.gqt_build_hamiltonian(lat, dE)
    r = torch.from_numpy(S.random_phase(lat.n, 1, seed=seed)).cuda()
    E = torch.linspace(-0.97 * dE, 0.97 * dE, 2001, dtype=torch.float64, device="cuda")
    n = lat.n
    fp64_peak = g.gqt_probe_fp64()
    with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
        bf16 = float(json.load(f)["bf16_tflops"])
    tf32_peak = bf16 * 1.1 / 2.25  # nominal dense TF32 : BF16 ratio of the part
    steps = max(1, args.steps)
    out = {"workload": f"haldane{L}x{L}_W1_M{M}", "n_orbitals": n, "moments": M, "vectors": 1,
           "metric": "Kubo-Bastin orbital-moment pairs/s (N R M^2 / time of gqt_kb_moments)",
           "energies": int(E.numel()), "modes": {}}
    sigmas = {}
    ham32 = g.gqt_build_hamiltonian(lat, dE, g.GQT_FP32_ACC64)
    r32 = r.to(torch.complex64)
    for mode, name in ((2, "fp32_chains_tensor_core"), (1, "tensor_core_split_tf32"), (0, "fp64")):
        if mode == 0 and args.hall_skip_fp64:
            continue
        h_, r_ = (ham32, r32) if mode == 2 else (ham, r)
        g.gqt_set_kb_contraction(h_, min(mode, 1))
        lam = torch.empty((M, M), dtype=torch.complex128, device="cuda")
        sig = torch.empty_like(E)
        for _ in range(max(1, args.warmup)):
            g.gqt_kb_moments(h_, r_, 1, M, 0, 1, lam)
            g.gqt_kubo_bastin(lam, E, dE, lat.volume, sig)
        torch.cuda.synchronize()
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(3)]
        g.gqt_profile_start()
        ev[0].record()
        for _ in range(steps):
            g.gqt_kb_moments(h_, r_, 1, M, 0, 1, lam)
        ev[1].record()
        for _ in range(steps):
            g.gqt_kubo_bastin(lam, E, dE, lat.volume, sig)
        ev[2].record()
        torch.cuda.synchronize()
        prof_ms, prof_n = g.gqt_profile_stop(10)
        t_mom = ev[0].elapsed_time(ev[1]) * 1e-3 / steps
        t_kb = ev[1].elapsed_time(ev[2]) * 1e-3 / steps
        gemm_s = prof_ms[8] * 1e-3 / max(int(prof_n[8]), 1)
        if mode == 0:
            macs = 28.0 * 4 * M * M * n  # 28 digit products per real product
            roof = {"kernel": "k_slice_gemm (FP64 contraction by exact 8-bit slices, TMA-fed tcgen05 kind::f16, slicing included)",
                    "bound": "tensor", "achieved": 2 * macs / gemm_s / 1e12, "peak": bf16,
                    "unit": "TFLOP/s (FP16)", "frac": 2 * macs / gemm_s / 1e12 / bf16,
                    "peak_source": "measured BF16 GEMM (MEASURED_PEAKS.json bf16_tflops)",
                    "method_flops": {"achieved": 8.0 * M * M * n / gemm_s / 1e9, "unit": "GFLOP/s (FP64)",
                                     "vs_fp64_pipe": 8.0 * M * M * n / gemm_s / 1e9 / fp64_peak}}
        else:
            macs = 3.0 * 2 * M * M * (2.0 * n)  # three split products, Re and Im, 2N real terms
            roof = {"kernel": "k_kb_gemm_tma (TMA-fed tcgen05 kind::tf32, 128 x 256 tiles, three split products)",
                    "bound": "tensor",
                    "achieved": 2 * macs / gemm_s / 1e12, "peak": tf32_peak, "unit": "TFLOP/s (TF32)",
                    "frac": 2 * macs / gemm_s / 1e12 / tf32_peak,
                    "peak_source": "measured BF16 GEMM (MEASURED_PEAKS.json bf16_tflops) x nominal TF32/BF16 1.1/2.25",
                    # the complex contraction's own work, 8 N M^2 real flops, each
                    # product counted once rather than as its three split products
                    "method_flops": {"achieved": 8.0 * M * M * n / gemm_s / 1e12,
                                     "frac": 8.0 * M * M * n / gemm_s / 1e12 / tf32_peak, "unit": "TFLOP/s"}}
        s_np = sig.cpu().numpy()
        sigmas[mode] = s_np
        e_np = E.cpu().numpy()
        i0 = int(np.argmin(np.abs(e_np)))
        out["modes"][name] = {
            "value": n * M * M / t_mom, "kb_moments_s": t_mom, "kubo_bastin_s": t_kb,
            "kernels": {"k_kb_step_ms_per_launch": prof_ms[7] / max(int(prof_n[7]), 1),
                        "k_kb_step_launches": int(prof_n[7]) // steps, "contraction_ms": gemm_s * 1e3,
                        "k_kb_series_ms": prof_ms[9] / max(int(prof_n[9]), 1)},
            "roofline": roof, "sigma_xy_gap_centre_e2_over_h": float(s_np[i0])}
    if 0 in sigmas:
        for mode, key in ((1, "tensor_core_split_tf32"), (2, "fp32_chains_tensor_core")):
            if mode in sigmas:
                out["modes"][key]["sigma_xy_max_abs_diff_vs_fp64"] = float(np.max(np.abs(sigmas[mode] - sigmas[0])))
    first = out["modes"]["fp32_chains_tensor_core"]
    out["value"] = first["value"]
    if not args.no_cpu_baseline:
        import oracle as O  # the CPU baseline leg only
        h = O.Hamiltonian(lat, dE)
        Mc = 24
        t0 = time.perf_counter()
        h.kb_moments(lat.dx, lat.dy, r.cpu().numpy(), Mc)
        dt = time.perf_counter() - t0
        out["cpu_baseline"] = {"value": n * Mc * Mc / dt, "unit": "orbital-moment pairs/s", "cores": 1,
                               "kind": "oracle", "sample": f"oracle Kubo-Bastin moments, M = {Mc} at full N = {n} "
                                                           f"(serial FP64 C++, {dt:.1f} s)"}
    return out


def cpu_baseline(small: bool, budget_s: float = 15.0, prepared=None):
    """Serial FP64 oracle on one host core: Chebyshev moments at full N, as many
    as fit in about budget_s seconds, scaled to orbital-moments/s."""
    w, lat, h, phi = prepared or _oracle_sample(small)
    t0 = time.perf_counter()
    h.cheb_moments(phi, phi, 2)
    t1 = time.perf_counter()
    per = max(t1 - t0, 1e-6)
    m = int(max(3, min(400, budget_s / per)))
    t0 = time.perf_counter()
    h.cheb_moments(phi, phi, m)
    dt = time.perf_counter() - t0
    return {"value": lat.n * m / dt, "unit": UNIT, "cores": 1, "kind": "oracle",
            "sample": f"{m} Chebyshev moments <phi|T_m(H~)|phi> of the same lattice at full N = {lat.n} "
                      f"(serial FP64 C++, {dt:.1f} s)"}


def run_reference(args):
    ws, rank, _ = _dist()
    if rank != 0:
        return
    prepared = _oracle_sample(args.small)
    w, lat = prepared[0], prepared[1]
    per_step = max(1.0, min(20.0, 150.0 / max(args.steps + args.warmup, 1)))
    for _ in range(args.warmup):
        cpu_baseline(args.small, per_step, prepared)
    vals = []
    t0 = time.perf_counter()
    for _ in range(args.steps):
        vals.append(cpu_baseline(args.small, per_step, prepared))
    elapsed = time.perf_counter() - t0
    value = statistics.mean(v["value"] for v in vals)
    out = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps,
           "warmup": args.warmup, "ms_per_step": elapsed * 1e3 / max(args.steps, 1), "higher_is_better": True,
           "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
           "config": {"workload": w.name if not args.small else w.name + "_small", "n_orbitals": lat.n,
                      "moments": w.M, "step": "bounded sample: serial oracle Chebyshev moments at full N"},
           "cpu_baseline": {"value": value, "unit": UNIT, "cores": 1, "kind": "oracle", "sample": vals[-1]["sample"]},
           "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
           "gpu_launches": 0}
    print(json.dumps(out))


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--small", action="store_true", help="reduced lattice, for tests")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--cpu-seconds", type=float, default=15.0)
    ap.add_argument("--cells", default=None, help="L1xL2 honeycomb cells (profiling captures only)")
    ap.add_argument("--moments", type=int, default=None, help="moments per row (profiling captures only)")
    ap.add_argument("--no-e2e", action="store_true", help="skip the host-buffer end-to-end pass")
    ap.add_argument("--temporal-blocking", type=int, default=1, choices=(0, 1),
                    help="two Chebyshev steps per launch on the honeycomb layout (gqt_set_temporal_blocking)")
    ap.add_argument("--no-fp32", action="store_true", help="skip the batched FP32 vs FP64 comparison")
    ap.add_argument("--no-ragged", action="store_true", help="skip the ragged-batch measurement")
    ap.add_argument("--fp32-moments", type=int, default=2048, help="moments of the FP32/FP64 comparison")
    ap.add_argument("--fp32-L", type=int, default=0, help="cubic L of the FP32 comparison (profiling captures only)")
    ap.add_argument("--only-fp32", action="store_true", help="run only the FP32/FP64 comparison (profiling)")
    ap.add_argument("--precision", action="store_true", help="FP32 vs FP64 per-result error table (C4 workload)")
    ap.add_argument("--latency", action="store_true", help="latency-bound workloads (C1 graphs on/off, C5 gradient)")
    ap.add_argument("--paper-examples", action="store_true", help="the paper's two examples (Sec. 5), timed")
    ap.add_argument("--precision-steps", type=int, default=200, help="VAC time steps of the error table")
    ap.add_argument("--precision-msd-steps", type=int, default=3, help="MSD time steps of the error table")
    ap.add_argument("--precision-ref-vectors", type=int, default=2, help="FP64 reference vectors of the error table")
    ap.add_argument("--precision-L", type=int, default=0, help="honeycomb cells per side of the error table (profiling)")
    ap.add_argument("--precision-moments", type=int, default=0, help="moments of the error table (profiling)")
    ap.add_argument("--hall", action="store_true", help="Hall conductivity (Kubo-Bastin) of the Haldane model")
    ap.add_argument("--hall-L", type=int, default=0, help="Haldane cells per side of the Hall run (profiling)")
    ap.add_argument("--hall-moments", type=int, default=0, help="Kubo-Bastin moments of the Hall run (profiling)")
    ap.add_argument("--hall-skip-fp64", action="store_true", help="time only the tensor-core contraction (profiling)")
    ap.add_argument("--fp64-arith", type=int, default=1, choices=[0, 1],
                    help="moment rows of the FP64 workload: 1 = pairs of FP32 numbers (default), 0 = FP64 FMAs")
    args = ap.parse_args()
    if args.impl == "reference":
        run_reference(args)
    elif args.hall:
        import torch
        import paper_1705_01387_gb300 as g
        print(json.dumps(hall(args, g, torch)))
    elif args.paper_examples:
        import torch
        import paper_1705_01387_gb300 as g
        print(json.dumps(paper_examples(args, g, torch)))
    elif args.latency:
        import torch
        import paper_1705_01387_gb300 as g
        print(json.dumps(latency(args, g, torch)))
    elif args.precision:
        import torch
        import paper_1705_01387_gb300 as g
        print(json.dumps(precision_table(args, g, torch)))
    elif args.only_fp32:
        import torch
        import paper_1705_01387_gb300 as g
        print(json.dumps(fp32_batched(args, g, torch)))
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
