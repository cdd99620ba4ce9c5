"""Performance cases of the library: what a transport calculation asks of it.

A case is one call sequence a program makes: moment rows of the density of states
(gqt_dos_moments), velocity-autocorrelation and mean-square-displacement rows with
their time evolution (gqt_vac_moments, gqt_msd_moments), the gradient of a
conductivity loss (gqt_vac_loss_grad), the Hall conductivity (gqt_kb_moments and
gqt_kubo_bastin) and the reconstruction of spectra from stored rows
(gqt_kpm_reconstruct, gqt_sigma_vac).  Lattices, disorder strengths, time steps and
moment counts are those of the library's workloads and of the method paper's two
examples, with fewer moments or time steps where a full run takes minutes: the work
of an order and of a time step is the same in each of them.

`exact` computes the same quantities by the plain recursions (Eqs. 17-31 of
arXiv:1705.01387) in 64 bits with torch.
"""
from __future__ import annotations

import math
import types

import numpy as np
import torch

import paper_1705_01387_gb300 as g

DEV = "cuda"
SQ3 = math.sqrt(3.0)
KINDS = {"chain": g.GQT_LATTICE_CHAIN, "square": g.GQT_LATTICE_SQUARE, "honeycomb": g.GQT_LATTICE_HONEYCOMB,
         "cubic": g.GQT_LATTICE_CUBIC}
SLOTS = {"chain": 2, "square": 4, "honeycomb": 3, "cubic": 6, "haldane": 9}
HOPPING = {"chain": -1.0, "square": -1.0, "honeycomb": -2.7, "cubic": -1.0, "haldane": -1.0}


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # the latency end: one random vector on 32 x 32 graphene cells, the size
        # of a check against diagonalisation
        dict(name="dos_small", op="dos", lattice="honeycomb", L1=32, L2=32, W=1.0, vacancies=0.0, field=0, fp32=False,
             R=1, M=512),
        # the Anderson model at its critical disorder with 32 random vectors in one
        # batch, FP32 storage: the high-throughput density of states
        dict(name="dos_cubic_batch", op="dos", lattice="cubic", L1=128, L2=1, W=16.5, vacancies=0.0, field=0,
             fp32=True, R=32, M=128),
        # disorder realisations of uneven size in one handle (finite-size scaling)
        dict(name="dos_ragged", op="ragged", count=16, Lmin=32, Lmax=64, W=16.5, fp32=True, R=1, M=512),
        # a whole time-resolved VAC calculation on the small system
        dict(name="vac_small", op="vac", lattice="honeycomb", L1=32, L2=32, W=1.0, vacancies=0.0, field=0, fp32=False,
             R=1, M=512, steps=10, dt=1.0),
        # one time step of the production calculation: 16.8 million orbitals
        dict(name="vac_large", op="vac", lattice="honeycomb", L1=4096, L2=2048, W=2.0, vacancies=0.0, field=0,
             fp32=False, R=1, M=500, steps=1, dt=2.0),
        # graphene with 1% vacancies, 8 random vectors, FP32 storage
        dict(name="vac_vacancy_batch", op="vac", lattice="honeycomb", L1=1024, L2=1024, W=0.5, vacancies=0.01,
             field=0, fp32=True, R=8, M=400, steps=1, dt=2.0),
        # one MSD time step of a production run at a quarter of the size
        dict(name="msd_honeycomb", op="msd", lattice="honeycomb", L1=2048, L2=1024, W=2.0, vacancies=0.0, field=0,
             fp32=False, R=1, M=1000, steps=1, dt=2.0),
        # the paper's diffusive example, a square lattice (a side that is no power
        # of two, as given by the user's input files)
        dict(name="msd_square", op="msd", lattice="square", L1=1001, L2=999, W=4.0, vacancies=0.0, field=0, fp32=False,
             R=1, M=600, steps=2, dt=0.4),
        # gradient of a conductivity loss for every site and bond
        dict(name="grad", op="grad", lattice="honeycomb", L1=256, L2=256, W=2.0, vacancies=0.0, field=0, fp32=False,
             M=1024, rows=3, dt=2.0),
        # Hall conductivity of a Chern insulator in FP64 (the default mode)
        dict(name="hall", op="hall", L1=96, L2=96, W=1.0, fp32=False, R=1, M=256, NE=1001),
        # the same with FP32 storage and the tensor-core contraction, larger
        dict(name="hall_fp32", op="hall", L1=256, L2=256, W=1.0, fp32=True, R=1, M=500, NE=2001),
        # spectra of a finished VAC run of 100 time steps
        dict(name="spectra", op="kpm", rows=100, M=3000, NE=1001),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["dos", "dos", "vac", "vac", "msd", "msd", "ragged", "grad", "hall", "hall", "kpm"])
    if op == "kpm":
        return dict(op=op, rows=_log_int(rng, 1, 200), M=_log_int(rng, 128, 3000), NE=_log_int(rng, 101, 1501))
    if op == "ragged":
        lo = rng.randint(12, 40)
        return dict(op=op, count=rng.randint(3, 24), Lmin=lo, Lmax=lo + rng.randint(0, 20), W=16.5, fp32=True,
                    R=rng.choice([1, 1, 2, 4]), M=_log_int(rng, 64, 512))
    if op == "hall":
        fp32 = rng.random() < 0.5
        top = 256 if fp32 else 96
        M = _log_int(rng, 48, 500 if fp32 else 256)
        return dict(op=op, L1=_log_int(rng, 16, top), L2=_log_int(rng, 16, top), W=1.0, fp32=fp32,
                    R=rng.choice([1, 1, 1, 2]) if M <= 200 else 1, M=M, NE=_log_int(rng, 201, 2001))
    if op == "grad":
        side = _log_int(rng, 24, 256)
        return dict(op=op, lattice=rng.choice(["honeycomb", "honeycomb", "square"]), L1=side, L2=_log_int(rng, 24, 256),
                    W=2.0, vacancies=0.0, field=0, fp32=rng.random() < 0.25, M=_log_int(rng, 64, 1024),
                    rows=rng.randint(1, 3), dt=2.0)
    lattice = rng.choice(["honeycomb", "honeycomb", "honeycomb", "square", "cubic", "chain"])
    fp32 = rng.random() < 0.4
    R = rng.choice([1, 2, 4, 8, 16, 32]) if fp32 else rng.choice([1, 1, 1, 1, 2])
    n = _log_int(rng, 1500, 4000000 // max(1, R // 2))  # sites
    if lattice == "honeycomb":
        L1 = _log_int(rng, 16, max(17, n // 64))
        if rng.random() < 0.6:  # sides as users choose them: mostly round
            L1 = max(32, L1 // 32 * 32)
        dims = (L1, max(3, n // (2 * L1)))
    elif lattice == "square":
        L1 = max(3, int(math.sqrt(n) * rng.uniform(0.5, 2.0)))
        dims = (L1, max(3, n // L1))
    elif lattice == "cubic":
        dims = (rng.choice([64, max(8, int(round(n ** (1 / 3))))]) if n > 200000 else max(8, int(round(n ** (1 / 3)))), 1)
    else:
        dims = (n, 1)
    case = dict(op=op, lattice=lattice, L1=dims[0], L2=dims[1], W=rng.choice([0.5, 1.0, 2.0, 4.0]),
                vacancies=rng.choice([0.0, 0.0, 0.01]),
                field=rng.choice([0, 0, 0, 3]) if lattice in ("honeycomb", "square") and n <= 500000 else 0,
                fp32=fp32, R=R)
    sites = _sites(case)
    steps = 1 if op == "dos" else rng.choice([1, 1, 2, 3])
    M = _log_int(rng, 60, 800)
    case["M"] = max(32, min(M, int(2.5e9 / (sites * R * steps))))
    if op != "dos":
        case.update(steps=steps, dt=rng.choice([0.2, 1.0, 2.0]))
    return case


# ------------------------------------------------------------------ models

def _sites(case):
    L1, L2 = case["L1"], case["L2"]
    return {"chain": L1, "square": L1 * L2, "cubic": L1 ** 3}.get(case.get("lattice"), 2 * L1 * L2)


def _scale(case):
    """Energy scale: 1.05 x the Gershgorin bound of the Anderson model."""
    lat = case.get("lattice", "haldane" if case["op"] == "hall" else "cubic")
    if lat == "haldane":
        return 1.05 * (3.0 + 6 * 0.15 + case["W"] / 2)
    return 1.05 * (SLOTS[lat] * abs(HOPPING[lat]) + case["W"] / 2)


def _key(seed, stream):
    m = (1 << 64) - 1
    z = (seed + (stream + 1) * 0x9E3779B97F4A7C15) & m
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & m
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & m
    return z ^ (z >> 31)


def _signed(v):
    return v - (1 << 64) if v >= 1 << 63 else v


def _draws(seed, stream, n):
    """Draws 0 .. n-1 of a SplitMix64 stream, as int64 bit patterns."""
    i = torch.arange(1, n + 1, dtype=torch.int64, device=DEV)
    z = i * _signed(0x9E3779B97F4A7C15) + _signed(_key(seed, stream))
    z = (z ^ ((z >> 30) & ((1 << 34) - 1))) * _signed(0xBF58476D1CE4E5B9)
    z = (z ^ ((z >> 27) & ((1 << 37) - 1))) * _signed(0x94D049BB133111EB)
    return z ^ ((z >> 31) & ((1 << 33) - 1))


def _uniform(seed, stream, n):
    return ((_draws(seed, stream, n) >> 11) & ((1 << 53) - 1)).double() * 2.0 ** -53


def _geometry(lattice, L1, L2):
    """Neighbours [n, K], bond displacements dx, dy [n, K], row coordinate y [n], length, volume."""
    if lattice in ("honeycomb", "haldane"):
        nc = L1 * L2
        c = torch.arange(nc, device=DEV)
        c1, c2 = c % L1, c // L1

        def cell(a, b):
            return a % L1 + L1 * (b % L2)

        K = SLOTS[lattice]
        idx = torch.empty((nc, 2, K), dtype=torch.int64, device=DEV)
        dx = torch.empty((nc, 2, K), dtype=torch.float64, device=DEV)
        dy = torch.empty_like(dx)
        near = [(0, 0, 0.0, 1.0), (1, -1, SQ3 / 2, -0.5), (0, -1, -SQ3 / 2, -0.5)]
        for k, (a, b, x, y) in enumerate(near):
            idx[:, 0, k] = 2 * cell(c1 + a, c2 + b) + 1
            idx[:, 1, k] = 2 * cell(c1 - a, c2 - b)
            dx[:, 0, k], dx[:, 1, k], dy[:, 0, k], dy[:, 1, k] = x, -x, y, -y
        if lattice == "haldane":
            for k, (a, b) in enumerate([(1, 0), (-1, 0), (-1, 1), (1, -1), (0, -1), (0, 1)]):
                for s in (0, 1):
                    idx[:, s, 3 + k] = 2 * cell(c1 + a, c2 + b) + s
                dx[:, :, 3 + k], dy[:, :, 3 + k] = a * SQ3 + b * SQ3 / 2, 1.5 * b
        y = c2.double().repeat_interleave(2)
        return idx.view(-1, K), dx.view(-1, K), dy.view(-1, K), y, L1 * SQ3, nc * 1.5 * SQ3
    n = {"chain": L1, "square": L1 * L2, "cubic": L1 ** 3}[lattice]
    dims = {"chain": (L1,), "square": (L1, L2), "cubic": (L1,) * 3}[lattice]
    s = torch.arange(n, device=DEV)
    cols, stride = [], 1
    for L in dims:
        x = (s // stride) % L
        cols += [s + ((x + 1) % L - x) * stride, s + ((x + L - 1) % L - x) * stride]
        stride *= L
    K = len(cols)
    dx = torch.zeros((n, K), dtype=torch.float64, device=DEV)
    dy = torch.zeros_like(dx)
    dx[:, 0], dx[:, 1] = 1.0, -1.0
    if K > 2:
        dy[:, 2], dy[:, 3] = 1.0, -1.0
    return torch.stack(cols, 1), dx, dy, (s // dims[0]).double(), float(L1), float(n)


class _Model:
    pass


def _model(case, seed):
    """The model in 64 bits on the GPU: idx, hop, onsite, dx, dy, volume."""
    m = _Model()
    if case["op"] == "ragged":
        sides = [case["Lmin"] + int(u * (case["Lmax"] - case["Lmin"] + 1)) for u in _uniform(seed, 3, case["count"]).tolist()]
        parts, off = [], [0]
        for q, L in enumerate(sides):
            idx, dx, dy, _, _, vol = _geometry("cubic", L, 1)
            parts.append((idx + off[-1], dx, case["W"] * (_uniform(seed, 100 + q, L ** 3) - 0.5)))
            off.append(off[-1] + L ** 3)
        m.idx, m.dx, m.onsite = (torch.cat([p[k] for p in parts]) for k in range(3))
        m.dy, m.hop, m.length, m.volume = None, torch.full(m.dx.shape, -1.0, dtype=torch.float64, device=DEV), 0.0, float(off[-1])
        m.seg = off
        m.n, m.K = m.idx.shape
        return m
    lattice = "haldane" if case["op"] == "hall" else case["lattice"]
    m.idx, m.dx, m.dy, y, m.length, m.volume = _geometry(lattice, case["L1"], case["L2"])
    m.n, m.K = m.idx.shape
    m.seg = None
    m.onsite = case["W"] * (_uniform(seed, 1, m.n) - 0.5)
    m.hop = torch.full((m.n, m.K), HOPPING[lattice], dtype=torch.float64, device=DEV)
    if lattice == "haldane":  # next-nearest hops i t2 with alternating sign, opposite on the two sublattices
        sign = torch.tensor([1.0, -1.0, 1.0, -1.0, 1.0, -1.0], dtype=torch.float64, device=DEV)
        m.hop = m.hop.to(torch.complex128)
        m.hop[0::2, 3:] = 0.15j * sign
        m.hop[1::2, 3:] = -0.15j * sign
    nv = round(case.get("vacancies", 0.0) * m.n)
    if nv:
        u = _draws(seed, 2, m.n) ^ -(1 << 63)  # unsigned order of the 64-bit draws
        gone = torch.zeros(m.n, dtype=torch.bool, device=DEV)
        gone[torch.argsort(u, stable=True)[:nv]] = True
        m.hop[gone[:, None] | gone[m.idx]] = 0.0
    if case.get("field"):  # perpendicular magnetic field: Peierls phases in the Landau gauge
        rows = float(y.max()) + 1
        phase = 2 * math.pi * case["field"] / rows * m.dx * 0.5 * (y[:, None] + y[m.idx])
        m.hop = torch.polar(m.hop.abs(), phase) * torch.sign(m.hop)
    return m


def _handle(case, seed):
    """The library handle of a case: built-in kinds by their parameters, the others
    through the paper's input form."""
    prec = g.GQT_FP32_ACC64 if case["fp32"] else g.GQT_FP64
    if case["op"] in ("dos", "vac", "msd", "grad") and not case["field"]:
        return g.gqt_build_hamiltonian(kind=KINDS[case["lattice"]], L1=case["L1"], L2=case["L2"],
                                       t=HOPPING[case["lattice"]], W=case["W"], vacancy_frac=case["vacancies"],
                                       seed=seed, energy_scale=_scale(case), precision=prec)
    m = _model(case, seed)
    lat = types.SimpleNamespace(
        n=m.n, max_nb=m.K, nb_count=np.full(m.n, m.K, np.int32), nb_idx=m.idx.to(torch.int32).cpu().numpy(),
        hop=m.hop.cpu().numpy(), onsite=m.onsite.cpu().numpy(), dx=m.dx.cpu().numpy(), length_x=m.length,
        volume=m.volume, seg_offsets=None if m.seg is None else np.array(m.seg, np.int64))
    if m.dy is not None:
        lat.dy = m.dy.cpu().numpy()
    return g.gqt_build_hamiltonian(lat, _scale(case), prec)


def _vectors(case, seed, n, seg=None):
    """Random-phase vectors of unit norm per segment, [n, R], as the program holds them."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    R = case.get("R", 1)
    theta = 2 * math.pi * torch.rand((n, R), dtype=torch.float64, device=DEV, generator=gen)
    if seg is None:
        amp = torch.full((n, 1), 1 / math.sqrt(n), dtype=torch.float64, device=DEV)
    else:
        size = torch.tensor(seg[1:], device=DEV) - torch.tensor(seg[:-1], device=DEV)
        amp = (1 / torch.sqrt(size.double())).repeat_interleave(size)[:, None]
    return torch.polar(amp.expand(n, R).contiguous(), theta).to(torch.complex64 if case["fp32"] else torch.complex128)


def _energies(case, dE):
    return torch.linspace(-0.97 * dE, 0.97 * dE, case["NE"], dtype=torch.float64, device=DEV)


def _loss_weights(case, seed):
    """Moment weights of a smooth energy window in each row, decaying like those of a damped series."""
    gen = torch.Generator().manual_seed(seed)
    x = 0.4 * torch.rand(case["rows"], 1, dtype=torch.float64, generator=gen) - 0.2
    k = torch.arange(case["M"], dtype=torch.float64)[None, :]
    damp = 0.5 * (1 + torch.cos(math.pi * k / case["M"]))
    return ((1 + (k > 0)) * torch.cos(k * torch.acos(x)) * torch.exp(-((8 * k / case["M"]) ** 2)) * damp).numpy()


# ------------------------------------------------------------------ one pass

def prepare(case, seed):
    s = types.SimpleNamespace(case=case, op=case["op"])
    if s.op == "kpm":
        gen = torch.Generator(device=DEV).manual_seed(seed)
        k = torch.arange(case["M"], dtype=torch.float64, device=DEV)
        s.mu = torch.randn((case["rows"], case["M"]), dtype=torch.float64, device=DEV, generator=gen) / (1 + k)
        s.E = torch.linspace(-8.0, 8.0, case["NE"], dtype=torch.float64, device=DEV)
        s.rho, s.sigma = (torch.empty((case["rows"], case["NE"]), dtype=torch.float64, device=DEV) for _ in range(2))
        s.dt = np.full(case["rows"], 2.0 / 2.7)
        return s
    s.ham = _handle(case, seed)
    s.R = case.get("R", 1)
    s.M = case["M"]
    seg = None
    if s.op == "ragged":
        seg = _model(case, seed).seg
    s.phi = _vectors(case, seed, s.ham.n, seg)
    if s.op in ("dos", "ragged"):
        s.mu = torch.empty((s.ham.nseg, s.R, s.M), dtype=torch.float64, device=DEV)
    elif s.op in ("vac", "msd"):
        s.x, s.y = torch.empty_like(s.phi), torch.empty_like(s.phi)
        s.dt = np.full(case["steps"], case["dt"] / abs(HOPPING[case["lattice"]]))
        s.mu = torch.empty((case["steps"], s.ham.nseg, s.R, s.M), dtype=torch.float64, device=DEV)
    elif s.op == "grad":
        s.dt = np.full(case["rows"], case["dt"] / abs(HOPPING[case["lattice"]]))
        s.beta = _loss_weights(case, seed)
        s.g_onsite = torch.empty(s.ham.n, dtype=torch.float64, device=DEV)
        s.g_slot = torch.empty((s.ham.n, SLOTS[case["lattice"]], 2), dtype=torch.float64, device=DEV)
    else:
        g.gqt_set_kb_contraction(s.ham, 1 if case["fp32"] else 0)
        s.lam = torch.empty((s.M, s.M), dtype=torch.complex128, device=DEV)
        s.E = _energies(case, s.ham.energy_scale)
        s.sigma = torch.empty_like(s.E)
    return s


def run(s):
    if s.op in ("dos", "ragged"):
        return g.gqt_dos_moments(s.ham, s.phi, s.R, s.M, s.mu)
    if s.op == "vac":
        g.gqt_vac_init(s.ham, s.phi, s.x, s.y, s.R)
        g.gqt_vac_moments(s.ham, s.x, s.y, s.R, s.dt, s.M, s.mu)
        return s.mu, s.x, s.y
    if s.op == "msd":
        g.gqt_msd_init(s.ham, s.phi, s.x, s.y, s.R)
        g.gqt_msd_moments(s.ham, s.x, s.y, s.R, s.dt, s.M, s.mu)
        return s.mu, s.x, s.y
    if s.op == "grad":
        loss = g.gqt_vac_loss_grad(s.ham, s.phi, s.dt, s.M, s.beta, s.g_onsite, s.g_slot)
        return loss, s.g_onsite, s.g_slot
    if s.op == "hall":
        g.gqt_kb_moments(s.ham, s.phi, s.R, s.M, 0, 1, s.lam)
        g.gqt_kubo_bastin(s.lam, s.E, s.ham.energy_scale, s.ham.volume, s.sigma)
        return s.lam, s.sigma
    g.gqt_kpm_reconstruct(s.mu, s.E, 9.555, 0.77, s.rho)
    g.gqt_sigma_vac(s.rho, s.dt, s.sigma)
    return s.rho, s.sigma


def work(case):
    """Bytes: the model, the vectors and the results once.  Flops: the recursions
    (two moments an order by the product identities), evolutions and contractions."""
    op = case["op"]
    if op == "kpm":
        rows, M, NE = case["rows"], case["M"], case["NE"]
        return {"bytes": 8 * (rows * M + NE + 2 * rows * NE), "flops": 2.0 * rows * M * NE}
    if op == "ragged":
        n = case["count"] * (0.5 * (case["Lmin"] + case["Lmax"])) ** 3
        K = 6
    else:
        n, K = _sites(case), SLOTS[case.get("lattice", "haldane")]
    R, M = case.get("R", 1), case["M"]
    e = 8 if case["fp32"] else 16
    cx = 4.0 if case.get("field") or op == "hall" else 2.0
    matrix = n * (K * (4 + (e if cx == 4.0 else e / 2)) + e / 2)
    order = n * R * (2 * cx * K + 4)  # one application of H and the recurrence
    if op in ("dos", "ragged"):
        return {"bytes": matrix + n * R * e + 8 * R * M, "flops": M / 2 * (order + 8 * n * R)}
    if op in ("vac", "msd"):
        Np = _orders(case)
        chains = 2 if op == "vac" else 1
        row = M / 2 * (chains * order + 8 * n * R)
        evolve = Np * (2 * order + 8 * n * R + (2 * cx * K * n * R if op == "msd" else 0))
        return {"bytes": matrix + 3 * n * R * e + 8 * case["steps"] * R * M, "flops": case["steps"] * (row + evolve)}
    if op == "grad":
        Np = _orders(case)
        step = 2 * order + n * (4 + 8 * K)  # forward and adjoint orders, the gradient terms
        rows = case["rows"]
        return {"bytes": matrix + n * e + 8 * n + 16 * n * K, "flops": rows * M * step + (rows - 1) * 2 * Np * (step + order)}
    chains = M * (3 * order)
    return {"bytes": matrix + 16 * n * K + n * R * e + 16 * M * M + 16 * case["NE"],
            "flops": chains + 8.0 * M * M * n * R + 4.0 * M * case["NE"]}


def _orders(case):
    x = _scale(case) * case["dt"] / abs(HOPPING[case["lattice"]])
    return int(x + 10 + 5 * x ** (1 / 3))


# ------------------------------------------------------------------ 64-bit values

def _bessel(x, count):
    """J_m(x), m < count, by backward recurrence."""
    top = 2 * ((max(count, int(x)) + 60) // 2)
    j = [0.0] * (top + 2)
    j[top] = 1e-280
    for m in range(top, 0, -1):
        j[m - 1] = 2 * m / x * j[m] - j[m + 1]
        if abs(j[m - 1]) > 1e200:
            j[m - 1:] = [v * 1e-200 for v in j[m - 1:]]
    norm = j[0] + 2 * sum(j[2::2])
    return [v / norm for v in j[:count]]


def _mul(m, h, x):
    """sum_k h[:, k] x[idx[:, k]], h [n, K]."""
    y = h[:, 0:1] * x.index_select(0, m.col[0])
    for k in range(1, m.K):
        y = y + h[:, k:k + 1] * x.index_select(0, m.col[k])
    return y


def _apply(m, x):
    """H~ x"""
    return _mul(m, m.h, x) + m.d * x


def _scaled(case, seed):
    m = _model(case, seed)
    dE = _scale(case)
    m.dE = dE
    m.h, m.d = m.hop / dE, (m.onsite / dE)[:, None]
    m.col = [m.idx[:, k].contiguous() for k in range(m.K)]
    return m


def _chebyshev(m, x):
    """T_0 x, T_1 x, ..."""
    a, b = x, _apply(m, x)
    yield a
    while True:
        yield b
        a, b = b, 2 * _apply(m, b) - a


def _dots(m, l, r, M):
    """Re <l|T_n(H~)|r> per segment and vector, [segments, R, M]."""
    rows = []
    for _, t in zip(range(M), _chebyshev(m, r)):
        p = l.real * t.real + l.imag * t.imag
        rows.append(torch.stack([p[a:b].sum(0) for a, b in zip(m.seg[:-1], m.seg[1:])]) if m.seg else p.sum(0)[None])
    return torch.stack(rows, -1)


def _velocity(m, x):
    return 1j * m.dE * _mul(m, m.dx * m.h, x)


def _coefs(m, dt, sign):
    x = m.dE * dt
    J = _bessel(x, int(x + 40 + 8 * x ** (1 / 3)))
    return [(1 if k == 0 else 2) * (-1j * sign) ** k * v for k, v in enumerate(J)]


def _evolve(m, x, dt, sign):
    out = 0
    for c, t in zip(_coefs(m, dt, sign), _chebyshev(m, x)):
        out = out + c * t
    return out


def _msd_step(m, p, px, dt):
    xh = -m.dx * m.h
    c = _coefs(m, dt, 1)
    u0, z0 = p, px
    u1, z1 = _apply(m, p), _mul(m, xh, p) + _apply(m, px)
    ap, ax = c[0] * u0 + c[1] * u1, c[0] * z0 + c[1] * z1
    for q in c[2:]:
        u0, u1, z0, z1 = u1, 2 * _apply(m, u1) - u0, z1, 2 * _mul(m, xh, u1) + 2 * _apply(m, z1) - z0
        ap, ax = ap + q * u1, ax + q * z1
    return ap, ax


def _gradient(case, m, phi, dt, beta):
    """Loss and its derivatives with respect to every on-site energy and every slot's hopping, by reverse mode."""
    onsite = m.onsite.clone().requires_grad_(True)
    hop = m.hop.to(torch.complex128).clone().requires_grad_(True)
    m.h, m.d = hop / m.dE, (onsite / m.dE)[:, None]
    a, b = phi, _velocity(m, phi)
    loss = 0.0
    beta = torch.from_numpy(beta).to(DEV)
    for k in range(case["rows"]):
        l = _velocity(m, a)
        acc = 0
        for w, t in zip(beta[k], _chebyshev(m, b)):
            acc = acc + w * t
        loss = loss + (l.real * acc.real + l.imag * acc.imag).sum()
        if k + 1 < case["rows"]:
            a, b = _evolve(m, a, dt[k], -1), _evolve(m, b, dt[k], -1)
    loss.backward()
    return float(loss), onsite.grad, torch.view_as_real(hop.grad).contiguous()


def _jackson(M):
    n, a = torch.arange(M, dtype=torch.float64, device=DEV), 1.0 / (M + 1)
    return (1 - n * a) * torch.cos(math.pi * n * a) + a * torch.sin(math.pi * n * a) / math.tan(math.pi * a)


def _hall(case, m, r):
    M, R = case["M"], case["R"]
    P, B = [], []
    for _, t, u in zip(range(M), _chebyshev(m, 1j * _mul(m, m.dx * m.h, r)), _chebyshev(m, r)):
        P.append(t.reshape(-1))
        B.append((1j * _mul(m, m.dy * m.h, u)).reshape(-1))
    lam = (m.n / R) * (torch.stack(P).conj() @ torch.stack(B).T)
    x = _energies(case, m.dE) / m.dE
    n = torch.arange(M, dtype=torch.float64, device=DEV)
    w = _jackson(M) * (1 + (n > 0))
    th = torch.acos(x)[:, None]
    T = w * torch.cos(n * th)
    A = w * torch.polar(torch.ones_like(T), -n * th) * torch.complex(x[:, None].expand_as(T), n * torch.sin(th))
    F = ((A @ lam.T) * T).sum(1).real + ((T.to(A.dtype) @ lam.T) * A.conj()).sum(1).real
    F = F / (1 - x * x) ** 2
    sigma = torch.zeros_like(F)
    sigma[1:] = torch.cumsum(0.5 * (x[1:] - x[:-1]) * (F[1:] + F[:-1]), 0)
    return lam, 2 / m.volume * sigma


def exact(case, seed):
    op = case["op"]
    if op == "kpm":
        s = prepare(case, seed)
        x = s.E / 9.555
        n = torch.arange(case["M"], dtype=torch.float64, device=DEV)
        T = torch.cos(n[:, None] * torch.acos(x)) * (_jackson(case["M"]) * (1 + (n > 0)))[:, None]
        rho = (s.mu @ T) * (2 * 0.77 / (math.pi * 9.555 * torch.sqrt(1 - x * x)))
        dt = torch.from_numpy(s.dt).to(DEV)[:-1, None]
        sigma = torch.zeros_like(rho)
        sigma[1:] = torch.cumsum(0.5 * dt * (rho[:-1] + rho[1:]), 0)
        return rho, sigma
    m = _scaled(case, seed)
    phi = _vectors(case, seed, m.n, m.seg).to(torch.complex128)
    M = case["M"]
    if op in ("dos", "ragged"):
        return _dots(m, phi, phi, M)
    if op in ("vac", "msd"):
        dt = case["dt"] / abs(HOPPING[case["lattice"]])
        x, y = (phi, _velocity(m, phi)) if op == "vac" else (phi, torch.zeros_like(phi))
        rows = []
        for _ in range(case["steps"]):
            if op == "vac":
                rows.append(_dots(m, _velocity(m, x), y, M))
                x, y = _evolve(m, x, dt, -1), _evolve(m, y, dt, -1)
            else:
                x, y = _msd_step(m, x, y, dt)
                rows.append(_dots(m, y, y, M))
        return torch.stack(rows), x, y
    if op == "grad":
        dt = np.full(case["rows"], case["dt"] / abs(HOPPING[case["lattice"]]))
        return _gradient(case, m, phi, dt, _loss_weights(case, seed))
    return _hall(case, m, phi)
