"""Evolution orders (Eq. 17) and the coupled commutator orders (Eqs. 18, 22, 24) with
the accumulator touched every third order: every length of the last group (expansions
of 1 to 7 orders and the full one), on every neighbour count.

  - FP64 handles with one vector above the size from which the orders run on pairs of
    FP32 numbers: within 1e-13 (U) and 1e-12 ([X,U]) of the FP64 kernels (arithmetic
    mode 0), the bounds of the pair arithmetic at smaller sizes;
  - FP32 handles, 1 to 32 vectors (scalar and two-wide lanes): within 2e-6 of the FP64
    handle on the same vectors (FP32 rounding of about 30 orders).

Bounds are on the difference's norm over the result's.
"""
import numpy as np
import pytest

import gqt_synth as S

torch = pytest.importorskip("torch")
g = pytest.importorskip("paper_1705_01387_gb300")

pytestmark = pytest.mark.gpu

LARGE = {
    "honeycomb": lambda: (S.honeycomb(160, 112, -2.7, 2.0, seed=3), S.energy_scale_rule(3, -2.7, 2.0)),
    "honeycomb_vac": lambda: (S.honeycomb(151, 113, -2.7, 2.0, seed=4, vacancy_frac=0.02),
                              S.energy_scale_rule(3, -2.7, 2.0)),
    "square": lambda: (S.square(191, 181, -1.0, 4.0, seed=5), S.energy_scale_rule(4, -1.0, 4.0)),
    "cubic": lambda: (S.cubic(33, -1.0, 16.5, seed=7), S.energy_scale_rule(6, -1.0, 16.5)),
    "chain": lambda: (S.chain(33001, -1.0, 4.0, seed=9), S.energy_scale_rule(2, -1.0, 4.0)),
}
SMALL = {
    "honeycomb": lambda: (S.honeycomb(13, 11, -2.7, 2.0, seed=3), S.energy_scale_rule(3, -2.7, 2.0)),
    "honeycomb_phases": lambda: (S.with_random_bond_phases(S.honeycomb(13, 11, -2.7, 2.0, seed=3), 4),
                                 S.energy_scale_rule(3, -2.7, 2.0)),
    "square": lambda: (S.square(17, 9, -1.0, 4.0, seed=5), S.energy_scale_rule(4, -1.0, 4.0)),
    "cubic": lambda: (S.cubic(7, -1.0, 16.5, seed=7), S.energy_scale_rule(6, -1.0, 16.5)),
    "chain": lambda: (S.chain(301, -1.0, 4.0, seed=9), S.energy_scale_rule(2, -1.0, 4.0)),
    "haldane": lambda: (S.haldane(7, 6, -1.0, 0.15, 1.2, 0.1, 1.0, seed=3), 1.05 * (3 + 0.9 + 0.1 + 0.5)),
}


def _orders(ham, psi, R, dt, sign, Np):
    """U(sign dt) psi and [X, U(dt)] psi; an expansion cut below the rule fails the norm
    check after writing its result."""
    out = []
    for f in (lambda d, o: g.gqt_evolve(ham, d, R, dt, sign, Np), lambda d, o: g.gqt_commutator_evolve(ham, d, o, R, dt, Np)):
        d, o = psi.clone(), torch.empty_like(psi)
        try:
            f(d, o)
        except g.GqtError as e:
            assert e.status == g.GQT_ENORM
        out.append((d if not out else o).to(torch.complex128))
    return out


def _off(x, y):
    return float(torch.linalg.norm(x - y) / torch.linalg.norm(y))


@pytest.mark.parametrize("name", list(LARGE))
@pytest.mark.parametrize("sign", [1, -1])
def test_pair_orders(name, sign):
    lat, dE = LARGE[name]()
    ham = g.gqt_build_hamiltonian(lat, dE)
    psi = torch.from_numpy(S.random_phase(lat.n, 1, seed=31)).cuda()
    for Np in [1, 2, 3, 4, 5, 6, 7, g.gqt_np_rule(dE * 0.7)]:
        g.gqt_set_fp64_arith(ham, 1)
        u, x = _orders(ham, psi, 1, 0.7, sign, Np)
        g.gqt_set_fp64_arith(ham, 0)
        ur, xr = _orders(ham, psi, 1, 0.7, sign, Np)
        assert _off(u, ur) < 1e-13, Np
        assert Np == 1 or _off(x, xr) < 1e-12, Np


@pytest.mark.parametrize("name", list(SMALL))
@pytest.mark.parametrize("R", [1, 2, 8, 32])
def test_fp32_orders(name, R):
    lat, dE = SMALL[name]()
    h64 = g.gqt_build_hamiltonian(lat, dE)
    h32 = g.gqt_build_hamiltonian(lat, dE, g.GQT_FP32_ACC64)
    psi = torch.from_numpy(S.random_phase(lat.n, R, seed=32)).cuda().to(torch.complex64)
    for Np in [1, 2, 3, 4, 5, 6, 7, g.gqt_np_rule(dE * 0.7)]:
        u, x = _orders(h32, psi, R, 0.7, -1, Np)
        ur, xr = _orders(h64, psi.to(torch.complex128), R, 0.7, -1, Np)
        assert _off(u, ur) < 2e-6, Np
        assert Np == 1 or _off(x, xr) < 2e-6, Np
