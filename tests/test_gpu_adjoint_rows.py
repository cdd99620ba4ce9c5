"""Gradients with the forward vectors kept (no stride given) and with checkpoints, for the
unrolled neighbour counts and the general one, few orders, real and complex hoppings, and
both storages: the kept vectors are the recomputed ones, so both ways agree to rounding
(1e-13 of the largest entry), and in FP64 with the oracle (1e-10, as the other gradient
tests)."""
import dataclasses

import numpy as np
import pytest

import gqt_synth as S
import oracle as O

torch = pytest.importorskip("torch")
g = pytest.importorskip("paper_1705_01387_gb300")

pytestmark = pytest.mark.gpu

LATTICES = {
    2: lambda: S.chain(131, -1.0, 1.0, seed=1),
    3: lambda: S.honeycomb(9, 8, -1.0, 1.0, seed=1),
    4: lambda: S.square(11, 13, -1.0, 1.0, seed=1),
    6: lambda: S.cubic(5, -1.0, 1.0, seed=1),
    9: lambda: dataclasses.replace(S.haldane(8, 9, -1.0, 0.15, 1.1, 0.0, 1.0, seed=1), dy=None),
}


def _nerr(x, y):
    return float(np.max(np.abs(x - y)) / max(float(np.max(np.abs(y))), 1e-300))


@pytest.mark.parametrize("K", list(LATTICES))
@pytest.mark.parametrize("M", [1, 2, 3, 4, 5, 30])
@pytest.mark.parametrize("prec", ["GQT_FP64", "GQT_FP32_ACC64"])
def test_kept_vectors_and_checkpoints(K, M, prec):
    lat = LATTICES[K]()
    if K == 4:
        lat = S.with_random_bond_phases(lat, 2)
    dE = S.energy_scale_rule(K, -1.0, 1.0)
    phi = S.random_phase(lat.n, 1, seed=M)[:, 0]
    dts = np.array([0.5, 0.3])
    Np = [O.np_rule(dE * d, 64) for d in dts]
    beta = np.random.default_rng(M).standard_normal((2, M))
    ham = g.gqt_build_hamiltonian(lat, dE, getattr(g, prec))
    d = torch.from_numpy(phi.reshape(-1, 1)).to(torch.complex128 if prec == "GQT_FP64" else torch.complex64).cuda()
    out = []
    for stride in (0, 4):
        ge = torch.empty(lat.n, dtype=torch.float64, device="cuda")
        gs = torch.empty((lat.n, lat.max_nb, 2), dtype=torch.float64, device="cuda")
        J = g.gqt_vac_loss_grad(ham, d, dts, M, beta, ge, gs, Np=Np, stride=stride)
        s = gs.cpu().numpy()
        out.append((J, ge.cpu().numpy(), s[..., 0] + 1j * s[..., 1]))
    (J, ge, gs), (Jc, gec, gsc) = out
    assert abs(J - Jc) <= 1e-13 * abs(Jc) and _nerr(ge, gec) < 1e-13 and _nerr(gs, gsc) < 1e-13
    if prec == "GQT_FP64":
        Jr, ger, gsr = O.Hamiltonian(lat, dE).vac_loss_grad(phi, dts, Np, beta)
        assert abs(J - Jr) <= 1e-10 * max(abs(Jr), 1e-3) and _nerr(ge, ger) < 1e-10 and _nerr(gs, gsr) < 1e-10
