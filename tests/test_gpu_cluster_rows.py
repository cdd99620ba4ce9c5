"""Cluster-resident rows with one site per thread (k_cheb_cluster1) at the edges of their
range: one to 512 sites per CTA (ring parts of 1 to 16 lanes), rows shorter than, equal
to and just past a whole ring of dots, 2, 3, 4 and 6 neighbour slots, real and complex
hoppings, and the sizes above it.  Against the oracle: 1e-10 for FP64 handles, 1e-5
(l = r rows) for FP32 ones, of the largest moment."""
import numpy as np
import pytest

import gqt_synth as S
import oracle as O

torch = pytest.importorskip("torch")
g = pytest.importorskip("paper_1705_01387_gb300")

pytestmark = pytest.mark.gpu

MODELS = {
    "chain3": lambda: (S.chain(3, -1.0, 4.0, seed=9), S.energy_scale_rule(2, -1.0, 4.0)),
    "chain513": lambda: (S.chain(513, -1.0, 4.0, seed=9), S.energy_scale_rule(2, -1.0, 4.0)),
    "chain8192": lambda: (S.chain(8192, -1.0, 4.0, seed=8), S.energy_scale_rule(2, -1.0, 4.0)),
    "chain8193": lambda: (S.chain(8193, -1.0, 4.0, seed=8), S.energy_scale_rule(2, -1.0, 4.0)),
    "honeycomb": lambda: (S.honeycomb(32, 32, -2.7, 1.0, seed=3), S.energy_scale_rule(3, -2.7, 1.0)),
    "honeycomb_phases": lambda: (S.with_random_bond_phases(S.honeycomb(9, 7, -2.7, 2.0, seed=3), 4),
                                 S.energy_scale_rule(3, -2.7, 2.0)),
    "square": lambda: (S.square(41, 29, -1.0, 4.0, seed=5), S.energy_scale_rule(4, -1.0, 4.0)),
    "cubic": lambda: (S.cubic(13, -1.0, 16.5, seed=7), S.energy_scale_rule(6, -1.0, 16.5)),
}


def nerr(x, y):
    return float(np.max(np.abs(x - y)) / max(float(np.max(np.abs(y))), 1e-300))


@pytest.mark.parametrize("name", list(MODELS))
@pytest.mark.parametrize("M", [1, 2, 3, 31, 32, 33, 65, 130])
def test_rows_match_oracle(name, M):
    lat, dE = MODELS[name]()
    h = O.Hamiltonian(lat, dE)
    phi = S.random_phase(lat.n, 1, seed=M)
    d = torch.from_numpy(phi).cuda()
    ham = g.gqt_build_hamiltonian(lat, dE)
    mu = np.empty((1, 1, M))
    g.gqt_dos_moments(ham, d, 1, M, mu)
    assert nerr(mu.ravel(), h.dos_moments(phi[:, 0], M).real) < 1e-10
    a, b = torch.empty_like(d), torch.empty_like(d)
    g.gqt_vac_init(ham, d, a, b, 1)
    vac = np.empty((2, 1, 1, M))
    Np = [O.np_rule(dE * 0.4, 64)] * 2
    g.gqt_vac_moments(ham, a, b, 1, [0.4, 0.4], M, vac, Np=Np)
    assert nerr(vac.reshape(2, M), h.vac_moments(phi[:, 0], [0.4, 0.4], Np, M)) < 1e-10
    h32 = g.gqt_build_hamiltonian(lat, dE, g.GQT_FP32_ACC64)
    g.gqt_dos_moments(h32, d.to(torch.complex64), 1, M, mu)
    assert nerr(mu.ravel(), h.dos_moments(phi[:, 0], M).real) < 1e-5


def test_scale_too_small_is_refused():
    lat, dE = MODELS["honeycomb"]()
    ham = g.gqt_build_hamiltonian(lat, 0.5 * dE)
    d = torch.from_numpy(S.random_phase(lat.n, 1, seed=1)).cuda()
    with pytest.raises(g.GqtError) as e:
        g.gqt_dos_moments(ham, d, 1, 256, np.empty((1, 1, 256)))
    assert e.value.status in (g.GQT_ERANGE, g.GQT_ENAN)
