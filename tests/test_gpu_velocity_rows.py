"""V x (Eq. 34) by the unrolled kernel and the general one: 2, 3, 4, 6 and 9 slots, one and
several vectors, pairs of vectors that are 16-byte aligned and that are not, with and
without row classes, real and complex hoppings, sizes around a CTA.  Reference in 64 bits;
bounds: 30 roundings of a row's terms, 30 * 2^-53 and 30 * 2^-24 of the largest entry."""
import dataclasses

import numpy as np
import pytest

import gqt_synth as S

torch = pytest.importorskip("torch")
g = pytest.importorskip("paper_1705_01387_gb300")

pytestmark = pytest.mark.gpu

LATTICES = {
    2: lambda: S.chain(255, -1.0, 1.0, seed=1),
    3: lambda: S.honeycomb(16, 8, -1.0, 1.0, seed=1),
    4: lambda: S.square(67, 71, -1.0, 1.0, seed=1),
    6: lambda: S.cubic(7, -1.0, 1.0, seed=1),
    9: lambda: S.haldane(8, 9, -1.0, 0.15, 1.1, 0.0, 1.0, seed=1),
}


@pytest.mark.parametrize("K", list(LATTICES))
@pytest.mark.parametrize("R", [1, 2, 8])
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("prec", ["GQT_FP64", "GQT_FP32_ACC64"])
@pytest.mark.parametrize("form", ["uniform", "phases", "relabelled"])
def test_velocity(K, R, shift, prec, form):
    lat = LATTICES[K]()
    if form == "phases":
        lat = S.with_random_bond_phases(lat, 2)
    elif form == "relabelled":
        p = np.random.default_rng(1).permutation(lat.n)
        q = np.argsort(p)
        lat = dataclasses.replace(lat, nb_count=lat.nb_count[q], nb_idx=p[lat.nb_idx[q]].astype(np.int32),
                                  hop=lat.hop[q], onsite=lat.onsite[q], dx=lat.dx[q], dy=None)
    fp64 = prec == "GQT_FP64"
    dE = S.energy_scale_rule(K, -1.0, 1.0)
    ham = g.gqt_build_hamiltonian(lat, dE, getattr(g, prec))
    ct = torch.complex128 if fp64 else torch.complex64
    v = torch.from_numpy(S.random_phase(lat.n, R, seed=K)).to(ct)

    def buffer():
        return torch.zeros(lat.n * R + 1, dtype=ct, device="cuda")[shift:shift + lat.n * R].view(lat.n, R)

    x, y = buffer(), buffer()
    x.copy_(v)
    g.gqt_apply_velocity(ham, x, y, R)
    w = v.to(torch.complex128).numpy()
    ref = 1j * sum((lat.dx * lat.hop)[:, k:k + 1] * w[lat.nb_idx[:, k]] for k in range(lat.max_nb))
    a, b = buffer(), buffer()
    g.gqt_vac_init(ham, x, a, b, R)
    tol = 30 * (2.0 ** -53 if fp64 else 2.0 ** -24) * np.abs(ref).max()
    assert np.abs(y.cpu().numpy() - ref).max() < tol
    assert torch.equal(b, y) and torch.equal(a, x)
