"""Blocked honeycomb rows with the band rows in shared memory, where the ring of rows can
go wrong: the fewest rows a lattice can have (three; two are not blocked), the three band widths, a piece longer than
the 256 rows whose halo columns are kept, more bands than resident CTAs, and the three
forms of hoppings.  DOS (one chain) and VAC (two chains) rows agree with the single-order
kernels within 1e-13 of mu_0 (the bound of the other blocked tests)."""
import numpy as np
import pytest

import gqt_synth as S

torch = pytest.importorskip("torch")
g = pytest.importorskip("paper_1705_01387_gb300")

pytestmark = pytest.mark.gpu


def _lattice(L1, L2, form):
    lat = S.honeycomb(L1, L2, -2.7, 2.0, seed=L1 + L2, vacancy_frac=0.01 if form == "values" else 0.0)
    if form == "phases":
        lat = S.with_random_bond_phases(lat, L2)
    return lat


@pytest.mark.parametrize("L1,L2,form", [(32, 2, "uniform"), (32, 3, "phases"), (64, 3, "values"), (128, 2, "values"),
                                        (160, 7, "phases"), (128, 700, "uniform"), (64, 300, "values"),
                                        (32 * 1021, 9, "uniform"), (32 * 1021, 5, "phases")])
def test_rows_agree_with_single_orders(L1, L2, form):
    lat = _lattice(L1, L2, form)
    dE = S.energy_scale_rule(3, -2.7, 2.0)
    M = 10
    a = torch.from_numpy(S.random_phase(lat.n, 1, seed=1)).cuda()
    b = torch.from_numpy(S.random_phase(lat.n, 1, seed=2)).cuda()
    rows = []
    for blocked in (True, False):
        ham = g.gqt_build_hamiltonian(lat, dE)
        g.gqt_set_cluster(ham, False)
        g.gqt_set_temporal_blocking(ham, blocked)
        dos, vac = np.empty((1, 1, M)), np.empty((1, 1, 1, M))
        g.gqt_profile_start()
        g.gqt_dos_moments(ham, a, 1, M, dos)
        g.gqt_vac_moments(ham, b.clone(), a.clone(), 1, [0.0], M, vac)
        torch.cuda.synchronize()
        _, n = g.gqt_profile_stop(12)
        assert (n[10] > 0 and n[11] > 0) == (blocked and L2 >= 3)
        rows.append((dos.ravel(), vac.ravel()))
    for x, y in zip(*rows):
        assert np.all(np.abs(x - y) < 1e-13)
