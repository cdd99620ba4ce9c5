"""Blocked honeycomb rows where a CTA walks several pieces: bands of rows cut into ranges
(more bands than an SM can hold CTAs of two warps, 32, on all SMs, so that a range crosses
the ends of bands), and pieces longer than the 256 rows whose halo columns are kept (as
many bands of 128 cells as leave one segment of 270 rows each at two or three CTAs of 128
registers or fewer per SM).  DOS (one chain) and VAC (two chains) rows agree with the
single-order kernels within 1e-13 of mu_0 (the bound of the other blocked tests)."""
import numpy as np
import pytest

import gqt_synth as S

torch = pytest.importorskip("torch")
g = pytest.importorskip("paper_1705_01387_gb300")

pytestmark = pytest.mark.gpu


def _rows(ham, blocked, M):
    g.gqt_set_cluster(ham, False)
    g.gqt_set_temporal_blocking(ham, blocked)
    a, b = (torch.empty((ham.n, 1), dtype=torch.complex128, device="cuda") for _ in range(2))
    g.gqt_random_phase(ham, 1, 1, a)
    g.gqt_random_phase(ham, 2, 1, b)
    dos, vac = np.empty((1, 1, M)), np.empty((1, 1, 1, M))
    g.gqt_profile_start()
    g.gqt_dos_moments(ham, a, 1, M, dos)
    g.gqt_vac_moments(ham, b, a, 1, [0.0], M, vac)
    torch.cuda.synchronize()
    _, n = g.gqt_profile_stop(12)
    assert (n[10] > 0 and n[11] > 0) == blocked
    return dos.ravel(), vac.ravel()


@pytest.mark.parametrize("form", ["uniform", "values", "phases"])
@pytest.mark.parametrize("bands,L2", [(None, 3), (None, 9), (301, 270)])
def test_pieces_agree_with_single_orders(bands, L2, form):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    L1 = 128 * bands if bands else 32 * (32 * sms + 135 | 1)
    if bands and form == "phases":
        pytest.skip("20.8M sites through the input form")
    dE = S.energy_scale_rule(3, -2.7, 2.0)
    if form == "phases":
        ham = g.gqt_build_hamiltonian(S.with_random_bond_phases(S.honeycomb(L1, L2, -2.7, 2.0, seed=L2), L2), dE)
    else:
        ham = g.gqt_build_hamiltonian(kind=g.GQT_LATTICE_HONEYCOMB, L1=L1, L2=L2, t=-2.7, W=2.0, seed=L2,
                                      vacancy_frac=0.01 if form == "values" else 0.0, energy_scale=dE)
    M = 10
    for x, y in zip(_rows(ham, True, M), _rows(ham, False, M)):
        assert np.all(np.abs(x - y) < 1e-13)
