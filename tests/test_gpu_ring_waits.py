"""Blocked honeycomb rows whose waits for their copies run out: with a limit of 0 polls every
CTA reports it, and every row that has not landed is drained before its slot is filled
again.  The call fails, the handle stays usable: with the default limit the next call
gives the bits of a handle whose waits never ran out.  One chain (DOS) and two (VAC),
each band width."""
import numpy as np
import pytest

import gqt_synth as S

torch = pytest.importorskip("torch")
g = pytest.importorskip("paper_1705_01387_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("graphs", [True, False])
@pytest.mark.parametrize("L1,L2", [(32, 3), (64, 40), (128 * 5, 300)])
def test_waits_that_run_out(L1, L2, graphs):
    ham = g.gqt_build_hamiltonian(kind=g.GQT_LATTICE_HONEYCOMB, L1=L1, L2=L2, t=-1.0, W=1.0, seed=1,
                                  energy_scale=S.energy_scale_rule(3, -1.0, 1.0))
    g.gqt_set_cluster(ham, False)
    g.gqt_set_graphs(ham, graphs)
    a, b = (torch.from_numpy(S.random_phase(ham.n, 1, seed=q)).cuda() for q in (0, 1))
    M = 12

    def rows():
        dos, vac = np.empty((1, 1, M)), np.empty((1, 1, 1, M))
        g.gqt_dos_moments(ham, a, 1, M, dos)
        g.gqt_vac_moments(ham, a.clone(), b.clone(), 1, [0.0], M, vac)
        return dos.tobytes() + vac.tobytes()

    want = rows()
    g.gqt_set_wait_limit(ham, 0)
    for call in (lambda: g.gqt_dos_moments(ham, a, 1, M, np.empty((1, 1, M))),
                 lambda: g.gqt_vac_moments(ham, a.clone(), b.clone(), 1, [0.0], M, np.empty((1, 1, 1, M)))):
        with pytest.raises(g.GqtError) as ei:
            call()
        assert ei.value.status == g.GQT_ETIMEOUT
        assert "drain" not in str(ei.value)
    g.gqt_set_wait_limit(ham, 1 << 24)
    assert rows() == want


def test_a_wait_that_ran_out_is_named_first():
    """A row of NaN whose waits run out: the status is that of the wait, whose consequence a
    NaN in a result may be."""
    ham = g.gqt_build_hamiltonian(kind=g.GQT_LATTICE_HONEYCOMB, L1=64, L2=40, t=-1.0, W=1.0, seed=1,
                                  energy_scale=S.energy_scale_rule(3, -1.0, 1.0))
    g.gqt_set_cluster(ham, False)
    a = torch.full((ham.n, 1), float("nan"), dtype=torch.complex128, device="cuda")
    for limit, status in ((1 << 24, g.GQT_ENAN), (0, g.GQT_ETIMEOUT)):
        g.gqt_set_wait_limit(ham, limit)
        with pytest.raises(g.GqtError) as ei:
            g.gqt_dos_moments(ham, a, 1, 12, np.empty((1, 1, 12)))
        assert ei.value.status == status
