"""The sliced FP64 Hall contraction whose device waits run out: with a limit of 0 polls every
role of a CTA gives up at once with copies in flight, which are drained, tensor memory is
freed and the call returns the status of a wait that gave up; with the default limit the
next call on the handle gives the bits of a handle whose waits never ran out."""
import math

import pytest

import gqt_synth as S

torch = pytest.importorskip("torch")
g = pytest.importorskip("paper_1705_01387_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,L1,L2", [(1, 3, 3), (130, 33, 17), (256, 40, 41)])
def test_waits_that_run_out(M, L1, L2):
    lat = S.haldane(L1, L2, -1.0, 0.15, math.pi / 2, 0.0, 1.0, seed=7)
    ham = g.gqt_build_hamiltonian(lat, 1.05 * (3 + 6 * 0.15 + 0.5))
    r = torch.from_numpy(S.random_phase(lat.n, 1, seed=35)).cuda()

    def moments():
        lam = torch.empty((M, M), dtype=torch.complex128, device="cuda")
        g.gqt_kb_moments(ham, r, 1, M, 0, 1, lam)
        return lam.cpu().numpy().tobytes()

    want = moments()
    g.gqt_set_wait_limit(ham, 0)
    with pytest.raises(g.GqtError) as ei:
        moments()
    assert ei.value.status == g.GQT_ETIMEOUT and "drain" not in str(ei.value)
    g.gqt_set_wait_limit(ham, 1 << 24)
    assert moments() == want
