"""Captured graphs and workspaces that move: a handle that has replayed its launches as
graphs is used at another number of vectors, whose larger workspace takes the place of
the one the graphs were captured with, and then as before.  The graphs are retired (the
same calls with the same arrays are launched anew) and the results are those of a
handle that has seen one number of vectors only."""
import numpy as np
import pytest

import gqt_synth as S

torch = pytest.importorskip("torch")
g = pytest.importorskip("paper_1705_01387_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,slots", [(g.GQT_LATTICE_CHAIN, 2), (g.GQT_LATTICE_HONEYCOMB, 3)])
@pytest.mark.parametrize("call", ["vac", "msd"])
def test_graphs_are_retired_with_their_workspaces(kind, slots, call):
    dE = S.energy_scale_rule(slots, -1.0, 1.0)

    def handle():
        return g.gqt_build_hamiltonian(kind=kind, L1=50000 if slots == 2 else 130, L2=193, t=-1.0, W=1.0, seed=5,
                                       energy_scale=dE, precision=g.GQT_FP32_ACC64)

    M, dts = 11, [0.5]
    hams = [handle(), handle()]
    n = hams[0].n
    start = {R: [torch.from_numpy(S.random_phase(n, R, seed=R + q)).to(torch.complex64).cuda() for q in (0, 1)]
             for R in (4, 16, 32)}
    state = {R: [x.clone() for x in v] for R, v in start.items()}

    def rows(ham, R):
        """Moments, final states and the number of launches of one call on the arrays of R."""
        for x, x0 in zip(state[R], start[R]):
            x.copy_(x0)
        mu = np.empty((1, 1, R, M))
        torch.cuda.synchronize()
        c0 = g.lib().gqt_launch_count()
        (g.gqt_vac_moments if call == "vac" else g.gqt_msd_moments)(ham, *state[R], R, dts, M, mu)
        c1 = g.lib().gqt_launch_count()
        return [mu.tobytes()] + [x.cpu().numpy().tobytes() for x in state[R]], c1 - c0

    want, first = rows(hams[0], 4)
    used = hams[1]
    g.gqt_evolve(used, state[32][0], 32, 0.5, 1)  # one set at R = 32: only the first buffers of a pair are this large
    assert rows(used, 4)[0] == want
    replayed, few = rows(used, 4)
    assert replayed == want and few < first
    rows(used, 16)  # the second buffers grow
    again, many = rows(used, 4)
    assert again == want
    assert many > few  # launched anew
    assert rows(used, 4) == (want, few)
