"""Threads, each with a handle of its own and a stream of its own, whose kernels are the
same and need different amounts of shared memory: rows and evolution on a cluster
(sites and moments), blocked honeycomb rows (rows of a band).  No call fails, and the rows
have the bits that they have alone."""
import threading

import numpy as np
import pytest

import gqt_synth as S

torch = pytest.importorskip("torch")
g = pytest.importorskip("paper_1705_01387_gb300")

pytestmark = pytest.mark.gpu


def _work(op, L1, L2, M, seed):
    """A callable that makes one call with a handle of its own, and one that returns its result."""
    ham = g.gqt_build_hamiltonian(kind=g.GQT_LATTICE_HONEYCOMB, L1=L1, L2=L2, t=-1.0, W=1.0, seed=seed,
                                  energy_scale=S.energy_scale_rule(3, -1.0, 1.0))
    g.gqt_set_cluster(ham, op != "blocked")
    g.gqt_set_vac_pair(ham, op != "cluster_row")
    g.gqt_set_graphs(ham, False)
    a, b = (torch.from_numpy(S.random_phase(ham.n, 1, seed=seed + q)).cuda() for q in (0, 1))
    mu = torch.empty((1, 1, 1, M), dtype=torch.float64, device="cuda")
    if op == "evolve":
        def call():  # there and back
            g.gqt_evolve(ham, a, 1, 0.8, 1)
            g.gqt_evolve(ham, a, 1, 0.8, -1)
        return call, None
    if op == "cluster_row":  # l != r rows by one recurrence
        dt = [0.0]
        return lambda: g.gqt_vac_moments(ham, a, b, 1, dt, M, mu), None
    return lambda: g.gqt_dos_moments(ham, a, 1, M, mu), lambda: mu.cpu().numpy().tobytes()


@pytest.mark.parametrize("op,large,small,times", [("evolve", (64, 60, 1), (4, 3, 1), 3000),
                                                  ("cluster", (64, 60, 400), (4, 3, 2), 3000),
                                                  ("cluster_row", (40, 40, 100), (4, 3, 2), 3000),
                                                  ("blocked", (2048, 256, 6), (128, 3, 6), 2000)])
def test_handles_of_different_size(op, large, small, times):
    errors, stop = [], threading.Event()

    def work(shape, seed, count):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                call, result = _work(op, *shape, seed)
                call()
                want = result and result()
                while count and not stop.is_set():
                    call()
                    count -= 1
                assert not result or result() == want
        except BaseException as e:
            errors.append(f"{shape}: {e!r}")

    others = [threading.Thread(target=work, args=(small, q, -1)) for q in (2, 3, 4)]
    for t in others:
        t.start()
    work(large, 1, times)
    stop.set()
    for t in others:
        t.join()
    assert not errors
