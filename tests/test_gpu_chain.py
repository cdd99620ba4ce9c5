"""Chains of overlapped launches: an order starts before the one it reads from has ended and
waits for it.  Rows, gradients' evolution orders and Hall chains give the same bits each
time, replayed as graphs or launched one by one, alone or beside another handle's chain
on another stream of another thread."""
import threading

import numpy as np
import pytest

import gqt_synth as S

torch = pytest.importorskip("torch")
g = pytest.importorskip("paper_1705_01387_gb300")

pytestmark = pytest.mark.gpu


def _work(kind, seed):
    """A callable that runs one chain and returns its result as bytes."""
    if kind.startswith("hall"):
        lat = S.haldane(30, 29, -1.0, 0.15, 1.2, 0.0, 1.0, seed=seed)
        dE = 1.05 * (3 + 0.9 + 0.5)
        fp64 = kind == "hall64"
        ham = g.gqt_build_hamiltonian(lat, dE, g.GQT_FP64 if fp64 else g.GQT_FP32_ACC64)
        g.gqt_set_kb_contraction(ham, 0 if fp64 else 1)
        r = torch.from_numpy(S.random_phase(lat.n, 1, seed=seed)).to(torch.complex128 if fp64 else torch.complex64).cuda()
        lam = torch.empty((48, 48), dtype=torch.complex128, device="cuda")

        def run():
            g.gqt_kb_moments(ham, r, 1, 48, 0, 1, lam)
            return lam.cpu().numpy().tobytes()
        return run, ham
    arith, prec = (1, g.GQT_FP64) if kind == "df" else (0, g.GQT_FP64) if kind == "fp64" else (0, g.GQT_FP32_ACC64)
    lat = S.square(90, 77, -1.0, 2.0, seed=seed)
    dE = S.energy_scale_rule(4, -1.0, 2.0)
    ham = g.gqt_build_hamiltonian(lat, dE, prec)
    g.gqt_set_cluster(ham, False)
    if prec == g.GQT_FP64:
        g.gqt_set_fp64_arith(ham, arith)
    ct = torch.complex128 if prec == g.GQT_FP64 else torch.complex64
    v = [torch.from_numpy(S.random_phase(lat.n, 1, seed=seed + q)).to(ct).cuda() for q in range(4)]
    M = 60

    def run():
        dos, vac, msd = np.empty((1, 1, M)), np.empty((1, 1, 2, M)), np.empty((1, 1, 2, M))
        w = [x.clone() for x in v]
        g.gqt_dos_moments(ham, w[0], 1, M, dos)
        g.gqt_vac_moments(ham, w[0], w[1], 1, [0.7, 0.4], M, vac)
        g.gqt_msd_moments(ham, w[2], w[3], 1, [0.7, 0.4], M, msd)
        return dos.tobytes() + vac.tobytes() + msd.tobytes()
    return run, ham


@pytest.mark.parametrize("kind", ["df", "fp64", "fp32", "hall64", "hall32"])
def test_same_bits_each_time(kind):
    run, ham = _work(kind, 3)
    want = run()
    g.gqt_profile_start()  # events between the launches, no graphs
    assert run() == want
    torch.cuda.synchronize()
    g.gqt_profile_stop(12)
    bad = []

    def other():
        with torch.cuda.stream(torch.cuda.Stream()):
            r2, _ = _work(kind, 4)
            w2 = r2()
            bad.extend(1 for _ in range(15) if r2() != w2)

    t = threading.Thread(target=other)
    t.start()
    for _ in range(25):
        assert run() == want
    t.join()
    assert not bad
