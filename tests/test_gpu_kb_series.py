"""gqt_kubo_bastin and gqt_kubo_bastin_fermi by the collapsed series (the M x M
moments summed along their diagonals once, then 2M - 1 angles per energy), at the
edges of its splits: one moment, the 32-row collapse and 512-angle re-anchoring
boundaries, rows per split above 32 (M > 1024), one energy, a warp's remainder, and
more energies than scan threads.  Bound: 1e-10 of the largest value, that of the
FP64 path."""
import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
g = pytest.importorskip("paper_1705_01387_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,NE", [(1, 5), (2, 1), (31, 33), (32, 1023), (33, 1025), (256, 130), (257, 9), (510, 40),
                                  (1100, 6)])
@pytest.mark.parametrize("kernel", [0, 1])
def test_series_matches_oracle(M, NE, kernel):
    rng = np.random.default_rng(M + NE)
    dE, area = 3.7, 12.5
    lam = (rng.standard_normal((M, M)) + 1j * rng.standard_normal((M, M))) / (1 + np.arange(M))[None, :]
    E = np.linspace(-0.95 * dE, 0.9 * dE, NE) if NE > 1 else np.array([0.3])
    d = torch.from_numpy(lam).cuda()
    sig = torch.empty(NE, dtype=torch.float64, device="cuda")
    g.gqt_kubo_bastin(d, torch.from_numpy(E).cuda(), dE, area, sig, kernel=kernel)
    ref = O.kubo_bastin(lam, E, dE, area, kernel)
    scale = max(float(np.max(np.abs(ref))), 1e-300)
    assert float(np.max(np.abs(sig.cpu().numpy() - ref))) <= 1e-10 * scale
    if NE < 2:
        return
    mu = np.array([-2.0, E[NE // 2], 1.7])
    out = torch.empty(3, dtype=torch.float64, device="cuda")
    g.gqt_kubo_bastin_fermi(d, torch.from_numpy(E).cuda(), dE, area, torch.from_numpy(mu).cuda(), 0.05, out,
                            kernel=kernel)
    ref = O.kubo_bastin_fermi(lam, E, dE, area, mu, 0.05, kernel)
    assert float(np.max(np.abs(out.cpu().numpy() - ref))) <= 1e-10 * max(float(np.max(np.abs(ref))), 1e-300)
