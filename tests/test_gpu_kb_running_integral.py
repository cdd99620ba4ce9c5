"""The running integral of gqt_kubo_bastin where a thread adds several panels (more energies
than threads): the lower limit is an empty sum, 0, also where the integrand is NaN, and
the values are the panels added one after another to rounding (1e-13 of the largest)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
g = pytest.importorskip("paper_1705_01387_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("NE", [3, 1024, 1025, 3001, 40000])
def test_lower_limit_and_order(NE):
    M, dE = 5, 2.0
    rng = np.random.default_rng(NE)
    lam = torch.from_numpy(rng.standard_normal((M, M)) + 1j * rng.standard_normal((M, M))).cuda()
    E = torch.linspace(-1.8, 1.8, NE, dtype=torch.float64, device="cuda")
    out = torch.empty_like(E)
    g.gqt_kubo_bastin(lam, E, dE, 3.0, out)
    got = out.cpu().numpy()
    # the panels from the two-point integrals of neighbouring energies
    pick = np.unique(np.linspace(0, NE - 2, 40).astype(int))
    two = torch.empty(2, dtype=torch.float64, device="cuda")
    for j in pick:
        g.gqt_kubo_bastin(lam, E[j:j + 2].contiguous(), dE, 3.0, two)
        assert abs((got[j + 1] - got[j]) - float(two[1])) <= 1e-13 * np.abs(got).max()
    lam[2, 1] = float("nan")
    g.gqt_kubo_bastin(lam, E, dE, 3.0, out)
    got = out.cpu().numpy()
    assert got[0] == 0.0 and np.isnan(got[1:]).all()
