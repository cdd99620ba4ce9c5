"""Angles of the reconstruction near the band edges, in the pass for a few rows and in the
sliced product: cos(n acos x) at x = E / dE rounded once, against extended precision.  The
energies are those whose quotient differs from the product with 1 / dE, by an ulp, which
an order n turns into n 2^-53 / sin th.  Bound: two ulp of th times n, and a ulp for
each of up to 64 rotations, three for the slices: 20 to 200 times below that."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
g = pytest.importorskip("paper_1705_01387_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sign", [1, -1])
@pytest.mark.parametrize("rows", [8, 9])
def test_quotient_near_the_band_edges(rows, sign):
    dE, M = 3.7, 1000
    E = dE * sign * (1 - np.geomspace(1e-6, 1e-3, 4000))
    x = E / dE
    pick = x != E * (1.0 / dE)
    assert pick.sum() > 200
    E, x = E[pick], x[pick].astype(np.longdouble)
    th = np.arccos(sign * x)  # small: near the other edge cos n th only changes sign
    order = M - 1 - 7 * np.arange(rows)
    mu = np.zeros((rows, M))
    mu[np.arange(rows), order] = 1.0
    out = torch.empty((rows, E.size), dtype=torch.float64, device="cuda")
    g.gqt_kpm_reconstruct(torch.from_numpy(mu).cuda(), torch.from_numpy(E).cuda(), dE, 1.0, out, kernel=1)
    got = out.cpu().numpy().astype(np.longdouble) * (np.pi * dE * np.sqrt((1 - x) * (1 + x)) / 2)
    want = 2 * np.cos(order[:, None] * th) * np.where(order % 2 == 1, sign, 1)[:, None]
    bound = 2 * (M * np.abs(th) * 2.0 ** -51 + 70 * 2.0 ** -52)
    if sign < 0:  # acos(x) near pi has an ulp of pi
        bound = bound + 2 * M * np.pi * 2.0 ** -52
    off = np.abs(got - want) / bound
    assert off.max() < 1
