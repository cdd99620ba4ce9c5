"""Reconstruction of moment rows: the pass for up to 8 rows and the sliced product with the
Chebyshev table for more, at the edges of their tiles (128 rows, 64 energies, 16 orders)
and blocks, energies at and outside the band edges, and rows that hold a NaN.  Reference:
the sum in 64-bit numpy, cos(n acos x); bound: 1e-12 of the row's sum of |moments|, the
rounding of n acos x at n = 2000 (2000 pi 2^-53 = 7e-13) among it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
g = pytest.importorskip("paper_1705_01387_gb300")

pytestmark = pytest.mark.gpu


def _reference(mu, E, dE, n_over_omega, kernel):
    M = mu.shape[1]
    n = np.arange(M)
    a = np.pi / (M + 1)
    gn = ((1 - n / (M + 1)) * np.cos(n * a) + np.sin(n * a) / np.tan(a) / (M + 1)) if kernel == 0 else np.ones(M)
    w = gn * np.where(n == 0, 1.0, 2.0)
    x = np.array(E) / dE
    with np.errstate(invalid="ignore"):
        scale = np.where(np.abs(x) < 1, 2 * n_over_omega / (np.pi * dE * np.sqrt((1 - x) * (1 + x))), np.nan)
        tab = np.cos(n[:, None] * np.arccos(x)[None, :])
    bound = scale * np.abs(mu * w).sum(1)[:, None]
    return (mu * w) @ np.nan_to_num(tab) * scale, bound


@pytest.mark.parametrize("kernel", [0, 1])
@pytest.mark.parametrize("rows,M,NE", [(1, 1, 1), (1, 33, 5), (2, 500, 65), (3, 513, 64), (8, 2000, 100), (9, 1, 1),
                                       (9, 16, 64), (9, 17, 65), (128, 100, 63), (129, 129, 130), (300, 2000, 257)])
def test_rows(rows, M, NE, kernel):
    rng = np.random.default_rng(rows + M + NE)
    mu = rng.standard_normal((rows, M)) / (1 + np.arange(M))
    dE, noo = 3.7, 0.8
    E = np.linspace(-dE * 0.9999, dE * 0.9999, NE) if NE > 1 else np.array([0.3])
    out = torch.empty((rows, NE), dtype=torch.float64, device="cuda")
    g.gqt_kpm_reconstruct(torch.from_numpy(mu).cuda(), torch.from_numpy(E).cuda(), dE, noo, out, kernel)
    ref, bound = _reference(mu, E, dE, noo, kernel)
    assert np.all(np.abs(out.cpu().numpy() - ref) <= 1e-12 * bound)


@pytest.mark.parametrize("rows", [2, 20])
def test_band_edges_and_nan(rows):
    rng = np.random.default_rng(rows)
    mu = rng.standard_normal((rows, 70))
    mu[0] *= 1e-200
    mu[1, 69] = np.nan
    dE = 2.0
    E = np.array([-2.5, -2.0, -1.0, 0.0, 1.999999, 2.0, np.nan])
    out = torch.empty((rows, 7), dtype=torch.float64, device="cuda")
    g.gqt_kpm_reconstruct(torch.from_numpy(mu).cuda(), torch.from_numpy(E).cuda(), dE, 1.0, out, 1)
    got = out.cpu().numpy()
    assert np.all(np.isnan(got[1])) and np.all(np.isnan(got[:, [0, 1, 5, 6]]))
    ref, bound = _reference(np.delete(mu, 1, 0), E, dE, 1.0, 1)
    inside = slice(2, 5)
    assert np.all(np.abs(np.delete(got, 1, 0)[:, inside] - ref[:, inside]) <= 1e-12 * bound[:, inside])


@pytest.mark.parametrize("rows,NE", [(9, 1_300_000), (4000, 9000)])
def test_energies_in_blocks(rows, NE):
    """More energies than one block holds (M = 16: 1.2 million, 2^25 results)."""
    mu = np.zeros((rows, 16))
    n = np.arange(rows) % 16
    mu[np.arange(rows), n] = 1.0
    E = torch.linspace(-0.99, 0.99, NE, dtype=torch.float64, device="cuda")
    out = torch.empty((rows, NE), dtype=torch.float64, device="cuda")
    g.gqt_kpm_reconstruct(torch.from_numpy(mu).cuda(), E, 1.0, 1.0, out, 1)
    n = torch.from_numpy(n.astype(float)).cuda()[:, None]
    ref = torch.cos(n * torch.acos(E)) * 2 / (np.pi * torch.sqrt(1 - E * E)) * torch.where(n == 0, 1.0, 2.0)
    assert float(((out - ref).abs() / ref.abs().amax(0)).max()) < 1e-12


def test_rows_in_blocks():
    """More rows than one block of slices holds (M = 4000: 4736), one and two blocks of energies."""
    rows, M = 4750, 4000
    mu = torch.zeros((rows, M), dtype=torch.float64, device="cuda")
    n = torch.arange(rows, device="cuda") % M
    mu[torch.arange(rows, device="cuda"), n] = 1.0
    for NE in (70, 7200):
        E = torch.linspace(-0.99, 0.99, NE, dtype=torch.float64, device="cuda")
        out = torch.empty((rows, NE), dtype=torch.float64, device="cuda")
        g.gqt_kpm_reconstruct(mu, E, 1.0, 1.0, out, 1)
        ref = torch.cos(n[:, None] * torch.acos(E)) * 2 / (np.pi * torch.sqrt(1 - E * E)) * torch.where(n == 0, 1.0, 2.0)[:, None]
        assert float(((out - ref).abs() / ref.abs().amax(0)).max()) < 2e-12  # n acos x rounds at 4000 pi 2^-53
