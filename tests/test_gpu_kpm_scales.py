"""Reconstruction of rows without a scale at which they could be sliced, among rows that have
one (more than 8 rows, the sliced product): an infinity, a NaN, nothing but denormals,
zeros; and rows whose largest moment stands anywhere.  Infinities and NaN as the sum has
them; the rest within 1e-12 of the row's sum of |moments|, the bound of the other rows
(and a few denormal units)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
g = pytest.importorskip("paper_1705_01387_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,M,NE", [(9, 40, 7), (17, 600, 300), (130, 33, 65)])
def test_rows_without_a_scale(rows, M, NE):
    rng = np.random.default_rng(rows)
    mu = rng.standard_normal((rows, M)) / (1 + np.arange(M))
    mu[1, M // 2] = np.inf
    mu[3, 0] = -np.inf
    mu[rows - 1, M - 1] = np.nan
    mu[4] *= 1e-310
    mu[5] = 0.0
    mu[6] = 1e-9 * rng.standard_normal(M)
    mu[6, M - 1] = 1.0
    dE = 3.7
    E = np.linspace(-0.99, 0.98, NE) * dE
    out = torch.empty((rows, NE), dtype=torch.float64, device="cuda")
    g.gqt_kpm_reconstruct(torch.from_numpy(mu).cuda(), torch.from_numpy(E).cuda(), dE, 1.0, out, 1)
    got = out.cpu().numpy()
    n = np.arange(M)
    x = E / dE
    scale = 2 / (np.pi * dE * np.sqrt((1 - x) * (1 + x)))
    with np.errstate(invalid="ignore"):
        tab = np.cos(n[:, None] * np.arccos(x)) * np.where(n == 0, 1.0, 2.0)[:, None]
        ref = np.array([(r[:, None] * tab).sum(0) for r in mu]) * scale
    for r in range(rows):
        if r in (1, 3, rows - 1):
            assert np.array_equal(got[r], ref[r], equal_nan=True)
        else:
            assert np.all(np.abs(got[r] - ref[r]) <= 1e-12 * scale * 2 * np.abs(mu[r]).sum() + 1e-322)
    assert not got[5].any() and got[4].any()
