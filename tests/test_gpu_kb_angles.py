"""Angles of the Kubo-Bastin series at thousands of moments: one moment Lambda_mm, whose
integrand is 2 cos m th (x cos m th + m sin th sin m th) / sin^4 th, at the angle th = acos x
that the GPU computes, in extended precision.  Bound: 40 roundings of the angles k th =
2 m th and 20 of everything else, times m (unrounded angles: k th 2^-53 is a thousand
roundings at m = 4000)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
g = pytest.importorskip("paper_1705_01387_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [300, 2000, 4000, 8192])
def test_one_moment_at_large_angles(M):
    dE, area, m = 3.7, 2.0, M - 1
    lam = torch.zeros((M, M), dtype=torch.complex128, device="cuda")
    lam[m, m] = 1.0
    rng = np.random.default_rng(M)
    for _ in range(25):
        E = np.sort(rng.uniform(-0.7, 0.7, 2)) * dE
        d = torch.from_numpy(E).cuda()
        x = d * torch.full_like(d, 1.0 / dE)  # the kernel's product, and its angle
        th = torch.acos(x).cpu().numpy().astype(np.longdouble)
        x = x.cpu().numpy().astype(np.longdouble)
        s = np.sqrt((1 - x) * (1 + x))
        F = 4 * 2 * np.cos(m * th) * (x * np.cos(m * th) + m * s * np.sin(m * th)) / s ** 4
        sig = torch.empty(2, dtype=torch.float64, device="cuda")
        g.gqt_kubo_bastin(lam, d, dE, area, sig, kernel=1)
        ref = 2 / area * 0.5 * (x[1] - x[0]) * (F[0] + F[1])
        size = 2 / area * 0.5 * (x[1] - x[0]) * (4 * 2 * (1 + m) / s ** 4).sum()
        assert abs(sig.cpu().numpy()[1] - ref) <= 60 * 2.0 ** -53 * size
