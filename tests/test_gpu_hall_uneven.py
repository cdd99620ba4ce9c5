"""FP64 Hall moments of vectors whose magnitude is very uneven: one site far above the rest,
so that the large elements of a row of v_a T_m r meet small ones of v_b T_n r.  Each
entry of Lambda is within the rounding of FP64 multiply-adds of the sum of its own
products (not of the rows' largest elements, which is what scaled integer slices keep).
Reference: extended precision; bound: 30 roundings for up to three orders of the chains,
2 x 512 for the products and sums of a split, one for each split, times the sum of the
products of the chains run on absolute values."""
import numpy as np
import pytest

import gqt_synth as S

torch = pytest.importorskip("torch")
g = pytest.importorskip("paper_1705_01387_gb300")

pytestmark = pytest.mark.gpu


def _chains(lat, dE, r, M, dtype):
    """P = T_m v_x r and B = v_y T_n r; with dtype real, on absolute values."""
    f = np.abs if dtype == np.longdouble else (lambda a: a)
    real = np.longdouble
    h = f((lat.hop / dE).astype(np.clongdouble)) if dtype != np.longdouble else np.abs(lat.hop / dE).astype(real)
    d = f((lat.onsite / dE).astype(real))[:, None]
    dx, dy = f(lat.dx.astype(real)), f(lat.dy.astype(real))
    minus = 1 if dtype == np.longdouble else -1
    unit = 1 if dtype == np.longdouble else 1j

    def mul(m, x):
        return sum(m[:, k:k + 1] * x[lat.nb_idx[:, k]] for k in range(lat.max_nb))

    def chain(x):
        out = [x]
        if M > 1:
            out.append(mul(h, x) + d * x)
        while len(out) < M:
            out.append(2 * (mul(h, out[-1]) + d * out[-1]) + minus * out[-2])
        return out

    x = f(r.astype(np.clongdouble)) if dtype != np.longdouble else np.abs(r).astype(real)
    return chain(unit * mul(dx * h, x)), [unit * mul(dy * h, t) for t in chain(x)]


@pytest.mark.parametrize("M", [1, 3])
@pytest.mark.parametrize("shape,R,sites", [((37, 40), 1, 1), ((11, 9), 2, 1), ((64, 61), 1, 3)])
@pytest.mark.parametrize("small", [1e-3, 1e-7, 1e-30])
def test_entries_of_disjoint_large_parts(M, shape, R, sites, small):
    lat = S.square(*shape, -1.0, 1.0, seed=M)
    dE = 5.0
    r = small * np.sqrt(lat.n) * S.random_phase(lat.n, R, seed=M)
    r[lat.n // 3:lat.n // 3 + 5 * sites:5] = 1.0
    ham = g.gqt_build_hamiltonian(lat, dE)
    lam = torch.empty((M, M), dtype=torch.complex128, device="cuda")
    g.gqt_kb_moments(ham, torch.from_numpy(r).cuda(), R, M, 0, 1, lam)
    got = lam.cpu().numpy()
    scale = np.longdouble(lat.n) / R
    P, B = _chains(lat, dE, r, M, np.clongdouble)
    Pa, Ba = _chains(lat, dE, r, M, np.longdouble)
    splits = lat.n * R // 512 + 1
    for m in range(M):
        for n in range(M):
            want = scale * (P[m].conj() * B[n]).sum()
            bound = (30 + 1024 + splits) * 2.0 ** -53 * scale * (Pa[m] * Ba[n]).sum()
            assert abs(got[m, n] - want) <= bound


def test_even_and_uneven_rows_side_by_side():
    """Rows of the first orders are uneven, later ones less so: tiles of both kinds, the same
    bits each time, and within the 64-bit path's bound of the largest entry."""
    lat = S.square(40, 37, -1.0, 1.0, seed=1)
    dE, M = 5.0, 150
    r = 1e-4 * np.sqrt(lat.n) * S.random_phase(lat.n, 1, seed=2)
    r[777] = 1.0
    ham = g.gqt_build_hamiltonian(lat, dE)
    lam = [torch.empty((M, M), dtype=torch.complex128, device="cuda") for _ in range(2)]
    for x in lam:
        g.gqt_kb_moments(ham, torch.from_numpy(r).cuda(), 1, M, 0, 1, x)
    assert torch.equal(lam[0], lam[1])
    P, B = _chains(lat, dE, r, M, np.clongdouble)
    want = lat.n * (np.array(P)[:, :, 0].conj() @ np.array(B)[:, :, 0].T)
    assert np.abs(lam[0].cpu().numpy() - want).max() <= 1e-13 * np.abs(want).max()


def test_rows_without_a_scale():
    """Zeros, denormals, an infinity and a NaN: as the multiply-adds have them."""
    lat = S.square(9, 8, -1.0, 1.0, seed=1)
    ham = g.gqt_build_hamiltonian(lat, 5.0)
    lam = torch.empty((4, 4), dtype=torch.complex128, device="cuda")
    r = torch.from_numpy(S.random_phase(lat.n, 1, seed=2)).cuda()
    for value in (0.0, 1e-310):
        g.gqt_kb_moments(ham, value * r, 1, 4, 0, 1, lam)
        assert not bool(lam.abs().max())
    for value in (float("inf"), float("nan")):
        bad = r.clone()
        bad[5] = value
        g.gqt_kb_moments(ham, bad, 1, 4, 0, 1, lam)
        assert not bool(torch.isfinite(lam.real).any())
