"""The FP64 Hall contraction by exact integer slices on the tensor cores (mode 0 of
gqt_set_kb_contraction), at the edges of its tiles (128 rows, 64 columns), stages (16
contraction elements, 8 stages per emptying) and blocks (slices of at most 1 GiB),
against the same moments in 64-bit torch; rows of very different magnitude; and rows
that hold a NaN.  Bound: 1e-13 of the largest entry (64-bit chains of up to 300 orders,
the contraction itself being exact to 2^-53)."""
import math

import numpy as np
import pytest

import gqt_synth as S

torch = pytest.importorskip("torch")
g = pytest.importorskip("paper_1705_01387_gb300")

pytestmark = pytest.mark.gpu


def _reference(lat, dE, r, M):
    idx = torch.from_numpy(lat.nb_idx.astype(np.int64)).cuda()
    h = torch.from_numpy(lat.hop).cuda() / dE
    d = (torch.from_numpy(lat.onsite).cuda() / dE)[:, None]
    dx, dy = torch.from_numpy(lat.dx).cuda(), torch.from_numpy(lat.dy).cuda()

    def mul(m, x):
        return sum(m[:, k:k + 1] * x[idx[:, k]] for k in range(lat.max_nb))

    def chain(x):
        a, b = x, mul(h, x) + d * x
        yield a
        while True:
            yield b
            a, b = b, 2 * (mul(h, b) + d * b) - a

    P = torch.stack([t.reshape(-1) for _, t in zip(range(M), chain(1j * mul(dx * h, r)))])
    B = torch.stack([(1j * mul(dy * h, t)).reshape(-1) for _, t in zip(range(M), chain(r))])
    return (lat.n / r.shape[1]) * (P.conj() @ B.T)


def _moments(lat, dE, r, M):
    ham = g.gqt_build_hamiltonian(lat, dE)
    lam = torch.empty((M, M), dtype=torch.complex128, device="cuda")
    g.gqt_kb_moments(ham, r, r.shape[1], M, 0, 1, lam)
    return lam


def _off(x, y):
    return float((x - y).abs().max() / y.abs().max())


@pytest.mark.parametrize("M,L1,L2,R", [(1, 3, 3, 1), (15, 4, 4, 1), (64, 5, 5, 2), (65, 8, 8, 1), (127, 9, 7, 1),
                                       (128, 8, 16, 1), (129, 13, 11, 3), (200, 33, 17, 1), (300, 40, 41, 2)])
def test_tiles_and_stages(M, L1, L2, R):
    lat = S.haldane(L1, L2, -1.0, 0.15, 1.1, 0.1, 1.0, seed=M)
    dE = 1.05 * (3 + 0.9 + 0.1 + 0.5)
    r = torch.from_numpy(S.random_phase(lat.n, R, seed=M)).cuda()
    assert _off(_moments(lat, dE, r, M), _reference(lat, dE, r, M)) < 1e-13


def test_blocks_of_the_contraction():
    """More sites than one block of slices holds: 1170 chunks of 16 at M = 1024."""
    lat = S.haldane(100, 97, -1.0, 0.15, math.pi / 2, 0.0, 1.0, seed=3)
    dE = 1.05 * (3 + 0.9 + 0.5)
    r = torch.from_numpy(S.random_phase(lat.n, 1, seed=5)).cuda()
    assert lat.n > 1170 * 16
    assert _off(_moments(lat, dE, r, 1024), _reference(lat, dE, r, 1024)) < 1e-12  # 1024 orders


def test_rows_of_different_scale_and_nan():
    lat = S.haldane(9, 8, -1.0, 0.15, 1.1, 0.1, 1.0, seed=2)
    dE = 1.05 * (3 + 0.9 + 0.1 + 0.5)
    M = 40
    r = torch.from_numpy(S.random_phase(lat.n, 1, seed=2)).cuda()
    ref = _reference(lat, dE, r, M)
    for scale in (2.0 ** 200, 2.0 ** -300):  # powers of two change no digit
        assert _off(_moments(lat, dE, r * scale, M) / scale / scale, ref) < 1e-13
    few = torch.zeros_like(r)  # elements from 1 to 1e-30 in one row
    few[::7] = 1.0
    few[1::7] = 1e-30
    assert _off(_moments(lat, dE, few, M), _reference(lat, dE, few, M)) < 1e-13
    r[5] = float("nan")
    assert bool(torch.isnan(_moments(lat, dE, r, M).real).all())
