"""Moment rows of several FP32 vectors that start at an address that is a multiple of 8 bytes
and not of 16: the same bits as from an aligned buffer, on every neighbour count of the
multi-vector kernels (2, 3, 4, 6 slots, with and without prefetch), on the blocked
honeycomb rows, and through the calls that hand over the caller's vectors (density of
states, VAC and MSD rows with their evolution)."""
import numpy as np
import pytest

import gqt_synth as S

torch = pytest.importorskip("torch")
g = pytest.importorskip("paper_1705_01387_gb300")

pytestmark = pytest.mark.gpu

LATTICES = {"chain": dict(kind=g.GQT_LATTICE_CHAIN, L1=333), "square": dict(kind=g.GQT_LATTICE_SQUARE, L1=19, L2=23),
            "honeycomb": dict(kind=g.GQT_LATTICE_HONEYCOMB, L1=13, L2=11),
            "blocked": dict(kind=g.GQT_LATTICE_HONEYCOMB, L1=64, L2=9), "cubic": dict(kind=g.GQT_LATTICE_CUBIC, L1=8)}
SLOTS = {"chain": 2, "square": 4, "honeycomb": 3, "blocked": 3, "cubic": 6}


@pytest.mark.parametrize("R", [2, 4, 8, 32])
@pytest.mark.parametrize("lattice", sorted(LATTICES))
def test_rows_of_vectors_on_8_byte_addresses(lattice, R):
    ham = g.gqt_build_hamiltonian(**LATTICES[lattice], t=-1.0, W=1.0, seed=3,
                                  energy_scale=S.energy_scale_rule(SLOTS[lattice], -1.0, 1.0),
                                  precision=g.GQT_FP32_ACC64)
    x, y = (torch.from_numpy(S.random_phase(ham.n, R, seed=q)).to(torch.complex64) for q in (1, 2))
    M, dts = 13, [0.6, 0.3]
    got = []
    for shifts in ((0, 0), (1, 1), (1, 0), (0, 1)):
        def vec(v, shift):
            b = torch.zeros(ham.n * R + 1, dtype=torch.complex64, device="cuda")[shift:shift + ham.n * R].view(ham.n, R)
            assert b.data_ptr() % 16 == 8 * shift
            return b.copy_(v)
        rows = []
        mu = np.empty((1, R, M))
        g.gqt_dos_moments(ham, vec(x, shifts[0]), R, M, mu)
        rows.append(mu.tobytes())
        for call in (g.gqt_vac_moments, g.gqt_msd_moments):
            mu, a, b = np.empty((2, 1, R, M)), vec(x, shifts[0]), vec(y, shifts[1])
            call(ham, a, b, R, dts, M, mu)
            rows += [mu.tobytes(), a.cpu().numpy().tobytes(), b.cpu().numpy().tobytes()]
        got.append(rows)
    for rows in got[1:]:
        assert rows == got[0]
