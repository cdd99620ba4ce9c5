"""Evolution and commutator orders of several FP32 vectors that start at an address that is
a multiple of 8 bytes and not of 16: the same values as from an aligned buffer (each
element's arithmetic is the same)."""
import pytest

import gqt_synth as S

torch = pytest.importorskip("torch")
g = pytest.importorskip("paper_1705_01387_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R", [2, 4, 8])
@pytest.mark.parametrize("lattice", ["honeycomb", "haldane"])
def test_vectors_on_8_byte_addresses(R, lattice):
    if lattice == "honeycomb":
        lat, K = S.honeycomb(13, 11, -1.0, 1.0, seed=1), 3
    else:
        lat, K = S.haldane(8, 9, -1.0, 0.15, 1.1, 0.0, 1.0, seed=1), 9
    ham = g.gqt_build_hamiltonian(lat, S.energy_scale_rule(K, -1.0, 1.0), g.GQT_FP32_ACC64)
    psi = torch.from_numpy(S.random_phase(lat.n, R, seed=2)).to(torch.complex64)
    got = []
    for shift in (0, 1):
        buf = [torch.zeros(lat.n * R + 1, dtype=torch.complex64, device="cuda")[shift:shift + lat.n * R].view(lat.n, R)
               for _ in range(3)]
        assert buf[0].data_ptr() % 16 == 8 * shift
        for b in buf[:2]:
            b.copy_(psi)
        g.gqt_evolve(ham, buf[0], R, 0.7, 1)
        g.gqt_commutator_evolve(ham, buf[1], buf[2], R, 0.7)
        got.append((buf[0].cpu(), buf[2].cpu()))
    for x, y in zip(*got):
        assert torch.equal(x, y)
