"""The scratch pool of the calls without a handle gives its memory back with a device's last
handle (in a process of its own, so that no other handle is alive)."""
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytest.importorskip("paper_1705_01387_gb300")

pytestmark = pytest.mark.gpu

PROGRAM = """
import torch
import paper_1705_01387_gb300 as g

def reconstruct():
    mu = torch.ones((60, 3000), dtype=torch.float64, device="cuda")
    E = torch.linspace(-0.9, 0.9, 20000, dtype=torch.float64, device="cuda")
    g.gqt_kpm_reconstruct(mu, E, 1.0, 1.0, torch.empty((60, 20000), dtype=torch.float64, device="cuda"))
    torch.cuda.synchronize()
    torch.cuda.empty_cache()

def handle():
    return g.gqt_build_hamiltonian(kind=g.GQT_LATTICE_CHAIN, L1=100, t=-1.0, energy_scale=2.1)

h = [handle(), handle()]
free = [torch.cuda.mem_get_info()[0]]
reconstruct()
reconstruct()
free.append(torch.cuda.mem_get_info()[0])
h.pop()
free.append(torch.cuda.mem_get_info()[0])
h.pop()
free.append(torch.cuda.mem_get_info()[0])
reconstruct()
print(*[free[0] - f >> 20 for f in free])
"""


def test_the_last_handle_empties_the_pool():
    r = subprocess.run([sys.executable, "-c", PROGRAM], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    _, used, one_left, none_left = map(int, r.stdout.split())
    assert used >= 32 and one_left >= used - 8  # the pool keeps memory, also while a handle is alive
    assert none_left <= used - 32
