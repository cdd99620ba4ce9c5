"""Scratch of the calls without a handle: the same bits from several threads and streams at
once, at sizes below and above what the pool keeps (128 MB), and no more than that kept
afterwards."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
g = pytest.importorskip("paper_1705_01387_gb300")

pytestmark = pytest.mark.gpu


def _call(kind, seed):
    rng = np.random.default_rng(seed)
    if kind == "kb":
        M, NE = 60, 300
        lam = torch.from_numpy(rng.standard_normal((M, M)) + 1j * rng.standard_normal((M, M))).cuda()
        E = torch.linspace(-0.9, 0.9, NE, dtype=torch.float64, device="cuda")
        out = torch.empty_like(E)
        return lambda: g.gqt_kubo_bastin(lam, E, 1.0, 10.0, out), out
    rows, M, NE = {"small": (3, 50, 70), "product": (40, 300, 500), "large": (500, 4000, 9000)}[kind]
    mu = torch.from_numpy(rng.standard_normal((rows, M))).cuda()
    E = torch.linspace(-0.9, 0.9, NE, dtype=torch.float64, device="cuda")
    out = torch.empty((rows, NE), dtype=torch.float64, device="cuda")
    return lambda: g.gqt_kpm_reconstruct(mu, E, 1.0, 1.0, out, 1), out


def test_threads_and_streams():
    bad = []

    def work(kind, seed):
        with torch.cuda.stream(torch.cuda.Stream()):
            run, out = _call(kind, seed)
            run()
            want = out.clone()
            for _ in range(12):
                out.zero_()
                run()
                if not torch.equal(out, want):
                    bad.append(kind)

    threads = [threading.Thread(target=work, args=(k, q)) for q, k in enumerate(("kb", "small", "product", "large", "small"))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


def test_what_is_kept_is_bounded():
    run, out = _call("large", 9)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    for _ in range(3):
        run()
    torch.cuda.synchronize()
    assert before - torch.cuda.mem_get_info()[0] <= (128 << 20) + (64 << 20)  # the pool's 128 MB, and granularity
