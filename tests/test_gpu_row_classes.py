"""Rows named by their class of neighbour offsets: lattices whose sites are relabelled at
random, with as many classes as a handle keeps (4096 sites, each its own class) and with
more (no classes, the index array is read), against the same lattice in its own order.
Every site's arithmetic is the same in both, so moments differ by the order of their sums
only: 1e-13 of mu_0 in FP64, 1e-6 in FP32 storage (compensated FP32 dots)."""
import dataclasses

import numpy as np
import pytest

import gqt_synth as S

torch = pytest.importorskip("torch")
g = pytest.importorskip("paper_1705_01387_gb300")

pytestmark = pytest.mark.gpu

LATTICES = {
    2: (lambda W: S.chain(4096, -1.0, W, seed=1), lambda W: S.chain(4099, -1.0, W, seed=1)),
    3: (lambda W: S.honeycomb(64, 32, -1.0, W, seed=1), lambda W: S.honeycomb(61, 34, -1.0, W, seed=1)),
    4: (lambda W: S.square(64, 64, -1.0, W, seed=1), lambda W: S.square(63, 66, -1.0, W, seed=1)),
    6: (lambda W: S.cubic(16, -1.0, W, seed=1), lambda W: S.cubic(17, -1.0, W, seed=1)),
}


def _relabelled(lat, seed):
    p = np.random.default_rng(seed).permutation(lat.n)  # site i becomes p[i]
    q = np.argsort(p)
    return dataclasses.replace(lat, nb_count=lat.nb_count[q], nb_idx=p[lat.nb_idx[q]].astype(np.int32), hop=lat.hop[q],
                               onsite=lat.onsite[q], dx=lat.dx[q], dy=None), q


def _rows(lat, dE, prec, arith, pair, vecs, M=41):
    ham = g.gqt_build_hamiltonian(lat, dE, prec)
    g.gqt_set_cluster(ham, False)
    g.gqt_set_temporal_blocking(ham, False)
    g.gqt_set_vac_pair(ham, pair)
    if prec == g.GQT_FP64:
        g.gqt_set_fp64_arith(ham, arith)
    R = vecs[0].shape[1]
    ct = torch.complex128 if prec == g.GQT_FP64 else torch.complex64
    a, b, p, px = (torch.from_numpy(np.ascontiguousarray(v)).to(ct).cuda() for v in vecs)
    dos, vac, msd = np.empty((R, 1, M)), np.empty((R, 1, 2, M)), np.empty((R, 1, 2, M))
    g.gqt_dos_moments(ham, a, R, M, dos)
    g.gqt_vac_moments(ham, a, b, R, [0.4, 0.3], M, vac)
    g.gqt_msd_moments(ham, p, px, R, [0.4, 0.3], M, msd)
    return [x.ravel() for x in (dos, vac, msd)]


@pytest.mark.parametrize("K", list(LATTICES))
@pytest.mark.parametrize("classes", [True, False])
@pytest.mark.parametrize("prec,arith,pair,R", [("GQT_FP64", 1, True, 1), ("GQT_FP64", 0, True, 1), ("GQT_FP64", 0, False, 1),
                                               ("GQT_FP64", 1, True, 2), ("GQT_FP32_ACC64", 1, True, 1),
                                               ("GQT_FP32_ACC64", 1, False, 1), ("GQT_FP32_ACC64", 1, True, 4)])
def test_relabelled_lattice(K, classes, prec, arith, pair, R):
    lat = LATTICES[K][0 if classes else 1](1.0)
    if not pair:
        lat = S.with_random_bond_phases(lat, 3)
    dE = S.energy_scale_rule(K, -1.0, 1.0)
    other, q = _relabelled(lat, K)
    vecs = [S.random_phase(lat.n, R, seed=s) for s in (1, 2, 3, 4)]
    x = _rows(lat, dE, getattr(g, prec), arith, pair, vecs)
    y = _rows(other, dE, getattr(g, prec), arith, pair, [v[q] for v in vecs])
    tol = 1e-13 if prec == "GQT_FP64" else 1e-6
    for u, v in zip(x, y):
        assert np.all(np.abs(u - v) < tol * max(1.0, np.abs(u).max()))


def test_common_hopping_of_fp32_handles_follows_updates():
    """One common hopping, another one, hoppings of each bond, and one again: a handle
    that is updated gives the same moments as a handle built anew."""
    lat = S.square(40, 31, -1.0, 1.0, seed=5)
    dE, M = S.energy_scale_rule(4, -1.3, 1.0), 33
    r = torch.from_numpy(S.random_phase(lat.n, 1, seed=1)).to(torch.complex64).cuda()
    ham = g.gqt_build_hamiltonian(lat, dE, g.GQT_FP32_ACC64)
    g.gqt_set_cluster(ham, False)
    lo, hi = np.minimum(np.arange(lat.n)[:, None], lat.nb_idx), np.maximum(np.arange(lat.n)[:, None], lat.nb_idx)
    each = -1.0 + 0.1 * np.cos(lo + 3.0 * hi)
    for hop in (np.full(lat.hop.shape, -1.0), np.full(lat.hop.shape, -0.7), each, np.full(lat.hop.shape, -1.2)):
        g.gqt_update_hamiltonian(ham, lat.onsite, hop)
        fresh = g.gqt_build_hamiltonian(dataclasses.replace(lat, hop=hop.astype(np.complex128)), dE, g.GQT_FP32_ACC64)
        g.gqt_set_cluster(fresh, False)
        mu = [np.empty((1, 1, M)), np.empty((1, 1, M))]
        for h, m in zip((ham, fresh), mu):
            for _ in range(2):  # the second call replays the captured graph
                g.gqt_dos_moments(h, r, 1, M, m)
        assert np.array_equal(mu[0], mu[1])


@pytest.mark.parametrize("what", ["regular", "too many in one range", "too many together"])
def test_classes_of_large_models(what):
    """Models whose rows are scanned in ranges by several threads (65536 sites and more):
    one whose classes agree across ranges, one range with more than 4096, and ranges with
    fewer each that have more together."""
    lat = S.square(331, 257, -1.0, 1.0, seed=3)
    n = lat.n
    p = np.arange(n)
    rng = np.random.default_rng(1)
    if what == "too many in one range":
        p[40000:48000] = rng.permutation(p[40000:48000])
    elif what == "too many together":
        for a in range(0, n - 3000, 10000):
            p[a:a + 700] = rng.permutation(p[a:a + 700])
    q = np.argsort(p)
    other = dataclasses.replace(lat, nb_count=lat.nb_count[q], nb_idx=p[lat.nb_idx[q]].astype(np.int32), hop=lat.hop[q],
                                onsite=lat.onsite[q], dx=lat.dx[q], dy=None)
    dE = S.energy_scale_rule(4, -1.0, 1.0)
    vecs = [S.random_phase(n, 1, seed=s) for s in (1, 2, 3, 4)]
    x = _rows(lat, dE, g.GQT_FP64, 1, True, vecs, M=11)
    y = _rows(other, dE, g.GQT_FP64, 1, True, [v[q] for v in vecs], M=11)
    for u, v in zip(x, y):
        assert np.all(np.abs(u - v) < 1e-13 * max(1.0, np.abs(u).max()))
