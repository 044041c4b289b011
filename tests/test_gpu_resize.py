"""A tree that outgrows its first node arrays: tight knots of n_leaf + 1
particles far apart, each at the end of a chain of some fifteen cells.  The
build cuts the tree at the level that does not fit (its last nodes then have
no children), the kernels after it run on the cut tree, and the call is
repeated with larger arrays: nodes and forces equal the oracle's, for the
moments of small systems, of large ones and of an ensemble.

Force bound: the FP32 path's 1e-5.  It needs a softening well above the
knots: coordinates relative to a group's centre are rounded to 2^-24 of its
size (0.1), 6e-9 or 6e-4 of a separation inside a knot (1e-5), and with eps =
1e-3 a knot's own force, m dx / eps^3 = 0.3 a particle, would carry that error
into the sum.  With eps = 0.05 it is 2e-6 a particle, of forces of order 1."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_1601_03138_gb300 import build as B
    B.build()
    import paper_1601_03138_gb300 as G
    return G


def knots(k, rng):
    centre = rng.random((k, 1, 3))
    return (centre + 1e-5 * rng.random((k, 17, 3))).reshape(-1, 3)


@pytest.mark.parametrize("quad", [False, True])
@pytest.mark.parametrize("k", [2000, 6000])
def test_node_arrays_grow(G, k, quad):
    rng = np.random.default_rng(k)
    pos = knots(k, rng)
    n = len(pos)
    mass, eps = np.full(n, 1.0 / n), np.full(n, 0.05)
    ref = oracle.Tree(pos, mass, eps, theta=0.7, n_leaf=16, n_grp=64, quad=quad)
    assert ref.n_nodes > n // 2 + 1024  # more than the first allocation
    with G.Context(0) as ctx:
        ps = G.ParticleSystem(ctx, n)
        tree = G.Tree(ctx, theta=0.7, n_leaf=16, n_grp=64, quad=quad)
        try:
            ps.set(pos, np.zeros_like(pos), mass, eps)
            tree.calc_force_all_and_write_back(ps)
            st = tree.stats()
            assert st["retries"] > 0 and st["n_nodes"] == ref.n_nodes
            keys, perm = tree.keys(n)
            kr, pr = ref.keys()
            np.testing.assert_array_equal(keys, kr)
            np.testing.assert_array_equal(perm, pr)
            _, _, acc, pot = ps.get()
            ar, phr, _ = ref.force()
            err = np.linalg.norm(acc - ar, axis=1) / np.linalg.norm(ar, axis=1)
            assert float(np.sqrt(np.mean(err ** 2))) <= 1e-5
            assert float(np.sqrt(np.mean((pot / phr - 1) ** 2))) <= 1e-5
        finally:
            tree.close()
            ps.close()


def test_ensemble_node_arrays_grow(G):
    rng = np.random.default_rng(7)
    sizes = [1500 * 17, 300, 2500 * 17]
    pos = np.concatenate([knots(1500, rng), rng.random((300, 3)), knots(2500, rng)])
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n = len(pos)
    mass, eps = np.full(n, 1.0 / n), np.full(n, 0.05)
    with G.Context(0) as ctx:
        ps = G.ParticleSystem(ctx, n)
        tree = G.Tree(ctx, theta=0.7, n_leaf=16, n_grp=64)
        try:
            ps.set_systems(off)
            ps.set(pos, np.zeros_like(pos), mass, eps)
            tree.calc_force_all_and_write_back(ps)
            assert tree.stats()["retries"] > 0
            _, _, acc, _ = ps.get()
            for a, b in zip(off[:-1], off[1:]):
                ar, _, _ = oracle.Tree(pos[a:b], mass[a:b], eps[a:b], theta=0.7, n_leaf=16, n_grp=64).force()
                err = np.linalg.norm(acc[a:b] - ar, axis=1) / np.linalg.norm(ar, axis=1)
                assert float(np.sqrt(np.mean(err ** 2))) <= 1e-5
        finally:
            tree.close()
            ps.close()
