"""The FP64 force kernel on both sides of the rule that gives groups of few
particles one CTA instead of a cluster, and, in an ensemble of mostly tiny
systems, one CTA with a group of several rounds: against the oracle.  Bound: as
for the cluster, 1e-12, of a potential and the self term m / eps that was
subtracted from it (a lone particle's potential is nothing but that rounding)."""
import numpy as np
import pytest

import ics
import oracle
from test_gpu_fp64_split import G, RMS_FP64  # noqa: F401

pytestmark = pytest.mark.gpu


def _check(acc, pot, ref, self_term):
    ar, pr, _ = ref.force()
    err = np.linalg.norm(acc - ar, axis=1) / np.maximum(np.linalg.norm(ar, axis=1), 1e-300)
    assert float(np.sqrt(np.mean(err ** 2))) <= RMS_FP64
    assert float(np.max(np.abs(pot - pr))) <= RMS_FP64 * float(np.max(np.abs(pr)) + self_term)


@pytest.mark.parametrize("quad", [False, True])
@pytest.mark.parametrize("n,n_grp,n_leaf", [(300, 1, 1), (1001, 8, 8), (1001, 9, 8), (16383, 16, 8), (16384, 16, 8),
                                            (131071, 32, 8), (131072, 32, 8)])
def test_both_sides_of_the_rule(G, n, n_grp, n_leaf, quad):
    pos, vel, mass, eps = ics.make("plummer", n, 17, 0.05)
    with G.Context(0) as ctx:
        ps = G.ParticleSystem(ctx, n)
        tree = G.Tree(ctx, theta=0.8, n_leaf=n_leaf, n_grp=n_grp, quad=quad, fp64=True)
        try:
            ps.set(pos, vel, mass, eps)
            tree.calc_force_all_and_write_back(ps)
            _, _, acc, pot = ps.get()
            _check(acc, pot, oracle.Tree(pos, mass, eps, theta=0.8, n_leaf=n_leaf, n_grp=n_grp, quad=quad),
                   float(np.max(mass / eps)))
        finally:
            tree.close()
            ps.close()


@pytest.mark.parametrize("quad", [False, True])
def test_tiny_systems_beside_a_large_group(G, quad):
    sizes = [1, 2, 3] * 150 + [1500, 8, 65, 257]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n = int(off[-1])
    assert n // len(sizes) <= 8
    pos = np.random.default_rng(3).normal(size=(n, 3))
    mass, eps = np.full(n, 1.0 / n), np.full(n, 0.05)
    with G.Context(0) as ctx:
        ps = G.ParticleSystem(ctx, n)
        tree = G.Tree(ctx, theta=0.8, n_leaf=8, n_grp=4096, quad=quad, fp64=True)
        try:
            ps.set_systems(off)
            ps.set(pos, np.zeros_like(pos), mass, eps)
            tree.calc_force_all_and_write_back(ps)
            _, _, acc, pot = ps.get()
            for a, b in list(zip(off[:-1], off[1:]))[-10:]:
                _check(acc[a:b], pot[a:b], oracle.Tree(pos[a:b], mass[a:b], eps[a:b], theta=0.8, n_leaf=8, n_grp=4096,
                                                       quad=quad), float(np.max(mass / eps)))
        finally:
            tree.close()
            ps.close()
