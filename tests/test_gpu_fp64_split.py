"""The FP64 force kernel's split of a group over a cluster of CTAs: group
sizes around the edges of its i-slots (a warp, a CTA, the most a CTA holds,
several rounds) and lists shorter than a cluster and longer than a chunk,
against the oracle.  Bound: at most about 3,000 terms a particle, each term
and partial sum rounded to 2^-53 of values no larger than a few times the
result, so 1e-12 leaves a factor of a few."""
import numpy as np
import pytest

import ics
import oracle

pytestmark = pytest.mark.gpu

RMS_FP64 = 1e-12


@pytest.fixture(scope="module")
def G():
    from paper_1601_03138_gb300 import build as B
    B.build()
    import paper_1601_03138_gb300 as G
    return G


@pytest.mark.parametrize("quad", [False, True])
@pytest.mark.parametrize("n,n_grp", [(2, 8), (7, 8), (9, 16), (31, 4096), (33, 4096), (65, 4096), (127, 4096),
                                     (129, 4096), (385, 4096), (511, 4096), (513, 4096), (1100, 4096),
                                     (2500, 96)])
def test_group_sizes(G, n, n_grp, quad):
    pos, vel, mass, eps = ics.make("plummer", n, 400 + n, 0.05)
    mass = mass * np.random.default_rng(n).uniform(0.5, 1.5, n)
    with G.Context(0) as ctx:
        ps = G.ParticleSystem(ctx, n)
        tree = G.Tree(ctx, theta=0.8, n_leaf=4, n_grp=n_grp, quad=quad, fp64=True)
        try:
            ps.set(pos, vel, mass, eps)
            tree.calc_force_all_and_write_back(ps)
            _, _, acc, pot = ps.get()
            ref = oracle.Tree(pos, mass, eps, theta=0.8, n_leaf=4, n_grp=n_grp, quad=quad)
            ar, pr, _ = ref.force()
            err = np.linalg.norm(acc - ar, axis=1) / np.linalg.norm(ar, axis=1)
            assert float(np.sqrt(np.mean(err ** 2))) <= RMS_FP64
            assert float(np.sqrt(np.mean((pot / pr - 1) ** 2))) <= RMS_FP64
        finally:
            tree.close()
            ps.close()
