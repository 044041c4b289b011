"""Order of the interaction lists: every group's superparticles come before
its opened leaves (the force kernel stages them apart), also where a list
outgrows its pool chunk, is all leaves (theta = 0) or is a single leaf, and
the FP32 forces on such lists agree with the oracle's.  Force bound: the
FP32 path's 1e-5."""
import numpy as np
import pytest

import ics
import oracle

pytestmark = pytest.mark.gpu

LEAF = np.uint32(0x80000000)


@pytest.fixture(scope="module")
def G():
    from paper_1601_03138_gb300 import build as B
    B.build()
    import paper_1601_03138_gb300 as G
    return G


@pytest.mark.parametrize("n,theta,n_leaf,n_grp,quad", [
    (3, 0.5, 8, 64, False),        # one leaf, no superparticle
    (4000, 0.0, 4, 64, False),     # all leaves
    (5000, 0.6, 8, 128, True),     # chunks of superparticles and leaf batches
    (30011, 0.3, 1, 32, True),     # one particle a leaf: several leaf batches
    (70001, 0.0, 1, 512, False),   # a list beyond one pool chunk, all leaves
])
def test_superparticles_precede_leaves(G, n, theta, n_leaf, n_grp, quad):
    pos, vel, mass, eps = ics.make("plummer", n, 900 + n, 0.05)
    with G.Context(0) as ctx:
        ps = G.ParticleSystem(ctx, n)
        tree = G.Tree(ctx, theta=theta, n_leaf=n_leaf, n_grp=n_grp, quad=quad)
        try:
            ps.set(pos, vel, mass, eps)
            tree.calc_force_all_and_write_back(ps)
            ng = len(tree.groups()["first"])
            g1 = min(ng, 200)
            offs, ent = tree.lists(0, g1)
            for g in range(g1):
                leaf = (ent[offs[g]:offs[g + 1]] & LEAF) != 0
                assert np.all(np.diff(leaf.astype(np.int8)) >= 0)
            if n > 65536:
                assert np.diff(offs).max() > 65536
                rows = np.arange(0, n, 997)
                ar, pr = oracle.direct(pos, mass, eps, rows)
            else:
                rows = np.arange(n)
                ar, pr, _ = oracle.Tree(pos, mass, eps, theta=theta, n_leaf=n_leaf, n_grp=n_grp, quad=quad).force()
            _, _, acc, pot = ps.get()
            err = np.linalg.norm(acc[rows] - ar, axis=1) / np.linalg.norm(ar, axis=1)
            assert float(np.sqrt(np.mean(err ** 2))) <= 1e-5
            assert float(np.sqrt(np.mean((pot[rows] / pr - 1) ** 2))) <= 1e-5
        finally:
            tree.close()
            ps.close()
