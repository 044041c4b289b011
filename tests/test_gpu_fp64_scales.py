"""The FP64 pipeline at the ends of its range: lengths scaled by a power of two
leave accelerations and potentials equal but for their own powers, for monopole
and quadrupole superparticles.  FP32 has neither the coordinates (2^216 is 1e65)
nor their squares.  Bound: the reciprocal root's and the sums' roundings, 1e-13."""
import numpy as np
import pytest

import ics

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_1601_03138_gb300 import build as B
    B.build()
    import paper_1601_03138_gb300 as G
    return G


def _force(G, ctx, pos, mass, eps, quad):
    n = len(pos)
    ps, tree = G.ParticleSystem(ctx, n), G.Tree(ctx, theta=0.6, n_leaf=8, n_grp=64, quad=quad, fp64=True)
    try:
        ps.set(pos, np.zeros_like(pos), mass, eps)
        tree.calc_force_all_and_write_back(ps)
        _, _, acc, pot = ps.get()
        return acc, pot, tree.stats()["interactions_spj"]
    finally:
        tree.close()
        ps.close()


@pytest.mark.parametrize("quad", [False, True])
@pytest.mark.parametrize("k", [-300, -216, -100, 100, 216, 300])
def test_forces_scale_with_lengths(G, k, quad):
    pos, _, mass, eps = ics.make("plummer", 3000, 5, 0.02)
    with G.Context(0) as ctx:
        a0, p0, spj = _force(G, ctx, pos, mass, eps, quad)
        a1, p1, spj1 = _force(G, ctx, np.ldexp(pos, k), mass, np.ldexp(eps, k), quad)
    assert spj == spj1 > 0
    err = np.linalg.norm(np.ldexp(a1, 2 * k) - a0, axis=1) / np.linalg.norm(a0, axis=1)
    assert float(err.max()) <= 1e-13
    assert float(np.max(np.abs(np.ldexp(p1, k) / p0 - 1))) <= 1e-13
