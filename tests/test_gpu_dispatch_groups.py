"""Group sizes and leaf sizes on both sides of the lines where the walk, the i-group
pass, the moments and the monopole force change their kernel by the estimated
number of groups or nodes: structure bit for bit and forces within 1e-5 RMS of the
oracle's."""
import numpy as np
import pytest

import ics
import oracle
from test_gpu_parity import G, check_structure, ctx, rms_rel, run_gpu  # noqa: F401

pytestmark = pytest.mark.gpu


def _check(G, ctx, n, n_grp, n_leaf, quad=False):
    pos, vel, mass, eps = ics.make("plummer", n, 29, 0.02)
    ps, tree = run_gpu(G, ctx, pos, vel, mass, eps, 0.7, n_leaf, n_grp, quad)
    try:
        ref = oracle.Tree(pos, mass, eps, theta=0.7, n_leaf=n_leaf, n_grp=n_grp, quad=quad)
        sample = np.random.default_rng(n).choice(ref.n_groups, min(40, ref.n_groups), replace=False)
        check_structure(G, tree, ref, n, sample)
        _, _, acc, pot = ps.get()
        acc_r, pot_r, tot = ref.force()
        assert rms_rel(acc, acc_r) <= 1e-5 and rms_rel(pot, pot_r) <= 1e-5
        st = tree.stats()
        assert st["interactions_epj"] + st["interactions_spj"] == tot[2] and st["interactions_spj"] == tot[3]
    finally:
        tree.close()
        ps.close()


@pytest.mark.parametrize("n,n_grp,n_leaf", [(2048, 1, 1), (2049, 1, 1), (16384, 32, 8), (16385, 32, 8), (32768, 64, 8),
                                            (32768, 8, 8), (32768, 1, 1)])
def test_walk_lines(G, ctx, n, n_grp, n_leaf):
    _check(G, ctx, n, n_grp, n_leaf)


@pytest.mark.parametrize("n,n_grp,n_leaf", [(4096, 1, 1), (4097, 1, 1), (16384, 16, 8), (16385, 16, 8)])
def test_group_pass_lines(G, ctx, n, n_grp, n_leaf):
    _check(G, ctx, n, n_grp, n_leaf)


@pytest.mark.parametrize("quad", [False, True])
@pytest.mark.parametrize("n,n_leaf", [(19115, 1), (19116, 1), (32768, 4), (32769, 4), (65536, 8), (65536, 16)])
def test_moments_lines(G, ctx, n, n_leaf, quad):
    _check(G, ctx, n, 64, n_leaf, quad)


@pytest.mark.parametrize("n,n_grp", [(3328, 16), (3329, 16), (53248, 64), (53249, 64), (100000, 1024), (212992, 128),
                                     (212993, 128)])
def test_monopole_force_lines(G, ctx, n, n_grp):
    _check(G, ctx, n, n_grp, 8)
