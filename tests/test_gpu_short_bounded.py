"""Neighbours on both sides of the rule that evaluates the kernel without clamps
(group box at most half the cutoff, the group's radii within a factor 8): counts
bit for bit, densities against the oracle.  Density bound: the FP32 path's 1e-5."""
import numpy as np
import pytest

import oracle
from test_gpu_short import G, _run, ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_grp", [1, 32, 300])
@pytest.mark.parametrize("mode", [0, 1])
def test_group_boxes_around_half_the_cutoff(G, ctx, mode, n_grp):
    n = 3001
    rng = np.random.default_rng(n_grp)
    pos = rng.random((n, 3)) * 3.0 + 70.0  # off the origin
    mass = rng.uniform(0.5, 1.5, n)
    for r in (0.02, 0.15, 0.3, 0.6, 2.0, 7.0):
        h = r * rng.uniform(0.9, 1.1, n)
        h[::97] *= 0.05  # groups whose radii differ by more than the rule allows
        cnt, rho, _ = _run(G, ctx, pos, mass, h, mode, r_fixed=r, n_leaf=min(8, n_grp), n_grp=n_grp)
        cr, rr = oracle.neighbors(pos, mass, h, mode, r_fixed=r)
        np.testing.assert_array_equal(cnt.astype(np.int64), cr)
        assert float(np.max(np.abs(rho - rr) / rr)) <= 1e-5
