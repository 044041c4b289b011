"""Neighbour counts of sets so small or large that the square of the grid
spacing, 1/H^2 or r^2 leave or come near the ends of FP32: exact."""
import numpy as np
import pytest

import oracle
from test_gpu_short import G, _run, ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [0, 1, 2, 3])
@pytest.mark.parametrize("scale", [1e-16, 1e-13, 1e12, 1e16, 3e17])
def test_counts_at_extreme_scales(G, ctx, scale, mode):
    n = 400
    pos = np.random.default_rng(2).random((n, 3)) * scale
    h = np.full(n, 0.2 * scale)
    cnt, _, _ = _run(G, ctx, pos, np.ones(n), h, mode, r_fixed=0.2 * scale)
    cr, _ = oracle.neighbors(pos, np.ones(n), h, mode, r_fixed=0.2 * scale)
    np.testing.assert_array_equal(cnt.astype(np.int64), cr)
