"""Neighbour counts where the squares of cutoffs and separations are subnormal FP32
numbers (spacing 1.4e-45, far above the relative bound of the pair decision):
exact, through the FP64 sequence."""
import numpy as np
import pytest

import oracle
from test_gpu_short import G, _run, ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [0, 1, 2, 3])
@pytest.mark.parametrize("scale", [1e-22, 3e-22, 1e-21, 3e-21, 1e-20, 1e-19, 4e-17])
def test_counts_with_subnormal_squares(G, ctx, scale, mode):
    n = 400
    pos = np.random.default_rng(2).random((n, 3)) * scale
    for f in (0.05, 0.2):
        h = np.full(n, f * scale)
        cnt, _, _ = _run(G, ctx, pos, np.ones(n), h, mode, r_fixed=f * scale)
        cr, _ = oracle.neighbors(pos, np.ones(n), h, mode, r_fixed=f * scale)
        np.testing.assert_array_equal(cnt.astype(np.int64), cr)
