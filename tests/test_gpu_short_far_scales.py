"""Neighbour counts of sets whose lengths are below or above what FP32 holds: exact,
through the FP64 sequence."""
import numpy as np
import pytest

import oracle
from test_gpu_short import G, _run, ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [0, 1, 2, 3])
@pytest.mark.parametrize("scale", [1e-60, 1e-46, 1e-40, 1e-33, 1e-27, 1e22, 1e30, 1e40, 1e50, 1e60])
def test_counts_beyond_fp32(G, ctx, scale, mode):
    n = 400
    pos = np.random.default_rng(2).random((n, 3)) * scale
    for f in (0.05, 0.2):
        h = np.full(n, f * scale)
        cnt, _, _ = _run(G, ctx, pos, np.ones(n), h, mode, r_fixed=f * scale)
        cr, _ = oracle.neighbors(pos, np.ones(n), h, mode, r_fixed=f * scale)
        np.testing.assert_array_equal(cnt.astype(np.int64), cr)
