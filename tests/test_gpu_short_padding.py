"""Neighbour counts of tight clumps in a box up to 1e11 times their cutoffs, at an
offset that FP32 represents: a tile of candidates is padded to an even number,
and a displacement of a few cutoffs is far below half an ulp of the clump's
coordinates.  Odd and even sizes around the tile, all four cutoff types, group
boxes below and above the cutoff: counts bit for bit."""
import numpy as np
import pytest

import oracle
from test_gpu_short import G, _run, ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [0, 1, 2, 3])
@pytest.mark.parametrize("ratio", [1e-11, 1e-10, 3e-10, 1e-9, 1e-8, 1e-7, 1e-6])
def test_counts_of_tight_clumps(G, ctx, ratio, mode):
    rng = np.random.default_rng(int(-10 * np.log10(ratio)) + mode)
    corners = np.array([[x, y, z] for x in (0.0, 1.0) for y in (0.0, 1.0) for z in (0.0, 1.0)])
    for m in (3, 8, 33, 97, 131):
        for width in (0.2, 3.0):
            pos = np.concatenate([corners, 0.75 + width * ratio * rng.random((m, 3))])
            h = ratio * rng.uniform(0.9, 1.1, len(pos))
            cnt, _, info = _run(G, ctx, pos, np.ones(len(pos)), h, mode, r_fixed=ratio, n_leaf=8, n_grp=64)
            cr, _ = oracle.neighbors(pos, np.ones(len(pos)), h, mode, r_fixed=ratio)
            np.testing.assert_array_equal(cnt.astype(np.int64), cr)
            assert info[0] == int(np.sum(cr))
