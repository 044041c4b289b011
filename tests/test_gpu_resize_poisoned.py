"""A first call whose tree outgrows its node arrays, on arrays whose memory held
hostile records: 0xFB in every byte reads as an internal node with 31 children
at an id far outside the tree.  Nothing may follow such a record: the cut tree's
nodes all get their own, and the walk is left out until the build has been
repeated.  The result equals that of a tree whose arrays fit at once."""
import ctypes

import numpy as np
import pytest

from test_gpu_resize import G, knots  # noqa: F401

pytestmark = pytest.mark.gpu


def poison(n, n_leaf):
    """Device memory of the sizes the node arrays will have, filled and freed."""
    rt = ctypes.CDLL("libcudart.so.13")
    cap = min(8 * n // n_leaf, 3 * n) + 1024 + 1
    held = []
    for _ in range(24):
        for size in (4 * cap, 8 * cap, 16 * cap, 32 * cap, 48 * cap):
            p = ctypes.c_void_p()
            assert rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(size)) == 0
            assert rt.cudaMemset(p, 0xFB, ctypes.c_size_t(size)) == 0
            held.append(p)
    assert rt.cudaDeviceSynchronize() == 0
    for p in held:
        assert rt.cudaFree(p) == 0


@pytest.mark.parametrize("quad", [False, True])
@pytest.mark.parametrize("k", [100, 1500, 2000, 6000])  # both sides of 2^15 and of 2^16 particles
def test_hostile_memory_behind_a_cut_tree(G, k, quad):
    pos = knots(k, np.random.default_rng(k))
    n = len(pos)
    mass, eps = np.full(n, 1.0 / n), np.full(n, 0.05)
    with G.Context(0) as ctx:
        ps = G.ParticleSystem(ctx, n)
        poison(n, 16)
        tree = G.Tree(ctx, theta=0.7, n_leaf=16, n_grp=64, quad=quad)
        try:
            ps.set(pos, np.zeros_like(pos), mass, eps)
            tree.calc_force_all_and_write_back(ps)
            assert tree.stats()["retries"] > 0 or k == 100
            first = ps.get()
            ps.set(pos, np.zeros_like(pos), mass, eps)
            tree.calc_force_all_and_write_back(ps)  # now the arrays fit
            for a, b in zip(first, ps.get()):
                np.testing.assert_array_equal(a, b)
        finally:
            tree.close()
            ps.close()
