"""The one-cluster sort of small sets and the tile-and-merge sort of the
allocation-free entry point, at the edges of a thread's, a tile's and a
CTA's share, with many equal keys (ties keep the input order): keys and
permutation bit for bit against the oracle's."""
import numpy as np
import pytest

import ics
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_1601_03138_gb300 import build as B
    B.build()
    import paper_1601_03138_gb300 as G
    return G


def _set(n, ties):
    rng = np.random.default_rng(n)
    pos = rng.normal(size=(n, 3)) + 3.0
    if ties:
        pos = np.round(pos * 2.0) / 2.0  # a few hundred distinct keys
    return np.ascontiguousarray(pos), np.full(n, 1.0 / n), np.full(n, 0.1)


@pytest.mark.parametrize("ties", [False, True])
@pytest.mark.parametrize("n", [1, 2, 255, 257, 7, 9, 2041, 2048, 2049, 4099, 8192, 16383, 16384, 16385, 20481, 65537, 262144])
def test_noalloc_sort(G, n, ties):
    torch = pytest.importorskip("torch")
    pos, mass, eps = _set(n, ties)
    keys_ref, perm_ref = oracle.Tree(pos, mass, eps, theta=0.5, n_leaf=8, n_grp=64).keys()
    # coordinate arrays on odd 8-byte boundaries as well
    xyz = [torch.tensor(np.concatenate([[0.0], pos[:, a]]), device="cuda")[1:] for a in range(3)]
    keys = torch.empty(n, dtype=torch.int64, device="cuda")
    perm = torch.empty(n, dtype=torch.int32, device="cuda")
    for _ in range(2):
        keys.fill_(-1)
        perm.fill_(-1)
        G.fdps_morton_sort_noalloc(*xyz, n, keys, perm, torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(perm.cpu().numpy().view(np.uint32), perm_ref)
        np.testing.assert_array_equal(keys.cpu().numpy().view(np.uint64), np.asarray(keys_ref)[np.asarray(perm_ref)])


@pytest.mark.parametrize("n", [1, 3, 8, 9, 256, 2048, 2049, 16384, 16385])
def test_pipeline_sort_over_steps(G, n):
    pos, mass, eps = _set(n, n % 2 == 0)
    vel = np.random.default_rng(n + 1).normal(size=(n, 3))
    with G.Context(0) as ctx:
        ps = G.ParticleSystem(ctx, n)
        tree = G.Tree(ctx, theta=0.6, n_leaf=8, n_grp=64)
        try:
            ps.set(pos, vel, mass, eps)
            tree.calc_force_all_and_write_back(ps)
            keys, perm = tree.keys(n)
            ref = oracle.Tree(pos, mass, eps, theta=0.6, n_leaf=8, n_grp=64)
            kr, pr = ref.keys()
            np.testing.assert_array_equal(keys, kr)
            np.testing.assert_array_equal(perm, pr)
            lo, L, s = tree.box()
            assert np.array_equal(lo, pos.min(0)) and L == (np.max(np.ptp(pos, axis=0)) or 1.0) and s == 2.0 ** 21 / L
            # the order of the last sort, moved a little, sorted again
            tree.step(ps, 1e-3)
            moved = ps.get_state()[0][np.asarray(perm)]
            keys, perm2 = tree.keys(n)
            kr, pr = oracle.Tree(np.ascontiguousarray(moved), mass, eps, theta=0.6, n_leaf=8, n_grp=64).keys()
            np.testing.assert_array_equal(keys, kr)
            np.testing.assert_array_equal(perm2, pr)
        finally:
            tree.close()
            ps.close()
