"""Scratch that handles keep for their next call (records of a large device-side
read, device copies of a neighbour search's host arrays) does not stand in the
way of an allocation: one that finds no room gives it back first, and the calls
after it work as before."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
N = (1 << 21) + 3


def free_bytes():
    rt = ctypes.CDLL("libcudart.so.13")
    a, b = ctypes.c_size_t(), ctypes.c_size_t()
    assert rt.cudaMemGetInfo(ctypes.byref(a), ctypes.byref(b)) == 0
    return a.value


def test_a_failed_allocation_gives_scratch_back():
    torch = pytest.importorskip("torch")
    from paper_1601_03138_gb300 import build as B
    B.build()
    import paper_1601_03138_gb300 as G
    pos = torch.rand(N, 3, dtype=torch.float64, device="cuda")
    one = torch.ones(N, dtype=torch.float64, device="cuda")
    zero3 = torch.zeros_like(pos)
    acc, pot = torch.empty_like(pos), torch.empty_like(one)
    out, vel = torch.empty_like(pos), torch.empty_like(pos)
    r = 0.5 * N ** (-1.0 / 3.0)
    torch.cuda.synchronize()
    with G.Context(0) as ctx:
        ps, tree = G.ParticleSystem(ctx, N), G.Tree(ctx, theta=0.8, n_leaf=8, n_grp=128)
        try:
            ps.set(pos, zero3, one, 0.01 * one)
            tree.calc_force_all_and_write_back(ps)
            f0 = free_bytes()
            G.fdps_psys_get(ctx.h, ps.h, None, None, acc, pot)  # forces alone: 32 bytes a particle beside 4 of the order
            f1 = free_bytes()
            assert 36 * N <= f0 - f1 <= 36 * N + (8 << 20)
            G.fdps_psys_get(ctx.h, ps.h, out, vel, acc, pot)
            cnt, rho, _ = tree.neighbors(ps, 0, r_fixed=r)
            assert torch.equal(out, pos)
            ref = (acc.clone(), pot.clone())
            held = free_bytes()
            with pytest.raises(G.FdpsError):  # 160 bytes for each of 2^31 particles: more than the GPU has
                G.ParticleSystem(ctx, 0x7FFFFFFF)
            assert free_bytes() - held >= 64 * N + 12 * N
            acc.zero_()
            pot.zero_()
            out.zero_()
            torch.cuda.synchronize()
            cnt2, rho2, _ = tree.neighbors(ps, 0, r_fixed=r)
            np.testing.assert_array_equal(cnt, cnt2)
            np.testing.assert_array_equal(rho, rho2)
            G.fdps_psys_get(ctx.h, ps.h, out, vel, acc, pot)
            assert torch.equal(out, pos) and torch.equal(acc, ref[0]) and torch.equal(pot, ref[1])
        finally:
            tree.close()
            ps.close()


def test_handles_may_outlive_the_giving_back_and_close_in_any_order():
    from paper_1601_03138_gb300 import build as B
    B.build()
    import paper_1601_03138_gb300 as G
    pos = np.random.default_rng(1).random((500, 3))
    with G.Context(0) as ctx:
        systems = [G.ParticleSystem(ctx, 500) for _ in range(4)]
        trees = [G.Tree(ctx, theta=0.5, n_leaf=8, n_grp=64) for _ in range(4)]
        for i in (2, 0, 3, 1):
            systems[i].set(pos, np.zeros_like(pos), np.ones(500), np.full(500, 0.01))
            trees[i].calc_force_all_and_write_back(systems[i])
            trees[i].close()
            systems[i].close()
        with pytest.raises(G.FdpsError):
            G.ParticleSystem(ctx, 0x7FFFFFFF)
