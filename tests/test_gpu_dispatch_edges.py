"""Set sizes on both sides of the lines where the tree kernels change their
split: 2^15 particles (build tiles, i-groups, walk, monopole force) and 2^16
(moments by one cluster or by the whole grid), and the device-side outputs by
records from 2^21 on.  Structure bit for bit and forces within 1e-5 RMS of the
oracle's; a captured run equals its steps bit for bit."""
import numpy as np
import pytest

import ics
import oracle
from test_gpu_parity import G, check_structure, ctx, rms_rel, run_gpu  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("quad", [False, True])
@pytest.mark.parametrize("n", [32767, 32768, 32769, 65536, 65537])
def test_split_lines(G, ctx, n, quad):
    pos, vel, mass, eps = ics.make("hernquist", n, 17, 0.01)
    ps, tree = run_gpu(G, ctx, pos, vel, mass, eps, 0.6, 8, 64, quad)
    try:
        ref = oracle.Tree(pos, mass, eps, theta=0.6, n_leaf=8, n_grp=64, quad=quad)
        sample = np.random.default_rng(n).choice(ref.n_groups, 60, replace=False)
        check_structure(G, tree, ref, n, sample)
        _, _, acc, pot = ps.get()
        acc_r, pot_r, tot = ref.force()
        assert rms_rel(acc, acc_r) <= 1e-5 and rms_rel(pot, pot_r) <= 1e-5
        st = tree.stats()
        assert st["interactions_epj"] + st["interactions_spj"] == tot[2] and st["interactions_spj"] == tot[3]
    finally:
        tree.close()
        ps.close()


@pytest.mark.parametrize("n", [32768, 65537])
def test_captured_run_equals_steps(G, ctx, n):
    pos, vel, mass, eps = ics.make("plummer", n, 23, 0.02)
    out = []
    for captured in (True, False):
        ps = G.ParticleSystem(ctx, n)
        tree = G.Tree(ctx, theta=0.6, n_leaf=8, n_grp=64)
        try:
            ps.set(pos, vel, mass, eps)
            tree.calc_force_all_and_write_back(ps)
            if captured:
                tree.run(ps, 1e-3, 4)
            else:
                for _ in range(4):
                    tree.step(ps, 1e-3)
            out.append(ps.get_state())
        finally:
            tree.close()
            ps.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("n", [(1 << 21) - 1, 1 << 21, (1 << 21) + 77])
def test_device_outputs_by_records(G, ctx, n):
    """Every combination of outputs, on the device, equals the host's."""
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(5)
    pos = rng.random((n, 3))
    ps = G.ParticleSystem(ctx, n)
    tree = G.Tree(ctx, theta=1.0, n_leaf=16, n_grp=256)
    try:
        ps.set(pos, rng.normal(size=(n, 3)), np.full(n, 1.0 / n), np.full(n, 0.01))
        tree.calc_force_all_and_write_back(ps)
        host = ps.get()
        assert np.array_equal(host[0], pos)
        for want in (0b1111, 0b0011, 0b1100, 0b0111, 0b0101, 0b1000):
            dev = [torch.full((n, 3) if k < 3 else (n,), np.nan, dtype=torch.float64, device="cuda")
                   if want >> k & 1 else None for k in range(4)]
            G.fdps_psys_get(ctx.h, ps.h, *dev)
            torch.cuda.synchronize()
            for h, d in zip(host, dev):
                if d is not None:
                    np.testing.assert_array_equal(d.cpu().numpy(), h)
    finally:
        tree.close()
        ps.close()
