"""Direct sums at the row counts where the split of rows over blocks, threads
and slices of the j range changes, with ragged j tiles, against the oracle's
FP64 sum: the result of a row does not depend on how many are asked for beyond
the order of its sum.  A softening whose square is no normal FP32 number (or
vanishes in FP32) takes the variant without the bare reciprocal root; the
particle's own term is skipped there too.

Bounds, of the sum of a row's terms by magnitude: a pair term is FP32 with a
reciprocal root of 2 ulp, cubed, some ten roundings of 2^-24 or 1e-6, and the
FP32 sum over a tile of 256 j-particles rounds by at most 256 * 2^-24 =
1.5e-5 of it; tiles are added with compensation.  Both are worst cases of
roundings that are independent: RMS 1e-6."""
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


def _terms(pos, mass, eps, i):
    d = pos - pos[i]
    r2 = np.sum(d * d, axis=1)
    with np.errstate(divide="ignore"):
        w = mass / (r2 + eps[i] ** 2) ** 1.5
    w[i] = 0.0
    return float(np.sum(w * np.sqrt(r2)))


def _check(G, pos, mass, eps, row_sets):
    with G.Context(0) as ctx:
        ps = G.ParticleSystem(ctx, len(pos))
        try:
            ps.set(pos, np.zeros_like(pos), mass, eps)
            for rows in row_sets:
                acc, pot = ps.direct(rows)
                ar, pr = oracle.direct(pos, mass, eps, rows)
                terms = np.array([_terms(pos, mass, eps, i) for i in rows])
                ea = np.linalg.norm(acc - ar, axis=1) / terms
                ep = np.abs(pot / pr - 1.0)
                assert ea.max() <= 1.6e-5 and ep.max() <= 1.6e-5  # (a NaN fails)
                assert np.sqrt(np.mean(ea ** 2)) <= 1e-6 and np.sqrt(np.mean(ep ** 2)) <= 1e-6
        finally:
            ps.close()


@pytest.mark.parametrize("n", [257, 1500, 20011])
def test_row_counts(G, n):
    pos, _, mass, eps = ics.make("plummer", n, 5, 1.0 / 64.0)
    rng = np.random.default_rng(n)
    counts = [1, 2, 15, 16, 17, 31, 32, 33, 64, 65, 128, 129, 256, 257, 511, 513, 1025]
    _check(G, pos, mass, eps, [rng.choice(n, k, replace=False) for k in counts if k <= n])


@pytest.mark.parametrize("e", [1e-18, 1e-20, 1e-30])
def test_softening_below_fp32(G, e):
    n = 700
    rng = np.random.default_rng(3)
    pos = rng.random((n, 3))
    eps = np.full(n, 0.01)
    eps[::7] = e
    _check(G, pos, np.full(n, 1.0 / n), eps, [np.arange(40), np.arange(n)])
