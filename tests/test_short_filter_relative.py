"""The pair decision on coordinates relative to the group's centre (taken where
the group's box is at most half the cutoff), restated in numpy float32:
thresholds with 5u hb + 2 Eabs in Eabs' place never contradict the exact FP64
decision, with the i-particle anywhere in the box and the candidate around the
cutoff; moved 1000-fold towards c^2 they do.  CPU only."""
import numpy as np
import pytest

import test_short_filter as S
from test_short_filter import U, f32, fma32, neighbour_fp64, split


def _decide(xi, xj, c, c0, g, hb, L, shrink=1.0):
    gh = [split(g[a] - c0[a]) for a in range(3)]

    def coords(x):
        p = [split(x[a] - c0[a]) for a in range(3)]
        return [f32(f32(p[a][0] - gh[a][0]) + f32(p[a][1] - gh[a][1])) for a in range(3)]
    ci, cj = coords(xi), coords(xj)
    d = [f32(cj[a] - ci[a]) for a in range(3)]
    r2 = fma32(d[0], d[0], fma32(d[1], d[1], f32(d[2] * d[2])))
    Eabs = fma32(f32(5.0) * U, hb, f32(2.0) * f32(1e-13) * f32(L))
    lo, hi = S.thresholds(c, float(Eabs) / 1e-13, shrink)
    return 1 if r2 < lo else 0 if r2 > hi else -1


def _cases(rng, count):
    for _ in range(count):
        L = 10.0 ** rng.uniform(-3, 3)
        c0 = rng.uniform(-0.5, 0.5, 3) * L
        c = L * 10.0 ** rng.uniform(-6, -1)
        half = rng.uniform(0.0, 0.5, 3) * c * rng.choice([1.0, 1e-3])
        g = c0 + rng.uniform(-0.5, 0.5, 3) * L
        xi = g + half * rng.uniform(-1.0, 1.0, 3)
        u = rng.normal(size=3)
        u /= np.linalg.norm(u)
        rel = rng.choice([-1.0, 1.0]) * 10.0 ** rng.uniform(-9, -1)
        yield L, c0, xi, xi + u * c * (1.0 + rel), c, g, f32(half.max() * (1.0 + 1e-6)), rel


@pytest.mark.parametrize("seed", [1, 2])
def test_relative_decision_never_contradicts_fp64(seed):
    decided = inside = far = 0
    for L, c0, xi, xj, c, g, hb, rel in _cases(np.random.default_rng(seed), 6000):
        got = _decide(xi, xj, c, c0, g, hb, L)
        if got < 0:
            inside += 1
            far += abs(rel) > 1e-5 and c > 1e-6 * L
        else:
            decided += 1
            assert bool(got) == neighbour_fp64(xi, xj, c), (L, c, rel)
    # (a band of 32u + 15u and more about c^2: 1e-5 of c covers it)
    assert far == 0 and decided > 0 and inside > 0


def test_relative_decision_with_shrunk_bound_contradicts_fp64():
    wrong = 0
    for L, c0, xi, xj, c, g, hb, rel in _cases(np.random.default_rng(3), 20000):
        got = _decide(xi, xj, c, c0, g, hb, L, 1e-3)
        wrong += got >= 0 and bool(got) != neighbour_fp64(xi, xj, c)
    assert wrong > 0
