"""The walk's first FP32 test, from centres rounded to FP32 and a box kept as
half-widths about its centre, restated in numpy float32: its thresholds (and
those of the hi/lo pairs, on the same half-widths) never contradict the exact
FP64 opening test, also where the set lies far from the origin (the box's two
sides then differ by the rounding of its centre) and for massless cells
(centre of mass at the origin); with the bounds shrunk they do.  CPU only."""
import numpy as np
import pytest

from test_walk_filter import _cases, f32, fma32, open_fp64, round_down, round_up, split, U

E0_HI, E0_PAIR = f32(6.2e-8), f32(1e-13)


def group(box, c0):
    cc = [(box[a] + box[3 + a]) * 0.5 for a in range(3)]
    lo = [round_down(box[a] - cc[a]) for a in range(3)]
    hi = [round_up(box[3 + a] - cc[a]) for a in range(3)]
    h = [max(-lo[a], hi[a]) for a in range(3)]
    asym = max(abs(f32(lo[a] + hi[a])) for a in range(3))
    return [split(cc[a] - c0[a]) for a in range(3)], h, asym


def thresholds(L, level, theta2, h, asym, e0rel, shrink):
    th2, Lf, hb = f32(theta2), f32(L), max(h)
    e0 = f32(e0rel * Lf + asym)
    mc1 = f32(1.01) * th2 * f32(25.0) * U
    mc2 = f32(1.01) * th2 * f32(7.0) * e0
    mc3 = f32(1.01) * th2 * f32(4.0) * e0 * e0
    ell = f32(np.ldexp(Lf, -level))
    l2 = ell * ell
    D0 = f32(np.sqrt(l2 / th2))
    Mb = D0 + f32(2.0) * hb
    Mo = f32(16.0) * U * l2 + fma32(fma32(mc1, Mb, mc2), Mb, mc3)
    lo = (l2 - Mo * f32(shrink)) / th2 * (f32(1.0) - f32(8.0) * U)
    coef = th2 - (f32(8.0) * U * th2 + f32(2.0) * mc1 + mc2 / (f32(2.0) * D0)) * f32(shrink)
    rhs = (l2 * (f32(1.0) + f32(8.0) * U * f32(shrink))
           + (f32(8.0) * mc1 * hb * hb + mc2 * (f32(0.5) * D0 + f32(2.0) * hb) + mc3) * f32(shrink))
    return lo, rhs * (f32(1.0) + f32(16.0) * U) / coef if coef > 0 else f32(np.inf)


def decide(L, level, theta2, com, box, c0, pair, fused, shrink=1.0):
    gc, h, asym = group(box, c0)
    fc = [split(com[a] - c0[a]) for a in range(3)]
    if pair:
        d = [(fc[a][0] - gc[a][0]) + (fc[a][1] - gc[a][1]) for a in range(3)]
    else:
        d = [fc[a][0] - gc[a][0] for a in range(3)]
    t = [max(abs(d[a]) - h[a], f32(0.0)) for a in range(3)]
    d2 = fma32(t[2], t[2], fma32(t[1], t[1], t[0] * t[0])) if fused else t[0] * t[0] + t[1] * t[1] + t[2] * t[2]
    lo, hi = thresholds(L, level, theta2, h, asym, E0_PAIR if pair else E0_HI, shrink)
    return 1 if d2 < lo else 0 if d2 > hi else -1


def cases(rng, count, shift):
    for L, level, theta, theta2, c0, box, com, rel, half, dist in _cases(rng, count):
        # the set moved by up to 10^5 root boxes: positions, box and centre in
        # FP64 at that distance; cells stay inside the root box
        off = rng.uniform(-1.0, 1.0, 3) * shift * L
        c = c0 + off
        lim = 0.5 * L
        b = np.clip(np.concatenate([box[:3] + off, box[3:] + off]), np.tile(c - lim, 2), np.tile(c + lim, 2))
        m = np.clip(com + off, c - lim, c + lim)
        yield L, level, theta2, c, b, m, rel, half, dist


@pytest.mark.parametrize("pair", [False, True])
@pytest.mark.parametrize("shift", [0.0, 1e2, 1e5])
def test_thresholds_never_contradict_the_fp64_test(pair, shift):
    rng = np.random.default_rng(20280 + 2 * int(shift) + pair)
    decided = 0
    for k, (L, level, theta2, c0, box, com, rel, half, dist) in enumerate(cases(rng, 4000, shift)):
        if k % 50 == 0:
            com = np.zeros(3)  # a cell without mass
        got = decide(L, level, theta2, com, box, c0, pair, bool(k & 1))
        if got >= 0:
            decided += 1
            assert bool(got) == open_fp64(L, level, theta2, com, box), (L, level, theta2, rel)
    # cells of levels 0 to 21 alike: those near 2^-24 L stay undecided
    assert decided > 1000


@pytest.mark.parametrize("pair,shrink", [(False, 1e-2), (True, 1e-3)])
def test_shrunk_thresholds_contradict_the_fp64_test(pair, shrink):
    rng = np.random.default_rng(20290 + pair)
    wrong = 0
    for L, level, theta2, c0, box, com, rel, half, dist in cases(rng, 6000, 0.0):
        got = decide(L, level, theta2, com, box, c0, pair, False, shrink)
        if got >= 0 and bool(got) != open_fp64(L, level, theta2, com, box):
            wrong += 1
    assert wrong > 0
