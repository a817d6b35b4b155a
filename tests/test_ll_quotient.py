"""The u16 remap's quotient by a constant (two residual corrections of a product
with the rounded reciprocal), restated in exact rationals: the correctly rounded
a / b; and the level pair that can hold a gray in its band."""

import random
from fractions import Fraction

import numpy as np


def rnd(x: Fraction) -> np.float32:
    """x rounded to f32, half to even (normal range)."""
    if x == 0:
        return np.float32(0)
    f = np.float32(float(x))
    best = min((abs(Fraction(float(c)) - x), int(c.view(np.uint32)) & 1, i, c)
               for i, c in enumerate((f, np.nextafter(f, np.float32(-np.inf)), np.nextafter(f, np.float32(np.inf)))))
    return best[3]


def q(x):
    return Fraction(float(x))


def div_by(a, b, rb):
    v = rnd(q(a) * q(rb))
    for _ in range(2):
        r = rnd(q(a) - q(v) * q(b))
        v = rnd(q(v) + q(r) * q(rb))
    return v


def test_quotient_is_correctly_rounded():
    rng = random.Random(1)
    sigmas = [0.1, 0.142, 0.05, 1 / 3, 1.0, 0.0625, 2.0 ** -20, 0.9999999, 1.0000001, 3e-4]
    sigmas += [rng.uniform(1e-3, 1.0) for _ in range(6)]
    for s in sigmas:
        b = np.float32(s)
        rb = rnd(1 / q(b))
        for _ in range(300):
            a = np.float32(rng.choice([rng.random(), rng.random() * s, 2.0 ** rng.uniform(-34, 1)]))
            assert div_by(a, b, rb) == rnd(q(a) / q(b)), (a, b)
        assert div_by(np.float32(0), b, rb) == 0


def test_bands_lie_in_the_two_levels_around_gray():
    """sigma as large as the streaming remap admits; grays at and next to every
    level and midpoint."""
    sigma = np.float32(1 / 7 - 6e-7)
    gk = [np.float32(k) / np.float32(7) for k in range(8)]
    grays = {np.float32(k / 14) for k in range(-2, 17)}
    for g in list(grays):
        up = dn = g
        for _ in range(6):
            up, dn = np.nextafter(up, np.float32(9)), np.nextafter(dn, np.float32(-9))
            grays |= {up, dn}
    for g in grays:
        k0 = min(max(int(np.floor(np.float32(g * np.float32(7)))), 0), 6)
        for k in range(8):
            if abs(np.float32(g - gk[k])) <= sigma:
                assert k in (k0, k0 + 1), (g, k)
