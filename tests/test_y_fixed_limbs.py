"""compute_Y's fixed point where U spans many powers of two (host walk, no GPU):
how a component is rounded, shifted and cut off, and what is left of Y."""
from fractions import Fraction

import numpy as np
import pytest

from paper_2011_12875_gb300 import inputs
from tests.test_tables_host import symmetric_u


@pytest.fixture(scope="module")
def snapmod():
    from paper_2011_12875_gb300 import build, snap
    build.build()
    snap.load()
    return snap


def test_one_component_of_any_size(snapmod):
    """2J = 0: Y = 3 beta U^2, one component, which is its atom's largest: held to
    2^-59 of the power of two above it down to 2^-150, in units of 2^-209 below."""
    rng = np.random.default_rng(5)
    beta = np.array([0.0, 0.8125])
    for e in list(range(-150, 400, 7)) + [-151, -160, -180, -205, -212, -400, -1060]:
        for sign in (1.0, -1.0):
            u = sign * np.ldexp(1.0 + rng.random(), e)
            y = snapmod.yi_host(0, beta, np.array([[u, 0.0]]), precision=0)[0, 0]
            # two factors and their product, the coefficient: each to its unit
            unit = max(Fraction(2) ** (e - 58), Fraction(2) ** -209)
            want, size = 3 * Fraction(beta[1]) * Fraction(u) ** 2, 3 * Fraction(beta[1]) * abs(Fraction(u))
            if e < -210:
                assert y == 0.0
            else:
                # (u + d)^2, |d| <= unit, and the product's own last place, 2 units of it
                err = 2 * size * unit + 3 * Fraction(beta[1]) * (unit * unit + 4 * unit * max(abs(Fraction(u)), Fraction(2) ** -150))
                assert abs(Fraction(float(y)) - want) <= err + abs(want) * Fraction(2) ** -52, e


def test_components_below_the_largest(snapmod):
    """2J = 1, beta of the component (1, 0, 1) alone: Y_1 = 2 beta U_0 U_1, so with
    U_0 = 1 each element of Y_1 shows how its own component was held: to nearest in
    units of 2^-58 (U_0 = 1 is below 2^1)."""
    names = [(t1, t2, t) for t1 in range(2) for t2 in range(t1 + 1) for t in range(t1 - t2, min(1, t1 + t2) + 1, 2) if t >= t1]
    beta = np.zeros(1 + len(names))
    beta[1 + names.index((1, 0, 1))] = 0.75
    at = [snapmod.half_index(1, 1, ma, 0) for ma in (0, 1)]
    one = np.zeros((snapmod.half_size(1), 2))
    one[0, 0] = one[at[0], 0] = 1.0
    c = snapmod.yi_host(1, beta, one, precision=1)[at[0], 0]
    assert c != 0.0
    rng = np.random.default_rng(9)
    cases = [np.ldexp(1.0 + rng.random(), -k) for k in range(1, 70)]
    # halves of the last place, the smallest one that counts, and below it
    cases += [2.0 ** -59, 1.5 * 2.0 ** -59, 0.99 * 2.0 ** -59, 2.0 ** -60, 5e-324, 2.0 ** -1022, 0.0]
    # U_0, c = 1.5 and the component are below 2, 2 and 2: the product is held in
    # units of 8 x 2^-58; half of one for its rounding, half for that of c U_0 and
    # the products of the low limbs
    assert c == 1.5
    tol = Fraction(8, 2 ** 58)
    for x in cases:
        for sx in (x, -x):
            u = np.zeros((snapmod.half_size(1), 2))
            u[0, 0] = 1.0
            u[at[0]] = (sx, -0.5 * sx)
            u[at[1]] = (0.25, sx)
            y = snapmod.yi_host(1, beta, u, precision=0)
            for e in at:
                for k in (0, 1):
                    want = Fraction(c) * Fraction(u[e, k])
                    assert abs(Fraction(y[e, k]) - want) <= tol + abs(want) / 2 ** 53, (x, e, k)


# |U| <= 1: a product is rounded at 2^-59 of the largest |U| times the largest sum
# of |c| over a record, a few times a row; an output has up to about 1000 rows:
# 1000 x 4 x 2^-59 = 7e-15 of it, and the outputs' largest is above a hundredth of
# the largest sum (as in the tests of the class stream).  The largest component
# is kept at its size, the others are spread below it.
@pytest.mark.parametrize("twojmax", [1, 4, 8, 14])
@pytest.mark.parametrize("shift", [-40, 0, 40])
def test_spread_components(snapmod, twojmax, shift):
    rng = np.random.default_rng(61 + twojmax)
    h = symmetric_u(snapmod, twojmax, rng)
    big = np.abs(h).max()
    p = rng.uniform(-80.0, 0.0, len(h)).round()
    for t in range(0, twojmax + 1, 2):  # the mirrored elements stay mirrors
        mb = t // 2
        for ma in range(mb + 1, t + 1):
            p[snapmod.half_index(twojmax, t, ma, mb)] = p[snapmod.half_index(twojmax, t, t - ma, mb)]
    h = h * 2.0 ** p[:, None]
    h[0] = (big, 0.0)
    h *= 2.0 ** shift
    beta = inputs.beta(twojmax, scale=1.0, seed=5)
    fx = snapmod.yi_host(twojmax, beta, h, precision=0)
    fp = snapmod.yi_host(twojmax, beta, h, precision=1)
    assert np.isfinite(fx).all() and np.abs(fp).max() > 0
    assert np.abs(fx - fp).max() <= 1e-12 * np.abs(fp).max()
