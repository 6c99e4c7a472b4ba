"""The integer arithmetic of csrc/s2_fixed.cuh in exact integers: every value
stays in its type and every result within its derived error."""
from fractions import Fraction

import numpy as np
import pytest

LIMB, MASK = 30, (1 << 30) - 1
# the weights of the pair fluxes, doubles as in the kernels
ACOEF = {1: (1 / 2,), 2: (2 / 3, -1 / 12), 3: (3 / 4, -3 / 20, 1 / 60), 4: (4 / 5, -1 / 5, 4 / 105, -1 / 280)}
# stencil weights over a common denominator and the bits that they add up to
C1 = {1: ((1,), 1), 2: ((8, -1), 5), 3: ((45, -9, 1), 7), 4: ((672, -168, 32, -3), 11)}
C2 = {1: ((-2, 1), 2), 2: ((-30, 16, -1), 6), 3: ((-490, 270, -27, 2), 11), 4: ((-14350, 8064, -1008, 128, -9), 15)}


def fits(x, bits):
    assert -(1 << (bits - 1)) <= x < (1 << (bits - 1)), (x, bits)
    return x


def total(terms):
    """FxSum of (weight, word) pairs."""
    hi = fits(sum(c * (fits(v, 64) >> 32) for c, v in terms), 64)
    pos = sum(c * (v & 0xffffffff) for c, v in terms if c > 0)
    neg = sum(-c * (v & 0xffffffff) for c, v in terms if c < 0)
    assert max(pos, neg) < 1 << 63
    return hi, fits(pos - neg, 64)


def value(hi, lo, bits):
    """FxSum::value: the integer and the bits cut from it."""
    t = fits(hi + (lo >> 32), 64)
    drop = 0 if -(1 << 30) <= t < 1 << 30 else bits
    r = (lo & 0xffffffff) + ((1 << drop) - 1 if t < 0 else 0)
    return fits((t << (32 - drop)) + (r >> drop), 64), drop


def cut(x, n):
    """x / 2^n towards zero."""
    return x >> n if x >= 0 else -(-x >> n)


@pytest.mark.parametrize("half", [1, 2, 3, 4])
def test_word_sums(half):
    """Derivatives of words at their extremes, at random and small: exact
    below 2^62, above it their last bits cut towards zero, and the same with
    the sign changed for the negative field."""
    rng = np.random.default_rng(half)
    top = (1 << 62) - (1 << 9)  # the largest double's word
    (c1, w1), (c2, w2) = C1[half], C2[half]
    assert 2 * sum(abs(c) for c in c1) <= 1 << w1 and abs(c2[0]) + 2 * sum(abs(c) for c in c2[1:]) <= 1 << w2
    for trial in range(300):
        def draw(signs):
            return [int(s) * (top if trial < 80 else int(rng.integers(0, top >> (trial % 60)))) for s in signs]

        up, dn, c = draw(rng.choice([-1, 1], half)), draw(rng.choice([-1, 1], half)), draw([1])[0]
        if trial < 10:  # every term of one sign
            up, dn = [int(np.sign(x)) * top for x in c1], [-int(np.sign(x)) * top for x in c1]
        if 10 <= trial < 20:
            c, up, dn = -top, [int(np.sign(x)) * top for x in c2[1:]], [int(np.sign(x)) * top for x in c2[1:]]
        for first in (True, False):
            def sums(s):
                pairs = zip(c1 if first else c2[1:], up, dn)
                terms = [(w, fits(s * a - s * b if first else s * a + s * b, 64)) for w, a, b in pairs]
                return terms if first else [(c2[0], s * c)] + terms

            w = w1 if first else w2
            exact = sum(a * b for a, b in sums(1))
            v, drop = value(*total(sums(1)), w)
            assert v == cut(exact, drop) and (drop == 0 or abs(exact) >= 1 << 62)
            assert value(*total(sums(-1)), w) == (-v, drop) or abs(exact) == 1 << 62


def test_loud_values():
    """The kernels' test of several values at once: bits from 2 L on in the
    sum with L, for a power of two L."""
    rng = np.random.default_rng(0)
    for loud in (1 << 22, 1 << 24, 1 << 27):
        edges = [-loud - 1, -loud, -loud + 1, -1, 0, 1, loud - 1, loud, -(1 << 29), 1 << 29]
        for _ in range(500):
            v = [int(x) for x in rng.choice(edges, 7)]
            bits = 0
            for x in v:
                bits |= (x + loud) & 0xffffffff
            assert (bits < 2 * loud) == all(-loud <= x < loud for x in v)


@pytest.mark.parametrize("half", [1, 2, 3, 4])
def test_flux_difference_error(half):
    """The flux difference of an order-2 half point against exact rationals, in
    units of 2^-60 of the exponents' largest product.  A sum of two pairs of
    limbs loses at most 1 in its cut, half of that enters the pair flux, which
    adds 1 for the cut and 1 for the weight; each pair flux meets field values
    of at most 1/2 twice (its own and the centre's): 2.5 per pair flux, of
    which there are 2 half; the last cut at most 2.  For velocities and field
    values near the loud bounds, 2^-5 of their exponents' powers of two, a pair
    flux is off by at most 0.5 + 1 + 2^-5 and meets values of at most 2^-6
    twice, 0.05 per pair flux, and the sum keeps lower bits: the error falls
    with the products."""
    rng = np.random.default_rng(100 + half)
    top = (1 << 59) - 1
    worst = 0
    for trial in range(300):
        def draw(n):
            return [int(s) * (top if trial < 150 else int(rng.integers(0, top))) for s in rng.choice([-1, 1], n)]

        rho, un, phi = (draw(2 * half + 1) for _ in range(3))
        if trial >= 220:
            un, phi = [x >> 5 for x in un], [x >> 5 for x in phi]
        if trial < 40:
            rho, un = [top] * len(rho), [top] * len(un)
            phi = [top if i >= half else -top for i in range(len(phi))]

        def limbs(x):
            s = -1 if x < 0 else 1
            return s * (abs(x) & MASK), s * (abs(x) >> LIMB)

        def mulhi(a, b):
            hl = fits(a[1] * b[0] + a[0] * b[1] + (fits(a[0] * b[0], 64) >> LIMB), 64)
            return fits(a[1] * b[1] + (hl >> LIMB), 64)

        def pair(i, j, l):
            P = mulhi(*[[fits(x + y, 32) for x, y in zip(limbs(f[i]), limbs(f[j]))] for f in (rho, un)])
            a = ACOEF[half][l - 1] * 0.5
            k = int(abs(a) * 2.0 ** 60)
            k = tuple((-1 if a < 0 else 1) * v for v in (k & MASK, k >> LIMB))
            m = mulhi((P & MASK, fits(P >> LIMB, 32)), k)
            return m & MASK, fits(m >> LIMB, 32)

        Ml = Mh = A = B = C = 0
        exact = Fraction(0)
        for l in range(1, half + 1):
            for s, i, j in ((1, half, half + l), (-1, half - l, half)):
                m = pair(i, j, l)
                Ml, Mh = Ml + s * m[0], Mh + s * m[1]
                v = limbs(phi[half + s * l])
                A, B = fits(A + s * m[1] * v[1], 64), fits(B + s * (m[1] * v[0] + m[0] * v[1]), 64)
                C = fits(C + s * m[0] * v[0], 64)
                exact += s * Fraction(ACOEF[half][l - 1]) / 2 * (rho[i] + rho[j]) * (un[i] + un[j]) \
                    * (phi[half] + phi[half + s * l])
        Mh, Ml = fits(Mh + (Ml >> LIMB), 32), Ml & MASK
        c = limbs(phi[half])
        A, B = fits(A + Mh * c[1], 64), fits(B + Mh * c[0] + Ml * c[1], 64)
        B = fits(B + (fits(Ml * c[0], 64) >> LIMB) + (C >> LIMB), 64)
        A = fits(A + (B >> LIMB), 64)
        up = min(62 - (A if A >= 0 else ~A).bit_length(), LIMB)
        assert up >= 0
        D = Fraction(fits((A << up) + ((B & MASK) >> (LIMB - up)), 64), 1 << up)
        error = abs(D - exact / 2 ** 120)
        worst = max(worst, error)
        assert trial < 220 or error <= 0.1 * half + 0.01
    bound = 5 * half + 2
    print("order %d: error %.2f, bound %d" % (2 * half, float(worst), bound))
    assert worst <= bound
