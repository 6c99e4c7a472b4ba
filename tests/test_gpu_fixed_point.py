"""The fixed-point stencils of the FP64 path (csrc/s2_fixed.cuh): limb
arithmetic at its bounds (CPU), and the right-hand side on both sides of the
rule that chooses between them and double precision (GPU, against the
oracle)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2304_05494_gb300 import workloads as W

L = 2 * np.pi
# one RHS against the oracle, of the flux scale (tests/test_gpu_parity.py)
RHS_TOL = 1e-13
LIMB = 30
MASK = (1 << LIMB) - 1
ACOEF = {1: (1 / 2,), 2: (2 / 3, -1 / 12), 3: (3 / 4, -3 / 20, 1 / 60), 4: (4 / 5, -1 / 5, 4 / 105, -1 / 280)}


def limbs(x):
    """Sign-magnitude limbs (lo, hi) of an integer, as fx_split makes them."""
    s = -1 if x < 0 else 1
    return s * (abs(x) & MASK), s * (abs(x) >> LIMB)


def fits(x, bits):
    assert -(1 << (bits - 1)) <= x < (1 << (bits - 1)), (x, bits)
    return x


def mulhi(a, b):
    hl = fits(a[1] * b[0] + a[0] * b[1], 64)
    return fits(a[1] * b[1] + (hl >> LIMB), 64)


@pytest.mark.parametrize("half", [1, 2, 3, 4])
def test_flux_accumulators_stay_in_range(half):
    """The flux difference in exact integers with fields and signs at their
    extremes and at random: every 32- and 64-bit value of the kernel stays
    in range, and the result is within the stated 2^-55 of the largest."""
    rng = np.random.default_rng(half)
    top = (1 << 59) - 1
    for trial in range(300):
        big = trial < 200
        def draw(n):
            return [int(s) * (top if big else int(rng.integers(0, top))) for s in rng.choice([-1, 1], n)]
        rho, un, phi = (draw(2 * half + 1) for _ in range(3))
        if trial < 40:  # every flux term of the same sign
            rho, un = [top] * len(rho), [top] * len(un)
            phi = [top if i >= half else -top for i in range(len(phi))]

        def pair(i, j, l):
            r = [fits(p + q, 32) for p, q in zip(limbs(rho[i]), limbs(rho[j]))]
            n = [fits(p + q, 32) for p, q in zip(limbs(un[i]), limbs(un[j]))]
            P = mulhi(r, n)
            a = ACOEF[half][l - 1] * 0.5
            k = int(abs(a) * 2.0 ** 60)
            k = tuple((-1 if a < 0 else 1) * v for v in (k & MASK, k >> LIMB))
            m = mulhi((P & MASK, fits(P >> LIMB, 32)), k)
            return m & MASK, fits(m >> LIMB, 32)

        Ml = Mh = 0
        pairs = []
        for l in range(1, half + 1):
            mp, mm = pair(half, half + l, l), pair(half - l, half, l)
            Ml = fits(Ml + mp[0] - mm[0], 32)
            Mh = fits(Mh + mp[1] - mm[1] + (Ml >> LIMB), 32)
            Ml &= MASK
            pairs.append((l, mp, mm))
        c = limbs(phi[half])
        A, B = Mh * c[1], fits(Mh * c[0] + Ml * c[1], 64)
        exact = 0
        for l, mp, mm in pairs:
            vp, vm = limbs(phi[half + l]), limbs(phi[half - l])
            A = fits(A + mp[1] * vp[1] - mm[1] * vm[1], 64)
            for t in (mp[1] * vp[0], mp[0] * vp[1], -mm[1] * vm[0], -mm[0] * vm[1]):
                B = fits(B + t, 64)
            for s, j in ((1, half + l), (-1, half - l)):
                exact += s * ACOEF[half][l - 1] * 0.5 * float((rho[half] + rho[j]) * (un[half] + un[j])) \
                    * (phi[half] + phi[j]) / 2.0 ** 60
        D = fits(A + (B >> LIMB), 64)
        assert abs(D - exact / 2.0 ** 60) < 64 + 2.0 ** -50 * 2.0 ** 60


# weights over a common denominator and the bits of their magnitudes (FxStencil)
C1 = {1: ((1,), 1), 2: ((8, -1), 5), 3: ((45, -9, 1), 7), 4: ((672, -168, 32, -3), 11)}
C2 = {1: ((-2, 1), 2), 2: ((-30, 16, -1), 6), 3: ((-490, 270, -27, 2), 11), 4: ((-14350, 8064, -1008, 128, -9), 15)}


def stencil_sum(hi, lo, bits):
    """fx_sum: the integer and the bits cut from it."""
    cut = max(bits - 3, 0)
    t = fits(hi + (lo >> LIMB), 64)
    drop = cut if cut and not -(1 << 32) <= t < (1 << 32) else 0
    return fits((t << (LIMB - drop)) + ((lo & MASK) >> drop), 64), drop


@pytest.mark.parametrize("half", [1, 2, 3, 4])
def test_stencil_sums_stay_in_range(half):
    """First derivatives and Laplacians of fields at their extremes and at
    random: values in range, and exact or cut as stated."""
    rng = np.random.default_rng(10 + half)
    top = (1 << 59) - 1
    (c1, w1), (c2, w2) = C1[half], C2[half]
    assert 2 * sum(abs(c) for c in c1) <= 1 << w1
    assert abs(c2[0]) + 2 * sum(abs(c) for c in c2[1:]) <= 1 << w2
    for trial in range(200):
        def draw(signs):
            return [int(s) * (top if trial < 60 else int(rng.integers(0, top >> (trial % 40)))) for s in signs]

        up, dn = (draw(rng.choice([-1, 1], half)) for _ in range(2))
        if trial < 10:
            up, dn = [int(np.sign(c)) * top for c in c1], [-int(np.sign(c)) * top for c in c1]
        lu, ld = [limbs(x) for x in up], [limbs(x) for x in dn]
        hi = sum(c * fits(a[1] - b[1], 32) for c, a, b in zip(c1, lu, ld))
        lo = sum(c * fits(a[0] - b[0], 32) for c, a, b in zip(c1, lu, ld))
        v, drop = stencil_sum(fits(hi, 64), fits(lo, 64), w1)
        exact = sum(c * (a - b) for c, a, b in zip(c1, up, dn))
        assert v == exact >> drop and (drop == 0 or abs(v) >= 1 << 53)
        # Laplacian: three directions with weights of any ratio
        acc, exact = [0, 0, 0], 0
        kmax = (1 << 60) - 1
        for d in range(3):
            up, dn, c = draw(rng.choice([-1, 1], half)), draw(rng.choice([-1, 1], half)), draw([1])[0]
            if trial < 10:
                c, up, dn = -top, [int(np.sign(x)) * top for x in c2[1:]], [int(np.sign(x)) * top for x in c2[1:]]
            k = kmax if d == trial % 3 or trial < 10 else int(rng.integers(0, kmax))
            kl, kh = k & MASK, k >> LIMB
            lc, lu, ld = limbs(c), [limbs(x) for x in up], [limbs(x) for x in dn]
            hi = c2[0] * lc[1] + sum(w * fits(a[1] + b[1], 32) for w, a, b in zip(c2[1:], lu, ld))
            lo = c2[0] * lc[0] + sum(w * fits(a[0] + b[0], 32) for w, a, b in zip(c2[1:], lu, ld))
            t = fits(hi, 64) + (fits(lo, 64) >> LIMB)
            r, t0, t1 = lo & MASK, t & MASK, fits(t >> LIMB, 32)
            acc = [fits(x, 64) for x in (acc[0] + t1 * kh, acc[1] + t1 * kl + t0 * kh, acc[2] + t0 * kl + r * kh)]
            exact += k * (c2[0] * c + sum(w * (a + b) for w, a, b in zip(c2[1:], up, dn)))
        v, drop = stencil_sum(acc[0], fits(acc[1] + (acc[2] >> LIMB), 64), w2 + 2)
        assert abs(v - (exact >> (60 + drop))) <= 8


def periodic_state(shape, contrast, which, unit, seed=5):
    """Smooth periodic box whose density or temperature spans the given
    factor, in units where the density is of the given size; w = 0."""
    nx, ny, nz = shape
    x, y, z = (np.arange(n) * L / n for n in shape)
    Z, Y, X = np.meshgrid(z, y, x, indexing="ij")
    span = np.exp(0.5 * np.log(contrast) * np.sin(X) * np.cos(Y + Z)) if contrast > 1 else np.ones_like(X)
    span = span * (1.0 + 1e-3 * np.cos(X - Z))
    rho, T = (span, np.ones_like(span)) if which == "rho" else (np.ones_like(span), span)
    u, v = 0.3 * np.sin(Y) * np.cos(X), 1e-9 * np.cos(Z + X)
    return W.conserved(unit * rho, u, v, np.zeros_like(u), T, 1.4, 0.7)


@pytest.mark.gpu
@pytest.mark.parametrize("order", [2, 6, 8])
@pytest.mark.parametrize("contrast,which,unit", [
    (1.0, "rho", 1.0), (30.0, "rho", 1.0), (30.0, "T", 1.0),      # fixed point
    (63.0, "rho", 1e-30), (63.0, "T", 1e40),                      # either side of a power of two
    (200.0, "rho", 1.0), (200.0, "T", 1.0), (1.5, "rho", 1e70),   # double precision
])
def test_rhs_on_both_sides_of_the_rule(contrast, which, unit, order):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2304_05494_gb300 import s2
    from tests.test_gpu_parity import flux_scale
    shape = (37, 21, 35)
    w0 = periodic_state(shape, contrast, which, unit)
    # the viscosity follows the density unit, so that every term keeps its
    # weight; WENO only near unit density (its weights multiply the squares
    # of squared differences and overflow above 1e38)
    kw = dict(mach=0.7, re=150.0 / unit, weno_order=5 if unit == 1.0 else 0, threshold=0.2, central_order=order, visc_order=order)
    pr = O.Problem(*shape, L, L, L, **kw)
    with s2.Solver(*shape, L, L, L, cfl=0.0, dt_fixed=1e-3, **kw) as sv:
        sv.set_state(w0)
        a = sv.rhs()
        b = sv.rhs()
        flags = sv.flags()
    assert np.array_equal(a, b)
    ref, of = O.rhs(pr, w0, flags=True)
    S = np.maximum(flux_scale(w0, pr), np.max(np.abs(ref), axis=(1, 2, 3)))
    e = np.max(np.abs(a - ref), axis=(1, 2, 3)) / np.where(S > 0, S, 1.0)
    print("contrast %g of %s, unit %g, order %d:" % (contrast, which, unit, order), e)
    for f, g in zip(flags, of) if kw["weno_order"] else ():
        assert np.array_equal(f, g)
    assert np.all(e < RHS_TOL), e
