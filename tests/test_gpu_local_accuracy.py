"""The FP64 right-hand side against extended precision, each point's error
measured by the terms of its own stencils: accuracy does not depend on larger
values, finer spacings or other magnitudes elsewhere in the box."""
import numpy as np
import pytest

from paper_2304_05494_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

L = 2 * np.pi
LD = np.longdouble
GAMMA, MACH, OMEGA = 1.4, 0.7, 0.76
R_GAS = 1.0 / (GAMMA * MACH ** 2)
A1 = {1: (1 / LD(2),), 2: (LD(2) / 3, -LD(1) / 12), 3: (LD(3) / 4, -LD(3) / 20, LD(1) / 60),
      4: (LD(4) / 5, -LD(1) / 5, LD(4) / 105, -LD(1) / 280)}
B2 = {1: (-LD(2), LD(1)), 2: (-LD(5) / 2, LD(4) / 3, -LD(1) / 12),
      3: (-LD(49) / 18, LD(3) / 2, -LD(3) / 20, LD(1) / 90),
      4: (-LD(205) / 72, LD(8) / 5, -LD(1) / 5, LD(8) / 315, -LD(1) / 560)}
# Each field of a term carries up to 3 roundings from the primitives, a pair
# flux 3, the sums over at most 9 points one per addition, the weights and the
# sums over the directions a few: below 64 roundings of 2^-53 of the sum of
# the terms' magnitudes.
TOL = 64 * 2.0 ** -53


@pytest.fixture(scope="module")
def s2():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2304_05494_gb300 import s2 as mod
    return mod


def prims(w):
    """rho, u, v, w, T of a conserved state in extended precision."""
    w = np.asarray(w, dtype=np.float64).astype(LD)
    rho = w[0]
    u = [w[1 + a] / rho for a in range(3)]
    e = w[4] / rho - (u[0] ** 2 + u[1] ** 2 + u[2] ** 2) / 2
    return rho, u, e * (LD(GAMMA) - 1) * LD(GAMMA) * LD(MACH) ** 2


def shift(f, d, l):
    return np.roll(f, -l, axis=2 - d)


def d1(f, d, h, half):
    return sum(a * (shift(f, d, l) - shift(f, d, -l)) for l, a in enumerate(A1[half], 1)) / LD(h)


def d2(f, d, h, half):
    b = B2[half]
    return (b[0] * f + sum(b[l] * (shift(f, d, l) + shift(f, d, -l)) for l in range(1, half + 1))) / LD(h) ** 2


def around(f, d, half):
    """Largest magnitude over each point's stencil along d."""
    return np.max([np.abs(shift(f, d, l)) for l in range(-half, half + 1)], axis=0)


@pytest.mark.parametrize("order", [2, 6, 8])
@pytest.mark.parametrize("aspect", [1.0, 1e3, 1e4, 1e6])
def test_diffusion_along_the_long_side_of_the_cells(s2, aspect, order):
    """A shear w(x) in cells up to 1e6 times as long in x as in y: its
    diffusion along x is accurate whatever the weights along y are."""
    half = order // 2
    nx, ny, nz = 16, 10, 9
    h = L / nx
    ly, lz = ny * h / aspect, nz * h
    x = np.arange(nx) * h
    one = np.ones((nz, ny, nx))
    w0 = W.conserved(one, 0 * one, 0 * one, one * (0.3 * np.sin(2 * x) + 0.1 * np.cos(x)), one, GAMMA, MACH)
    with s2.Solver(nx, ny, nz, L, ly, lz, y=np.arange(ny) * (ly / ny), mach=MACH, re=1.0, weno_order=0, cfl=0.0,
                   dt_fixed=1e-3, central_order=order, visc_order=order) as sv:
        sv.set_state(w0)
        got = sv.rhs()[3]
    rho, u, T = prims(w0)
    mu = np.power(T, np.full(T.shape, LD(OMEGA)))
    want = mu * d2(u[2], 0, h, half) + OMEGA * mu / T * d1(T, 0, h, half) * d1(u[2], 0, h, half)
    big = np.max(np.abs(u[2]))
    scale = big / h ** 2 * (2 * np.max(np.abs(B2[half])) + 4) + 4 * big ** 2 / h
    err = np.max(np.abs(got - want)) / scale
    print("aspect %g, order %d: error %.2e" % (aspect, order, err))
    assert err < TOL


def jet(c, contrast, unit):
    """A state uniform along direction c whose velocities fall from 0.4 in the
    middle of the box to 1e-30 at its edge, with the density between unit and
    unit times the contrast.  (Along c the pressure differences are exactly
    zero, so the c momentum shows the transport and diffusion alone.)"""
    n = [40, 36, 44]
    n[c] = 9
    X = np.meshgrid(*(np.arange(m) * L / m for m in n[::-1]), indexing="ij")[::-1]
    p, q = X[(c + 1) % 3], X[(c + 2) % 3]
    far = np.exp(-((p - np.pi) ** 2 + (q - np.pi) ** 2) / 0.25)
    u = [None] * 3
    u[(c + 1) % 3] = 0.3 * far * np.sin(3 * p + q)
    u[(c + 2) % 3] = 0.2 * far * np.cos(2 * p)
    u[c] = 0.4 * far * np.cos(p + 2 * q)
    rho = unit * contrast ** (0.5 + 0.5 * np.cos(p + q)) * (1.0 + 0.1 * np.sin(q))
    return n, W.conserved(rho, *u, 1.0 + 0.1 * np.cos(p), GAMMA, MACH)


@pytest.mark.parametrize("order", [2, 6, 8])
@pytest.mark.parametrize("contrast,unit", [(1.0, 1.0), (1e9, 1.0), (1.0, 1e-70), (1.0, 1e50), (1.0, 1e-100)])
@pytest.mark.parametrize("c", [0, 1, 2])
def test_quiet_regions(s2, c, contrast, unit, order):
    """Mass and momentum along c, each point by the values around it."""
    half = order // 2
    n, w0 = jet(c, contrast, unit)
    h = [L / m for m in n]
    re = 50.0 / unit
    with s2.Solver(*n, L, L, L, mach=MACH, re=re, weno_order=0, cfl=0.0, dt_fixed=1e-3, central_order=order,
                   visc_order=order) as sv:
        sv.set_state(w0)
        got = sv.rhs()
    rho, u, T = prims(w0)
    mu = np.power(T, np.full(T.shape, LD(OMEGA))) / LD(re)
    sa, sb = sum(abs(a) for a in A1[half]), abs(B2[half][0]) + 2 * sum(abs(b) for b in B2[half][1:])
    want = [np.zeros_like(rho), np.zeros_like(rho)]
    scale = [np.zeros_like(rho), np.zeros_like(rho)]
    phi = u[c]
    for d in range(3):
        for l, a in enumerate(A1[half], 1):
            m = a / 4 * (rho + shift(rho, d, l)) * (u[d] + shift(u[d], d, l))
            b = shift(m, d, -l)
            want[0] = want[0] - 2 * (m - b) / h[d]
            want[1] = want[1] - (m * (phi + shift(phi, d, l)) - b * (phi + shift(phi, d, -l))) / h[d]
        flux = 4 * sa * around(rho, d, half) * around(u[d], d, half) / h[d]
        scale[0] += flux
        scale[1] += flux * around(phi, d, half) + mu * sb * around(phi, d, half) / h[d] ** 2
        want[1] = want[1] + mu * d2(phi, d, h[d], half) + OMEGA * mu / T * d1(T, d, h[d], half) * d1(phi, d, h[d], half)
    err = [np.max(np.abs(got[f] - w) / s) for f, w, s in zip((0, 1 + c), want, scale)]
    print("along %d, contrast %g, unit %g, order %d: errors %.2e %.2e" % (c, contrast, unit, order, *err))
    assert max(err) < TOL


def test_quiet_regions_do_not_depend_on_tiles(s2):
    """Which stencils are quiet follows from the fields alone: a jet's steps
    are the same bit for bit with other tiles and in a batch."""
    out = []
    for c in (0, 2):
        n, w0 = jet(c, 30.0, 1.0)
        kw = dict(mach=MACH, re=50.0, weno_order=5, threshold=0.05, cfl=0.5, dt_every=1)
        got = []
        for tiles in ([0, 0, 0], [1, 1, 1]):
            with s2.Solver(*n, L, L, L, **kw) as sv:
                sv.set_tiles(tiles)
                sv.set_state(w0)
                sv.step(3)
                got.append(sv.get_state())
        out.append((n, w0, kw, got[0]))
        assert np.array_equal(got[0], got[1])
    solvers = [s2.Solver(*n, L, L, L, **kw) for n, _, kw, _ in out]
    for sv, (_, w0, _, _) in zip(solvers, out):
        sv.set_state(w0)
    with s2.Batch(solvers, mode="worklist_all") as b:
        b.step(3)
        b.sync()
    states = [sv.get_state() for sv in solvers]
    for sv in solvers:
        sv.close()
    for w, (_, _, _, want) in zip(states, out):
        assert np.array_equal(w, want)
