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
