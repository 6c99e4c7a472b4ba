"""The power law and the logarithm of csrc/s2_power.cuh against extended
precision: inside the tables' range, at its edges and around 1, where the
general functions take over, and for arguments that are no temperatures."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    out = str(tmp_path_factory.mktemp("power") / "libs2_power.so")
    nvcc = "/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else "nvcc"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared",
                    "-Xcompiler", "-fPIC", "-I", os.path.join(os.path.dirname(HERE), "include"),
                    os.path.join(HERE, "gpu_power.cu"), "-o", out], check=True)
    lb = C.CDLL(out)
    lb.power_run.argtypes = [C.c_int, C.POINTER(C.c_double), C.POINTER(C.c_double), C.c_int, C.c_double]
    lb.power_run.restype = C.c_int
    return lb


def run(lib, which, x, omega=0.76):
    x = np.ascontiguousarray(x, dtype=np.float64)
    out = np.zeros_like(x)
    dp = C.POINTER(C.c_double)
    assert lib.power_run(which, x.ctypes.data_as(dp), out.ctypes.data_as(dp), x.size, omega) == 0
    return out


def arguments(span):
    rng = np.random.default_rng(3)
    k = np.arange(129) / 128.0 + 1.0  # the table's cell edges
    near = np.concatenate([k, np.nextafter(k, 0), np.nextafter(k, 4)])
    x = [near * 2.0 ** e for e in (-2, -1, 0, 1)]
    x += [rng.uniform(0.2, 5.0, 20000), 1.0 + rng.uniform(-1e-3, 1e-3, 5000), 2.0 ** rng.uniform(-span, span, 20000)]
    return np.concatenate(x)


@pytest.mark.parametrize("omega", [0.76, 0.5, 1.0, 0.666, 2.5, 4.0, -0.7, 0.0])
def test_power_law(lib, omega):
    """Within 0.54 ulp where the tables serve (exponent within 30/|omega| and
    32; the roundings of E add up to 1.04 2^-58, those of the exponential to
    less than 2^-59, of a last place of 2^-53), within 4 ulp where the general function does (T up to 2^60)."""
    x = arguments(60)
    y = run(lib, 0, x, omega)
    # (array exponents: numpy takes a scalar 0.5 through another root)
    ref = np.power(x.astype(np.longdouble), np.full(x.size, omega, dtype=np.longdouble))
    hi = ref.astype(np.float64)
    lo = (ref - hi.astype(np.longdouble)).astype(np.float64)
    err = np.abs((y - hi) - lo) / np.spacing(hi)
    print("omega %g: largest error %.3f ulp at x = %s" % (omega, np.max(err), float(x[np.argmax(err)]).hex()))
    inside = np.abs(np.floor(np.log2(x))) <= (min(32, np.floor(30.0 / abs(omega)) - 1) if omega else 32)
    assert np.max(err[inside]) <= 0.54, np.max(err[inside])
    assert np.all(err <= 4.0), np.max(err)


def test_power_law_beyond_its_exponents_and_arguments(lib):
    x = np.array([0.3, 1.0, 7.0])
    assert np.allclose(run(lib, 0, x, 4.5), x ** 4.5, rtol=1e-15, atol=0)  # the general function
    bad = run(lib, 0, np.array([-1.0, np.nan]))
    assert np.all(np.isnan(bad))
    # pow(-inf, 0.76) is +inf in C
    assert np.array_equal(run(lib, 0, np.array([0.0, np.inf, -np.inf])), [0.0, np.inf, np.inf])


def test_logarithm(lib):
    """To 2^-56 absolute plus the result's rounding."""
    x = arguments(45)  # beyond 2^40 the library's logarithm
    y = run(lib, 1, x).astype(np.longdouble)
    ref = np.log(x.astype(np.longdouble))
    assert np.max(np.abs(y - ref) - np.spacing(np.abs(ref).astype(np.float64))) <= 2.0 ** -56
    bad = run(lib, 1, np.array([-1.0, np.nan, 0.0, np.inf]))
    assert np.isnan(bad[0]) and np.isnan(bad[1]) and bad[2] == -np.inf and bad[3] == np.inf
