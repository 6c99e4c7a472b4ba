"""sqrt_pos (csrc/s2_internal.cuh) against extended precision: over its range,
at the edges where the library root takes over, and for special values."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def root(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    out = str(tmp_path_factory.mktemp("roots") / "libs2_roots.so")
    nvcc = "/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else "nvcc"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared",
                    "-Xcompiler", "-fPIC", "-I", os.path.join(os.path.dirname(HERE), "include"),
                    os.path.join(HERE, "gpu_roots.cu"), "-o", out], check=True)
    lb = C.CDLL(out)
    dp = C.POINTER(C.c_double)
    lb.roots_run.argtypes = [dp, dp, C.c_int]
    lb.roots_run.restype = C.c_int

    def run(x):
        x = np.ascontiguousarray(x, dtype=np.float64)
        y = np.zeros_like(x)
        assert lb.roots_run(x.ctypes.data_as(dp), y.ctypes.data_as(dp), x.size) == 0
        return y

    return run


def test_roots_within_half_an_ulp(root):
    """The seed is within 2^-22.6 (2^-22.9 of the approximate root, 2^-25 of
    the rounding of its argument) and so is the factor of each step: relative
    errors 1.5 * 2^-45.2 after the first step and 2^-67 after the second, less
    than 2^-13 of a last place, before the final rounding."""
    rng = np.random.default_rng(4)
    x = np.concatenate([rng.uniform(1.0, 4.0, 400000), 2.0 ** rng.uniform(-100, 100, 100000),
                        np.arange(1.0, 2000.0) ** 2, np.nextafter(np.arange(1.0, 2000.0) ** 2, 0),
                        [2.0 ** -100, np.nextafter(2.0 ** 101, 0), 2.0 ** 100]])
    y = root(x)
    ref = np.sqrt(x.astype(np.longdouble))
    near = ref.astype(np.float64)
    err = np.abs((y - near) - (ref - near).astype(np.float64)) / np.spacing(near)
    print("largest error %.6f ulp, %d of %d not the nearest" % (np.max(err), np.sum(y != near), x.size))
    assert np.max(err) <= 0.5 + 2.0 ** -12


def test_roots_beyond_the_range_and_special_values(root):
    """The library root, which is correctly rounded."""
    x = np.array([np.nextafter(2.0 ** -100, 0), 2.0 ** 101, 1e-300, 1e300, 5e-324, 0.0, -0.0, np.inf])
    assert np.array_equal(root(x), np.sqrt(x)) and np.signbit(root(np.array([-0.0]))[0])
    assert np.all(np.isnan(root(np.array([-1.0, -1e-200, -np.inf, np.nan]))))
