"""The fixed-point functions of the likelihood kernels themselves (fast_fixed.cuh,
faddeeva.cuh), compiled for the host by helpers/fixed_point_host.cpp, against 50-digit
mpmath: dense arguments over each function's range and the edges of its formats
(mantissas up to 2 - 2^-52, where a 63-bit magnitude is fullest).  Every signed
operation is checked for overflow as it runs.  The tolerances are the bounds that the
functions' comments state, plus the rounding of the result to a double."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")
HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CUDA = "/usr/local/cuda/include"


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA, "cuda_runtime.h")):
        pytest.skip("no host compiler or CUDA headers")
    so = str(tmp_path_factory.mktemp("host") / "fixed_point_host.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared",
                    "-fsanitize=signed-integer-overflow", "-I" + CUDA, "-I" + os.path.join(ROOT, "include"),
                    "-I" + os.path.join(ROOT, "paper_1706_01420_gb300", "csrc"), "-o", so,
                    os.path.join(HERE, "helpers", "fixed_point_host.cpp")], check=True, capture_output=True)
    d = ctypes.CDLL(so)
    d.overflows.restype = ctypes.c_longlong
    d.set_seed_factor.argtypes = [ctypes.c_float]
    d.to_double.restype = ctypes.c_double
    d.to_double.argtypes = [ctypes.c_int64, ctypes.c_int]
    d.angles_ok.argtypes = [ctypes.c_double] * 3
    with mp.workdps(50):
        yield d
    assert d.overflows() == 0


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def call(lib, f, x, dtype=np.float64, width=1):
    """f elementwise (n arguments, n x width results); no signed overflow on the way."""
    x = np.ascontiguousarray(x, dtype=np.float64)
    n = x.shape[0]
    y = np.empty(n * width, dtype)
    before = lib.overflows()
    f(_p(x), _p(y), ctypes.c_int64(n))
    assert lib.overflows() == before
    return y if width == 1 else y.reshape(n, width)


# just below every power of two, down to the last bit
FULL = np.concatenate([2.0 ** e * (1.0 - 2.0 ** -np.arange(2.0, 54.0)) for e in range(-8, 11)])


def test_gaussian_exponential(lib):
    rng = np.random.default_rng(11)
    a = -np.concatenate([[0.0, 5e-324, 1e-300, 1e-20, 705.0], rng.uniform(0.0, 705.0, 4000),
                         10.0 ** rng.uniform(-12.0, 2.8, 4000), FULL])
    a = a[a >= -705.0]
    y = call(lib, lib.exp_neg, a)
    for v, x in zip(y, a):
        ref = mp.exp(mp.mpf(float(x)))
        bound = mp.mpf(2) ** -53 + max(mp.mpf(2) ** -54, -mp.mpf(float(x)) * mp.mpf(2) ** -59)
        assert abs(mp.mpf(float(v)) - ref) <= bound * ref, (x, v)


def test_log(lib):
    rng = np.random.default_rng(12)
    x = np.concatenate([2.0 ** rng.uniform(-126.0, 126.9, 4000), rng.uniform(0.5, 2.0, 4000), [1.0],
                        1.0 + np.arange(128) / 128.0, np.nextafter(1.0 + np.arange(1, 129) / 128.0, 0.0), FULL,
                        FULL * 2.0 ** -110, FULL * 2.0 ** 110])
    y = call(lib, lib.log_q56, x, np.int64)
    for v, a in zip(y, x):
        e = abs(int(np.frexp(a)[1]) - 1)
        assert abs(int(v) - mp.log(mp.mpf(float(a))) * 2 ** 56) <= 2 + e / 3.0, (a, v)
