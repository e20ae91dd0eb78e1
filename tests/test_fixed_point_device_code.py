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


def test_erfcx(lib):
    rng = np.random.default_rng(13)
    x = np.concatenate([rng.uniform(0.0, 6.25, 4000), np.arange(26) / 4.0, np.nextafter(np.arange(1, 26) / 4.0, 0.0),
                        [0.0, 5e-324, 1e-300, 6.25]])
    y = call(lib, lib.erfcx_fixed, x)
    for v, a in zip(y, x):
        a = mp.mpf(float(a))
        ref = mp.exp(a * a) * mp.erfc(a)
        assert abs(mp.mpf(float(v)) - ref) <= mp.mpf(10) ** -15 * ref, (a, v)      # the tables' 2e-16 and sums' 2^-57
    assert np.array_equal(call(lib, lib.erfcx_fixed, [7.0, np.inf]), call(lib, lib.erfcx_fixed, [6.25, 6.25]))


@pytest.mark.parametrize("seed", [1.0, 1.0 - 2.0 ** -22, 1.0 + 2.0 ** -22])
def test_faddeeva(lib, seed):
    """Where both factors' edges are: the real and imaginary axes, Z near +-1 (z near 0 and at
    infinity), large |z|; the reciprocal's seed two units off either way."""
    rng = np.random.default_rng(14)
    z = np.concatenate([rng.uniform(-8.0, 8.0, 1500) + 1j * 10.0 ** rng.uniform(-8.0, 3.0, 1500),
                        np.linspace(-8.0, 8.0, 101), 1j * np.linspace(0.0, 12.0, 61), [0.0, 1e-300, 1e-8j, 1e30j]])
    lib.set_seed_factor(np.float32(seed))
    try:
        w = call(lib, lib.faddeeva_fixed, np.stack([z.real, z.imag], 1), width=2)
    finally:
        lib.set_seed_factor(1.0)
    for got, a in zip(w[:, 0] + 1j * w[:, 1], z):
        a = mp.mpc(complex(a))
        if abs(a) > 1e6:
            ref = mp.mpc(0, 1) / (mp.sqrt(mp.pi) * a)
        else:
            ref = mp.exp(-a * a) * mp.erfc(-mp.mpc(0, 1) * a)
        assert abs(mp.mpc(complex(got)) - ref) <= mp.mpf(2e-15) * abs(ref), (a, got)
    flip = call(lib, lib.faddeeva_fixed, np.stack([-z.real, z.imag], 1), width=2)
    assert np.array_equal(flip, w * [1.0, -1.0])


@pytest.mark.parametrize("Gamma, mu, c_exp, most", [(0.66, 0.0, 4e-4, 15.0), (0.7025, 0.03, 0.01, 15.0),
                                                    (5.0, -1.3, 0.5, 40.0), (0.66e-9, 7e8, 0.0, 1.5e10),
                                                    (0.66e12, 1e-14, 1e-3, 15e-12), (-0.3, 0.0, 0.0, 8.0),
                                                    (40.0, 0.0, 0.0, 15.99)])
def test_decay_exponential(lib, Gamma, mu, c_exp, most):
    """Relative error 2^-53 (the rounding) and y's last places, (2 + 2^-47 / ulp) of them: y =
    64 log2 of the value, |y| < 2^ey, has 60 - max(ey, 6) fraction bits and its constant is a double."""
    rng = np.random.default_rng(15)
    t = np.concatenate([rng.uniform(-most, most, 1500), most * (1.0 - 2.0 ** -np.arange(1.0, 54.0)), [0.0, most, -most]])
    y, ok = np.empty(t.size), np.zeros(t.size, np.int32)
    before = lib.overflows()
    args = [ctypes.c_double(v) for v in (Gamma, mu, c_exp, most)]
    assert lib.exp_line(*args, _p(t), _p(y), _p(ok), ctypes.c_int64(t.size)) == 1
    assert lib.overflows() == before
    size = 64.0 * (1.0 + (abs(Gamma) * (most + abs(mu)) + c_exp) / np.log(2.0))
    ey = max(6, int(np.ceil(np.log2(size))))
    bound = mp.mpf(2) ** -53 + (2 * mp.mpf(2) ** (ey - 60) + mp.mpf(2) ** (ey - 53)) * mp.log(2) / 64
    for v, o, a in zip(y, ok, t):
        e = -mp.mpf(Gamma) * (mp.mpf(float(a)) - mp.mpf(mu)) + mp.mpf(c_exp)
        if not o:
            assert abs(e) > 700
            continue
        ref = 2 * mp.exp(e)
        assert abs(mp.mpf(float(v)) - ref) <= bound * ref, (a, v)


@pytest.mark.parametrize("Dm, mu, ph0, most", [(17.77, 0.0, 0.024, 15.0), (-17.77, 0.03, -0.5, 15.0), (0.5, 0.0, 0.0, 15.0),
                                               (60.0, -1.3, 3.0, 40.0), (17.77e12, 1e-14, 0.02, 15e-12), (0.0, 0.0, 0.3, 1.0)])
def test_phase(lib, Dm, mu, ph0, most):
    """Absolute error: a few 2^-60 and the phase's last places (as above, in units of pi / 32)."""
    rng = np.random.default_rng(16)
    t = np.concatenate([rng.uniform(-most, most, 1500), most * (1.0 - 2.0 ** -np.arange(1.0, 54.0)), [0.0, most, -most]])
    y = np.empty(2 * t.size, np.int64)
    before = lib.overflows()
    args = [ctypes.c_double(v) for v in (Dm, mu, ph0, most)]
    assert lib.phase_line(*args, _p(t), _p(y), ctypes.c_int64(t.size)) == 1
    assert lib.overflows() == before
    size = (abs(Dm) * (most + abs(mu)) + abs(ph0)) * 32.0 / np.pi
    ey = max(6, int(np.ceil(np.log2(max(size, 1.0)))))
    bound = mp.mpf(2) ** -58 + (2 * mp.mpf(2) ** (ey - 60) + mp.mpf(2) ** (ey - 53)) * mp.pi / 32
    for s, c, a in zip(y[0::2], y[1::2], t):
        ph = mp.mpf(Dm) * (mp.mpf(float(a)) - mp.mpf(mu)) - mp.mpf(ph0)
        assert abs(mp.mpf(int(s)) / 2 ** 62 - mp.sin(ph)) <= bound and abs(mp.mpf(int(c)) / 2 ** 62 - mp.cos(ph)) <= bound


@pytest.mark.parametrize("seed", [1.0, 1.0 - 2.0 ** -22, 1.0 + 2.0 ** -22])
def test_angular_products(lib, seed):
    """Up to the angles' limits (fx_angles_ok), on the axes and in between: an absolute error of
    2^-58 (a few 2^-60 per factor), and with q = sqrt(a b) what the last places of a = sin^2 thK and
    b = sin^2 thmu (2^-62 each) make of it: (a + b) / (2 q) of them, up to 2^-55 at the limits."""
    rng = np.random.default_rng(17)
    top = np.nextafter(1.0 - 2.0 ** -17, 0.0)
    edge = np.array([0.0, 1e-300, 0.5, -0.5, top, -top, 1.0 - 2.0 ** -16, 2.0 ** -30])
    phi = np.array([0.0, np.pi, -np.pi, np.pi / 2, 3.9999, -3.9999, np.pi / 32 * 3.5, 1e-300])
    a = np.concatenate([np.stack([rng.uniform(-1, 1, 600) * top, rng.uniform(-1, 1, 600) * top,
                                  rng.uniform(-np.pi, np.pi, 600)], 1),
                        np.array([(x, y, p) for x in edge for y in edge for p in phi])])
    assert all(lib.angles_ok(*row) for row in a)
    assert not any(lib.angles_ok(*row) for row in ((1.0 - 2.0 ** -17, 0, 0), (0, -1.0, 0), (0, 0, 4.0), (np.nan, 0, 0)))
    lib.set_seed_factor(np.float32(seed))
    try:
        g = call(lib, lib.basis, a, np.int64, 10)
    finally:
        lib.set_seed_factor(1.0)
    for row, (ck, cl, ph) in zip(g, a):
        ck, cl, ph = (mp.mpf(float(v)) for v in (ck, cl, ph))
        sk2, sl2, sp, cp = 1 - ck * ck, 1 - cl * cl, mp.sin(ph), mp.cos(ph)
        G, q = sk2 * sl2, mp.sqrt(sk2 * sl2)
        ref = (sl2, sk2, G, G * cp * cp, G * sp * cp, q * cl * cp * ck, q * cl * sp * ck, q * cl * cp, q * cl * sp, ck * sl2)
        root = mp.mpf(2) ** -62 * (sk2 + sl2) / (2 * q)
        for k, (v, r) in enumerate(zip(row, ref)):
            assert abs(mp.mpf(int(v)) / 2 ** 62 - r) <= mp.mpf(2) ** -58 + (root if 5 <= k < 9 else 0), (ck, cl, ph, k, v)


def test_to_double(lib):
    rng = np.random.default_rng(18)
    for v in [0, 1, -1, 2 ** 53 + 1, -(2 ** 54) - 2, 2 ** 62, 2 ** 63 - 1, -(2 ** 63) + 1, -(2 ** 63)] + \
            [int(x) >> int(s) for x, s in zip(rng.integers(-2 ** 63, 2 ** 63 - 1, 500), rng.integers(0, 62, 500))]:
        for e2 in (0, 5, -300, 400):
            got = mp.mpf(lib.to_double(v, e2))
            ref = mp.mpf(v) * mp.mpf(2) ** (e2 - 62)
            assert abs(got - ref) <= abs(ref) * mp.mpf(2) ** -53, (v, e2)
