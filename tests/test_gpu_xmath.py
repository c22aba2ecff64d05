"""The plain FP64 form's own scalar arithmetic against CUDA's operations, bit
for bit: the reciprocal and quotients by it, products on the integer pipe,
the paired exponential, the fast paths of exponential and logarithm,
comparisons on bit patterns and the stage count's root.  Operands: random
bit patterns, random significands at ordinary sizes, the ends of every range
and their neighbours, significands next to all ones, exact and nearly exact
quotients, products that tie, signed zeros, subnormals, infinities, NaN."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1611_02274_gb300 import build as NB

pytestmark = pytest.mark.gpu

N = 1 << 20


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "xmath_probe.cu")
    out = str(tmp_path_factory.mktemp("xmath") / "xmath_probe.so")
    subprocess.run([NB.nvcc(), *NB.ARCH, *NB.NVCC_FLAGS, "--fmad=false", "-shared", "-cudart=static", src, "-o", out],
                   check=True, capture_output=True)
    f = ctypes.CDLL(out).xmath_check
    f.restype = ctypes.c_longlong
    f.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_longlong, ctypes.c_void_p]
    return f


def differ(lib, what, a, b):
    a, b = (np.ascontiguousarray(x, dtype=np.float64) for x in np.broadcast_arrays(a, b))
    first = np.zeros(2)
    n = lib(what, a.ctypes.data, b.ctypes.data, a.size, first.ctypes.data)
    return n, [float(v).hex() for v in first]


def specials():
    e = [0.0, np.inf, np.nan, 5e-324, 2.0 ** -1022, np.nextafter(2.0 ** -1022, 0), np.finfo(float).max, 1.0, 3.0, 1e-20]
    for k in (-745, -709, -707, -700, -600, -400, -100, -60, -1, 0, 1, 60, 100, 400, 600, 700, 707, 709, 745):
        if abs(k) <= 700:
            e += [2.0 ** k, np.nextafter(2.0 ** k, 0), np.nextafter(2.0 ** k, np.inf), 1.5 * 2.0 ** k]
        e += [float(k), np.nextafter(float(k), 0), np.nextafter(float(k), 1e3)]
    e = np.array(e)
    return np.concatenate([e, -e])


def significands(rng, n, lo, hi):
    return np.ldexp(1.0 + rng.integers(0, 1 << 52, n) / 2.0 ** 52, rng.integers(lo, hi + 1, n))


def near_ones(rng, n, lo, hi):
    """significands a few units below 2: the hard reciprocals, all ones among them"""
    return np.ldexp(2.0 - (1 + rng.integers(0, 64, n)) / 2.0 ** 52, rng.integers(lo, hi + 1, n))


def pairs(rng):
    s = specials()
    bits = [rng.integers(0, 1 << 64, N, dtype=np.uint64).view(np.float64) for _ in range(2)]
    yield "specials", np.repeat(s, s.size), np.tile(s, s.size)
    yield "patterns", bits[0], bits[1]
    yield "special dividends", np.tile(s, N // s.size), significands(rng, N // s.size * s.size, -102, 102)
    yield "ordinary", significands(rng, N, -30, 30) * rng.choice([-1.0, 1.0], N), significands(rng, N, -30, 30)
    yield "wide", significands(rng, N, -702, 702) * rng.choice([-1.0, 1.0], N), significands(rng, N, -102, 102)
    yield "near ones", significands(rng, N, -5, 5), near_ones(rng, N, -100, 99)
    b = significands(rng, N, -3, 3)
    q = significands(rng, N, -3, 3)
    yield "nearly exact", q * b, b  # quotients within an ulp of q: the residual is small or zero
    yield "nearly halfway", b * (q + np.spacing(q) / 2) + rng.integers(-2, 3, N) * np.spacing(q * b), b


@pytest.mark.parametrize("what", [0, 1], ids=["reciprocal", "quotient"])
def test_reciprocal_and_quotient(lib, what):
    rng = np.random.default_rng(10 + what)
    with np.errstate(all="ignore"):
        for name, a, b in pairs(rng):
            n, first = differ(lib, what, a, b)
            assert n == 0, (name, n, first)


def test_integer_products(lib):
    rng = np.random.default_rng(12)
    with np.errstate(all="ignore"):
        for name, a, b in pairs(rng):
            n, first = differ(lib, 2, a, b)
            assert n == 0, (name, n, first)
    # 27 x 27 odd bits: 53- and 54-bit products, the latter exact ties; and 26 x 28
    for wa, wb in ((27, 27), (26, 28), (20, 34), (53, 1)):
        a = np.ldexp((rng.integers(1 << (wa - 1), 1 << wa, N) | 1).astype(np.float64), rng.integers(-300, 300, N))
        b = np.ldexp((rng.integers(1 << (wb - 1), 1 << wb, N) | 1).astype(np.float64), rng.integers(-300, 300, N))
        n, first = differ(lib, 2, a, b)
        assert n == 0, (wa, wb, n, first)


def test_exponentials(lib):
    rng = np.random.default_rng(13)
    s = specials()
    for a, b in ((np.repeat(s, s.size), np.tile(s, s.size)), (rng.uniform(-720, 720, N), rng.uniform(-720, 720, N)),
                 (rng.uniform(-40, 40, N), rng.normal(size=N) * 1e-8),
                 (np.log(2.0) * rng.integers(-1000, 1000, N) * (1 + rng.integers(-3, 4, N) * 2.0 ** -52),
                  np.log(2.0) * (rng.integers(-1000, 1000, N) + 0.5)),
                 (rng.integers(0, 1 << 64, N, dtype=np.uint64).view(np.float64), rng.uniform(-1, 1, N))):
        n, first = differ(lib, 3, a, b)
        assert n == 0, (n, first)


def test_logarithm_comparisons_and_roots(lib):
    rng = np.random.default_rng(14)
    s = specials()
    k = rng.integers(1, 1 << 31, N).astype(np.float64)
    for what in (4, 5, 6):
        for a, b in ((np.repeat(s, s.size), np.tile(s, s.size)),
                     tuple(rng.integers(0, 1 << 64, N, dtype=np.uint64).view(np.float64) for _ in range(2)),
                     (significands(rng, N, -2, 2), significands(rng, N, -2, 2)),
                     (np.sqrt(0.5) * (1 + rng.integers(-4, 5, N) * 2.0 ** -52), k),
                     (np.exp(rng.uniform(0, 43, N)), k), (k * k - 1 + rng.integers(-1, 2, N), k)):
            n, first = differ(lib, what, a, b)
            assert n == 0, (what, n, first)


def test_a_negative_zero_keeps_its_sign(lib):
    b = np.array([1.0, 3.0, 0.1, 2.0 ** 100, 2.0 ** -100, 1e30])
    for z in (0.0, -0.0):
        assert differ(lib, 1, np.full(b.size, z), b)[0] == 0
        assert differ(lib, 1, np.full(b.size, z), -b)[0] == 0
