"""The output scale of the integer A (make_scale, fx_scale of fixed.cuh), compiled for the host:
ca diag^2 as split words against exact rationals, around every power of two that a mass can put
it next to.  The scale holds 62 bits or more (2^-60 of it allowed), its product with a row sum
floors once and leaves out the low words' product (2 units)."""
import ctypes
import math
import random
import subprocess
from fractions import Fraction

import pytest

import __graft_entry__ as G

SRC = r"""
#include "%s/fixed.cuh"
extern "C" void scale(double ca, double diag, int* out) {
  const mgk::FxScale q = mgk::make_scale(ca, diag);
  out[0] = q.lo; out[1] = q.hi; out[2] = q.exp;
}
extern "C" long long apply(long long y, int lo, int hi, int exp) { return mgk::fx_scale(y, mgk::FxScale{lo, hi, exp}); }
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed")
    (d / "t.cu").write_text(SRC % G.CSRC)
    subprocess.run([G._nvcc(), *G.ARCH, "-std=c++17", "-O1", "-shared", "-Xcompiler", "-fPIC", "-o", str(d / "t.so"),
                    str(d / "t.cu")], check=True, capture_output=True)
    L = ctypes.CDLL(str(d / "t.so"))
    L.scale.argtypes = [ctypes.c_double, ctypes.c_double, ctypes.POINTER(ctypes.c_int)]
    L.apply.argtypes = [ctypes.c_longlong, ctypes.c_int, ctypes.c_int, ctypes.c_int]
    L.apply.restype = ctypes.c_longlong
    return L


def _check(L, ca, diag):
    out = (ctypes.c_int * 3)()
    L.scale(ca, diag, out)
    lo, hi, exp = out
    q, want = (hi << 32) + lo, Fraction(ca) * Fraction(diag) ** 2
    got = Fraction(q) * Fraction(2) ** (exp - 64)
    assert abs(got - want) <= abs(want) / 2 ** 60, (ca, diag, float(got), float(want))
    assert abs(q) >= 2 ** 61
    for y in (1, -1, 2 ** 58 + 12345678901, -(2 ** 62) + 987654321):
        assert abs(L.apply(y, lo, hi, exp) - Fraction(y * q, 2 ** 64)) <= 2, (ca, diag, y)


def _neighbours(v):
    out, a, b = [v], v, v
    for _ in range(1000):
        a, b = math.nextafter(a, 0.0), math.nextafter(b, math.inf)
        out += [a, b]
    return out + [v + s * 10.0 ** -k for k in range(9, 13) for s in (-1, 1)]


@pytest.mark.parametrize("centre", [1.5, 2.0, math.sqrt(2) * 2, 4.0, math.sqrt(2) * 4, 8.0, 16.0, 32.0, 64.0])
def test_next_to_powers_of_two(host, centre):
    for diag in _neighbours(centre):
        for ca in (1.0, -1.0):
            _check(host, ca, diag)


def test_masses_reached_in_steps(host):
    for start, step, n in ((-2.5, 0.05, 60), (0.0, -0.1, 24), (0.5, -0.05, 60)):
        m = start
        for _ in range(n):
            _check(host, 1.0, 4.0 + m)
            m += step
    for m in (-2.0000000000000004, -2.0000000000000018, -4.5e-16, -1e-15, -2.0000000001):
        _check(host, 1.0, 4.0 + m)


def test_epilogue_factors(host):
    rng = random.Random(5)
    for _ in range(4000):
        diag = rng.uniform(1.5, 64.0)
        _check(host, rng.choice([-1, 1]) * 2.0 ** rng.uniform(-40, 10), diag)
        near = 2.0 ** rng.randint(-30, 10) / diag ** 2        # ca diag^2 just below and above a power of two
        for ca in (near, math.nextafter(near, 0.0), math.nextafter(near, 1e300), near * (1 - 1e-10)):
            _check(host, ca, diag)
            _check(host, -ca, diag)
