"""The fixed-point arithmetic of the FP64 kernels (csrc/fixed.cuh) on the host, against exact integers."""

import ctypes
import math
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include "fixed.cuh"
using namespace dwf;
extern "C" {
int block_exponent(const double *x, int n)
{
    uint32_t m = 0, low = 0;
    for (int k = 0; k < n; ++k) {
        const int64_t b = fx_bits_of(x[k]);
        const uint32_t h = (uint32_t)(b >> 32) & 0x7fffffffu;
        if (h > m) m = h;
        low |= (uint32_t)b;
    }
    return fx_exponent(m, low);
}
int64_t from_double(double x, int e, int B) { return fx_from_double(x, e, B); }
double to_double(int64_t r, int s) { return fx_to_double(r, s); }
void limbs(int64_t x, int kind, int32_t *l, int32_t *h)
{
    if (kind == 0) fx_limbs31(x, *l, *h);
    else if (kind == 1) fx_limbs31s(x, *l, *h);
    else fx_limbs29(x, *l, *h);
}
int64_t product(int64_t a, int64_t b, int kind_a, int kind_b, int shift)
{
    int32_t al, ah, bl, bh;
    limbs(a, kind_a, &al, &ah);
    limbs(b, kind_b, &bl, &bh);
    int64_t hh = 0, x = (int64_t)1 << (shift - 1);
    fx_mad(al, ah, bl, bh, hh, x);
    return hh + (x >> shift);
}
int64_t align(int64_t v, int bits, int down) { return fx_align(v, bits, down); }
}
"""


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    (d / "fx.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2602_14454_gb300", "csrc"),
                    "-o", str(d / "fx.so"), str(d / "fx.cpp")], check=True)
    L = ctypes.CDLL(str(d / "fx.so"))
    i, q, r = ctypes.c_int, ctypes.c_int64, ctypes.c_double
    L.block_exponent.argtypes = [ctypes.POINTER(r), i]
    L.from_double.argtypes, L.from_double.restype = [r, i, i], q
    L.to_double.argtypes, L.to_double.restype = [q, i], r
    L.limbs.argtypes = [q, i, ctypes.POINTER(ctypes.c_int32), ctypes.POINTER(ctypes.c_int32)]
    L.product.argtypes, L.product.restype = [q, q, i, i, i], q
    L.align.argtypes, L.align.restype = [q, i, i], q
    return L


def exponent(fx, xs):
    return fx.block_exponent((ctypes.c_double * len(xs))(*xs), len(xs))


EDGE = [5e-324, 2.0 ** -1022, 1.0, 1.0 - 2.0 ** -53, 2.0, 1.7976931348623157e308]


def test_blocks(fx):
    rng = random.Random(1)
    for trial in range(300):
        xs = [rng.gauss(0, 1) * 2.0 ** rng.randint(-20, 0) * 2.0 ** rng.randint(-900, 900) for _ in range(24)]
        xs = [x * 0 if rng.random() < 0.1 else x for x in xs] if trial else EDGE
        e = exponent(fx, xs)
        top = max(abs(x) for x in xs)
        assert math.frexp(top)[1] == e or top < 2.0 ** -1022
        for x in xs:
            for B in (57, 58, 59):
                F = fx.from_double(x, e, B)
                m, k = math.frexp(x)
                n = int(m * 2 ** 53)
                want = n << (k - 53 + B - e) if k - 53 + B - e >= 0 else abs(n) >> (e - B + 53 - k)
                assert abs(F) == abs(want) and (F == 0 or (F < 0) == (x < 0)), (x, e, B)
    assert exponent(fx, [0.0, -0.0]) == -0x4000
    assert exponent(fx, [1.0, math.inf]) == exponent(fx, [math.nan, 0.0]) == 0x4000


def test_to_double_rounds_once(fx):
    rng = random.Random(2)
    for _ in range(20000):
        R = rng.getrandbits(63) >> rng.randint(0, 62)
        R = -R if rng.random() < 0.5 else R
        s = rng.randint(-900, 900)
        assert fx.to_double(R, s) == math.ldexp(float(R), s)   # int -> float rounds to nearest even
    for R in (0, 1, -1, 2 ** 53 + 1, 2 ** 54 + 2, 2 ** 54 + 6, 2 ** 62 - 1, -(2 ** 62)):
        assert fx.to_double(R, 3) == float(R) * 8
    assert fx.to_double(3, -1074) == 3 * 5e-324 and fx.to_double(1, 1100) == math.inf


@pytest.mark.parametrize("kind,radix,bits", [(0, 31, 60), (1, 31, 60), (2, 29, 58)])
def test_limbs(fx, kind, radix, bits):
    rng = random.Random(3)
    l, h = ctypes.c_int32(), ctypes.c_int32()
    for x in [0, 1, -1, 2 ** (radix - 1), 2 ** (radix - 1) - 1, -2 ** (radix - 1), 2 ** radix - 1, 2 ** bits - 1,
              -2 ** bits] + [rng.randint(-2 ** bits, 2 ** bits) for _ in range(2000)]:
        fx.limbs(x, kind, ctypes.byref(l), ctypes.byref(h))
        assert h.value * 2 ** radix + l.value == x
        assert (0 <= l.value) if kind == 0 else (-2 ** (radix - 1) <= l.value < 2 ** (radix - 1))


@pytest.mark.parametrize("ka,kb,radix,ba,bb", [(0, 1, 31, 60, 59), (2, 2, 29, 58, 58)])
def test_products(fx, ka, kb, radix, ba, bb):
    """hi hi + cross products rounded at 2^radix: off by half a unit and the dropped lo lo, below one unit."""
    rng = random.Random(4)
    for _ in range(5000):
        a, b = rng.randint(-2 ** ba, 2 ** ba), rng.randint(-2 ** bb, 2 ** bb)
        got = fx.product(a, b, ka, kb, radix)
        assert abs(got * 2 ** (2 * radix) - a * b) <= 2 ** (2 * radix - 1) + 2 ** (2 * radix - 1)


def test_align(fx):
    for v in (1, -1, 2 ** 40 + 3, -(2 ** 62), 2 ** 62 - 1):
        bits = (v ^ (v >> 63)).bit_length()
        bits = max(bits, 1)
        for down in (4, 5, 30, 63, 90):
            assert fx.align(v, bits, down) == (v << (63 - bits)) >> min(down, 63)
