"""The exponent words of fixed-point blocks (csrc/fixed.cuh) on the host: halves, marks, halves that lie near."""

import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include "fixed.cuh"
using namespace dwf;
extern "C" {
int word(int p, int m) { return fx_word(p, m); }
int half(int w, int chi) { return chi ? fx_half<1>(w) : fx_half<0>(w); }
int is_raw(int w) { return fx_is_raw(w); }
int near_word(int p, int m) { fx_near(p, m); return fx_word(p, m); }
}
"""
RAW, ZERO, NEAR = 0x4000, -0x4000, 4


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    d = tmp_path_factory.mktemp("fxh")
    (d / "fx.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2602_14454_gb300", "csrc"),
                    "-o", str(d / "fx.so"), str(d / "fx.cpp")], check=True)
    return ctypes.CDLL(str(d / "fx.so"))


EXPONENTS = [ZERO, -6000, -1074, -2, -1, 0, 1, 5, 1024, 6000]


@pytest.mark.parametrize("p", EXPONENTS)
@pytest.mark.parametrize("m", EXPONENTS)
def test_words(fx, p, m):
    w = fx.word(p, m)
    assert (fx.half(w, 0), fx.half(w, 1)) == (p, m) and not fx.is_raw(w) and w < fx.word(RAW, RAW)
    n = fx.near_word(p, m)
    want = (max(p, m),) * 2 if abs(p - m) <= NEAR else (p, m)
    assert (fx.half(n, 0), fx.half(n, 1)) == want
    assert fx.is_raw(max(w, fx.word(RAW, RAW)))


def test_near_bound(fx):
    for d in (NEAR, NEAR + 1):
        assert fx.half(fx.near_word(7, 7 - d), 1) == (7 if d <= NEAR else 7 - d)
        assert fx.half(fx.near_word(7 - d, 7), 0) == (7 if d <= NEAR else 7 - d)
