"""The integer arithmetic of csrc/fixed_point.cuh, compiled for the host,
against exact rational arithmetic: conversion truncates and shifts round as
they say, and a row of products keeps the bound that the header states."""
import ctypes
import math
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_1601_06681_gb300 import build

SRC = r"""
#include "fixed_point.cuh"
using namespace ehdg;
extern "C" long long t_from_double(double x, int emax) { return fx_from_double(x, emax); }
extern "C" long long t_shift(long long v, int s) { return fx_shift(v, s); }
extern "C" long long t_row(int n, const long long* c, const long long* x) {
  Acc t(0);
  for (int i = 0; i < n; ++i) {
    const Limb l = fx_split(c[i]);
    t.mac(Cfx{l.h, l.l}, fx_limb(fx_pack(fx_split(x[i]))));
  }
  return t.get();
}
"""


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    src, so = str(d / "fx.cu"), str(d / "fx.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run([build.nvcc(), "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", build.CSRC]
                   + build.ARCH + ["-o", so, src], check=True)
    lib = ctypes.CDLL(so)
    lib.t_from_double.argtypes = [ctypes.c_double, ctypes.c_int]
    lib.t_shift.argtypes = [ctypes.c_longlong, ctypes.c_int]
    P = ctypes.POINTER(ctypes.c_longlong)
    lib.t_row.argtypes = [ctypes.c_int, P, P]
    for f in (lib.t_from_double, lib.t_shift, lib.t_row):
        f.restype = ctypes.c_longlong
    return lib


def biased(x):
    """The exponent field of x, that of zero and the subnormals counted as 1."""
    return max(1, math.frexp(x)[1] + 1022) if x else 1


def test_conversion_truncates_below_a_unit(fx):
    rng = np.random.default_rng(0)
    xs = [0.0, -0.0, 1.0, -1.0, 5e-324, -2.5e-308, 1.7e308] + list(
        rng.standard_normal(500) * 2.0 ** rng.integers(-80, 3, 500))
    for x in xs:
        for up in (0, 1, 3, 4, 17, 55, 57, 58, 63, 200):
            emax = biased(x) + up
            got = fx.t_from_double(x, emax)
            want = Fraction(x) / Fraction(2) ** (emax - 1078)
            assert got == math.trunc(want) and abs(got) < 1 << 56, (x, up)
            assert up > 3 or got == want


def test_shift_rounds_and_keeps_zero(fx):
    rng = np.random.default_rng(1)
    for v in [0, 1, -1, (1 << 61) - 1, 1 - (1 << 61)] + [int(i) for i in rng.integers(-2**60, 2**60, 200)]:
        for s in list(range(0, 64)) + [70, 1000, 40000]:
            got = fx.t_shift(v, s)
            assert abs(got - Fraction(v, 1 << s)) <= Fraction(1, 2), (v, s)
            if v == 0:
                assert got == 0


@pytest.mark.parametrize("n", [1, 8, 28, 64, 108])
def test_row_keeps_the_stated_bound(fx, n):
    rng = np.random.default_rng(n)
    arr = lambda v: (ctypes.c_longlong * n)(*v)   # noqa: E731
    for rep in range(40):
        # coefficients below 2 with a sum of magnitudes below 32, some far below the largest
        c = rng.uniform(-2, 2, n) * 2.0 ** -rng.integers(0, 1 + 20 * (rep % 3), n)
        c *= min(1.0, 31.9 / np.abs(c).sum())
        x = rng.standard_normal(n) * 2.0 ** -rng.integers(0, 1 + 20 * (rep % 2), n)
        emax = max(biased(v) for v in x)
        C = [round(Fraction(v) * 2 ** 56) for v in c]
        X = [fx.t_from_double(v, emax) for v in x]
        got = fx.t_row(n, arr(C), arr(X))
        exact = sum(Fraction(a) * Fraction(b) for a, b in zip(c, x)) / Fraction(2) ** (emax - 1078)
        bound = np.abs(c).sum() + 0.75 * n + 0.5
        assert abs(got - exact) <= bound
