"""The running sums of csrc/sums.cuh, compiled for the host (no GPU), against exact sums.

Bounds: a triple holds h + m + l with two error-free additions a term; what it drops is the
rounding of l, n 2^-72 sum |x|, and the conversion to FP64 rounds twice (2^-53 of the value each).
The quotient is the FP32 rounding of a value within 2^-46 of the exact one: half an ulp and 2^-22
of it."""
import ctypes as C
import math
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_2511_06788_gb300 import build as B

SRC = r"""
#include "sums.cuh"
using namespace opevo;
// the sum of x in `groups` interleaved sums that are then joined
static Sum3 total(const float *x, int n, int groups) {
  Sum3 s;
  for (int g = 0; g < groups; ++g) {
    Sum3 t;
    for (int i = g; i < n; i += groups) t.add(x[i]);
    s.add(t);
  }
  return s;
}
extern "C" int sum3(const float *x, int n, int groups, double *out) {
  const Sum3 s = total(x, n, groups);
  *out = s.value();
  return s.finite();
}
extern "C" int ratio(const float *x, int n, const float *y, int m, float *q) {
  return quotient(total(x, n, 1), total(y, m, 1), q);
}
"""


@pytest.fixture(scope="module")
def sums(tmp_path_factory):
    d = tmp_path_factory.mktemp("sums")
    src, so = os.path.join(d, "sums_host.cu"), os.path.join(d, "sums_host.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run([B._nvcc(), *B.ARCH, "-std=c++17", "-O2", "-Xcompiler", "-fPIC,-ffp-contract=off",
                    "-I", B.CSRC, "-shared", "-o", so, src], check=True)
    lib = C.CDLL(so)
    return lib


def ptr(x):
    return x.ctypes.data_as(C.POINTER(C.c_float))


def terms(rng, kind, n):
    x = rng.standard_normal(n)
    if kind == "wide":  # 60 binary orders
        x = np.ldexp(x, rng.integers(-30, 30, n))
    if kind == "cancel":  # a sum far below its terms
        x[n // 2:2 * (n // 2)] = -x[:n // 2]
        x[0] *= 1.0 + 2.0**-20
    if kind == "small":  # down to the subnormals
        x = np.ldexp(x, rng.integers(-148, -120, n))
    return x.astype(np.float32)


@pytest.mark.parametrize("kind", ["ordinary", "wide", "cancel", "small"])
@pytest.mark.parametrize("n,groups", [(1, 1), (2, 1), (7, 4), (228, 4), (5000, 16)])
def test_sum_keeps_what_an_fp64_sum_keeps(sums, kind, n, groups):
    rng = np.random.default_rng(n + groups)
    for _ in range(20):
        x = terms(rng, kind, n)
        out = C.c_double()
        assert sums.sum3(ptr(x), n, groups, C.byref(out)) == 1
        exact = sum((Fraction(float(v)) for v in x), Fraction(0))
        mag = sum(abs(Fraction(float(v))) for v in x)
        bound = Fraction(2)**-52 * abs(exact) + (n + groups) * Fraction(2)**-70 * mag + Fraction(2)**-149 * n
        if kind == "small":
            assert Fraction(out.value) == exact or abs(Fraction(out.value) - exact) <= Fraction(2)**-52 * abs(exact)
        assert abs(Fraction(out.value) - exact) <= bound


def test_sums_outside_the_fp32_range_are_reported(sums):
    out = C.c_double()
    for x in ([3e38, 3e38, -3e38], [1.0, math.inf], [math.nan, 1.0], [3e38] * 9):
        x = np.array(x, np.float32)
        assert sums.sum3(ptr(x), len(x), 1, C.byref(out)) == 0
    x = np.array([3e38, -3e38, 2e38], np.float32)
    assert sums.sum3(ptr(x), 3, 1, C.byref(out)) == 1 and out.value == float(x[2])


@pytest.mark.parametrize("scale,of", [(0, 0), (-60, -60), (90, 90), (30, -50), (-50, 30)])
def test_quotient_is_rounded_once(sums, scale, of):
    rng = np.random.default_rng(scale + 200)
    out = C.c_float()
    for _ in range(2000):
        n, m = rng.integers(1, 40, 2)
        x = np.ldexp(rng.random(n) + 2.0**-9, scale).astype(np.float32)
        y = np.ldexp(rng.random(m) + 2.0**-9, of).astype(np.float32)
        assert sums.ratio(ptr(x), int(n), ptr(y), int(m), C.byref(out)) == 1
        q = Fraction(float(out.value))
        exact = sum(Fraction(float(v)) for v in x) / sum(Fraction(float(v)) for v in y)
        ulp = Fraction(2)**(math.frexp(float(exact))[1] - 24)
        assert abs(q - exact) <= ulp * (Fraction(1, 2) + Fraction(2)**-22)


def test_quotient_leaves_the_rest_to_fp64(sums):
    out = C.c_float()
    one = np.ones(1, np.float32)
    for v in (1e-30, 2e30, math.inf, math.nan, 0.0, -1.0):
        x = np.array([v], np.float32)
        assert sums.ratio(ptr(x), 1, ptr(one), 1, C.byref(out)) == 0
    for v in (1e-30, 2e30, math.inf, -math.inf, math.nan):
        x = np.array([v], np.float32)
        assert sums.ratio(ptr(one), 1, ptr(x), 1, C.byref(out)) == 0
    for v in (0.0, -1.0):  # no quotient: 0
        x = np.array([v], np.float32)
        assert sums.ratio(ptr(one), 1, ptr(x), 1, C.byref(out)) == 1 and out.value == 0.0
