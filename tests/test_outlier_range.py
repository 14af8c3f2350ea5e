"""The quantizer's search for the fp32 values at the ends of a unit's inlier range (csrc/outlier_range.h), compiled for the host:
it finds them for ordinary units and says so where there are none or they are far away, always from the same few candidates."""
import ctypes as C
import math
import os
import subprocess

import numpy as np
import pytest

from paper_2207_05022_b200 import build

SOURCE = """
#include "outlier_range.h"
extern "C" int outlier(float x, double mu, double inv2var, double c0) { return sti::is_outlier(x, mu, inv2var, c0); }
extern "C" int end(int sign, double mu, double inv2var, double c0, float* t) {       // what a half of a warp does
  unsigned in = 0;
  for (int i = 0; i < sti::kEndCandidates; ++i) in |= (sti::is_outlier(sti::end_candidate(*t, i, sign), mu, inv2var, c0) ? 0u : 1u) << i;
  const int at = sti::end_index(in);
  if (at >= 0) *t = sti::end_candidate(*t, at, sign);
  return at >= 0;
}
extern "C" float candidate(float t, int i, int sign) { return sti::end_candidate(t, i, sign); }
extern "C" int index(unsigned inliers) { return sti::end_index(inliers); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("outlier_range")
    (d / "probe.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", build.CSRC, str(d / "probe.cpp"), "-o", str(d / "probe.so")], check=True)
    so = C.CDLL(str(d / "probe.so"))
    so.outlier.argtypes = [C.c_float] + [C.c_double] * 3
    so.end.argtypes = [C.c_int] + [C.c_double] * 3 + [C.POINTER(C.c_float)]
    so.candidate.argtypes, so.candidate.restype = [C.c_float, C.c_int, C.c_int], C.c_float
    return so


def _search(lib, mu, var):
    """(smallest, largest) inlier as the kernel looks for them, None for an end that was given up; and the test's parameters."""
    c0, inv2var = -0.5 * math.log(2.0 * math.pi * var), 1.0 / (2.0 * var)
    radius = math.sqrt(2.0 * var * (c0 + 4.0))
    ends = []
    for sign in (-1, 1):
        t = C.c_float(mu + sign * radius)
        ends.append(t.value if lib.end(sign, mu, inv2var, c0, C.byref(t)) else None)
    return ends, (mu, inv2var, c0)


@pytest.mark.parametrize("mu", [0.0, 1e-6, -0.013, 3.0, -250.0])
@pytest.mark.parametrize("sigma", [1e-5, 1e-3, 0.02, 0.5, 4.0, 13.0, 16.0, 21.0])
def test_finds_the_ends_of_the_range(lib, mu, sigma):
    (least, most), p = _search(lib, mu, sigma * sigma)
    assert least is not None and most is not None and least <= most
    for end, away in ((least, -np.inf), (most, np.inf)):
        assert not lib.outlier(end, *p)
        assert lib.outlier(float(np.nextafter(np.float32(end), np.float32(away))), *p)


@pytest.mark.parametrize("mu,var", [
    (3.0e8 + 16, 256.0),                   # fp32 values 32 apart around the mean, all outside a radius of 12.6
    (-3.0e8 - 16, 256.0),
    (1.0e15, 300.0),
])
def test_gives_up_where_no_value_passes(lib, mu, var):
    (least, most), _ = _search(lib, mu, var)
    assert least is None and most is None


def test_gives_up_where_the_ends_are_millions_of_values_away(lib):
    # a deviation at which the radius is the difference of two nearly equal numbers, about a mean of zero: what passes ends
    # at about 1.4 times the computed radius, half an exponent's worth of fp32 values away
    var = math.exp(8.0) / (2.0 * math.pi)
    while -0.5 * math.log(2.0 * math.pi * var) + 4.0 <= 0.0:
        var = math.nextafter(var, 0.0)
    (least, most), p = _search(lib, 0.0, var)
    for end in (least, most):
        assert end is None or not lib.outlier(end, *p)
    assert least is None and most is None


@pytest.mark.parametrize("t", [1.5, -1.5, 1.0, -2.0, 0.0, -0.0, 1e-45, -3e-45, 1.1754944e-38, 3.0e38])
def test_candidates_are_consecutive_values(lib, t):
    for sign in (-1, 1):
        vals = np.array([lib.candidate(t, i, sign) for i in range(16)], np.float32)
        assert vals[8] == np.float32(t)
        steps = [np.nextafter(a, np.float32(sign * np.inf)) == b or (a == 0 and b == 0) for a, b in zip(vals[:-1], vals[1:])]
        assert all(steps)


def test_end_index(lib):
    for mask in range(1 << 16):
        assert lib.index(mask) == (mask.bit_length() - 1 if 0 < mask < 1 << 15 else -1)
