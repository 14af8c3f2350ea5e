"""The bounds a decode task is held to (csrc/decode_task.h), compiled for the host."""
import ctypes as C
import subprocess

import numpy as np
import pytest

from paper_2207_05022_b200 import build

SOURCE = """
#include "decode_task.h"
extern "C" int place(int narrow, uint32_t origin, uint32_t rc, uint32_t* row, uint32_t* col) {
  sti::DecodeTask t{};
  t.narrow = static_cast<uint8_t>(narrow);
  t.origin = origin;
  return sti::outlier_place(t, rc, *row, *col);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("decode_task")
    (d / "probe.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", build.CSRC, str(d / "probe.cpp"), "-o", str(d / "probe.so")], check=True)
    so = C.CDLL(str(d / "probe.so"))
    so.place.argtypes = [C.c_int, C.c_uint32, C.c_uint32, C.POINTER(C.c_uint32), C.POINTER(C.c_uint32)]
    return so


@pytest.mark.parametrize("narrow,row0,col0", [(0, 0, 0), (0, 32, 128), (0, 992, 896), (1, 0, 0), (1, 64, 0), (1, 960, 0)])
def test_an_outlier_is_placed_inside_its_task_or_not_at_all(lib, narrow, row0, col0):
    rows, cols = (64, 64) if narrow else (32, 128)
    row, col = C.c_uint32(), C.c_uint32()
    edges_r = {0, 1, row0 - 1, row0, row0 + 1, row0 + rows - 1, row0 + rows, row0 + 2 * rows, 0xffff}
    edges_c = {0, 1, col0 - 1, col0, col0 + 1, col0 + cols - 1, col0 + cols, col0 + 2 * cols, 0xffff}
    rng = np.random.default_rng(row0 + col0)
    pairs = [(r, c) for r in edges_r for c in edges_c if r >= 0 and c >= 0]
    pairs += [tuple(p) for p in rng.integers(0, 1 << 16, (20000, 2)).tolist()]
    pairs += [(row0 + int(r), col0 + int(c)) for r, c in zip(rng.integers(0, rows, 500), rng.integers(0, cols, 500))]
    for r, c in pairs:
        inside = bool(lib.place(narrow, row0 << 16 | col0, r << 16 | c, C.byref(row), C.byref(col)))
        assert inside == (row0 <= r < row0 + rows and col0 <= c < col0 + cols), (r, c)
        if inside:
            assert (row.value, col.value) == (r - row0, c - col0)
