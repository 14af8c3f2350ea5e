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
extern "C" int in_bounds(const uint32_t* f, uint32_t n_rows, uint32_t k_total, size_t bytes) {
  sti::DecodeTask t{};
  const uint8_t* unit = reinterpret_cast<const uint8_t*>(4096);       // never followed
  t.codes = unit + static_cast<int32_t>(f[0]);
  t.table = f[1]; t.out_rc = f[2]; t.out_val = f[3];
  t.n_out = static_cast<uint16_t>(f[4]); t.bits = static_cast<uint8_t>(f[5]); t.narrow = static_cast<uint8_t>(f[6]);
  t.row0 = static_cast<uint16_t>(f[7]); t.kcore0 = static_cast<uint16_t>(f[8]);
  return sti::task_in_bounds(t, n_rows, k_total, unit, bytes);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("decode_task")
    (d / "probe.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", build.CSRC, str(d / "probe.cpp"), "-o", str(d / "probe.so")], check=True)
    so = C.CDLL(str(d / "probe.so"))
    so.place.argtypes = [C.c_int, C.c_uint32, C.c_uint32, C.POINTER(C.c_uint32), C.POINTER(C.c_uint32)]
    so.in_bounds.argtypes = [C.POINTER(C.c_uint32), C.c_uint32, C.c_uint32, C.c_size_t]
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


# a unit of 64 x 256 weights at 3 bits: 6144 bytes of indexes, 32 of table, nine outliers
UNIT = dict(codes=1536, table=6144 - 1536, out_rc=6176 - 1536, out_val=6224 - 1536, n_out=9, bits=3, narrow=0, row0=32, kcore0=16)
UNIT_BYTES = 6272
RAW = dict(codes=512, table=0, out_rc=0, out_val=1024, n_out=0, bits=32, narrow=0, row0=0, kcore0=0)


def _in_bounds(lib, task, bytes_, n_rows=64, k_total=256):
    names = ("codes", "table", "out_rc", "out_val", "n_out", "bits", "narrow", "row0", "kcore0")
    return bool(lib.in_bounds((C.c_uint32 * 9)(*[task[k] & 0xffffffff for k in names]), n_rows, k_total, bytes_))


def test_tasks_that_stay_inside_are_taken(lib):
    assert _in_bounds(lib, UNIT, UNIT_BYTES)
    assert _in_bounds(lib, dict(UNIT, codes=0, table=6144, out_rc=6176, out_val=6224, row0=0, kcore0=0), UNIT_BYTES)
    assert _in_bounds(lib, dict(UNIT, codes=4608, table=1536, out_rc=6176 - 4608, out_val=6224 - 4608), UNIT_BYTES)     # the last task
    assert _in_bounds(lib, RAW, 32 * 1024)                                        # rows 0..31, columns 128..255
    assert _in_bounds(lib, dict(UNIT, narrow=1, row0=0, kcore0=24), UNIT_BYTES)


@pytest.mark.parametrize("change", [
    dict(codes=-16), dict(codes=6144), dict(codes=1544), dict(codes=UNIT_BYTES + 16), dict(table=UNIT_BYTES - 1536 - 16), dict(table=0xffffff00),
    dict(table=4610), dict(out_rc=UNIT_BYTES - 1536 - 32), dict(out_val=UNIT_BYTES - 1536 - 32), dict(out_val=0xfffffffc), dict(n_out=13),
    dict(bits=0), dict(bits=1), dict(bits=7), dict(bits=6, codes=4608), dict(row0=33), dict(row0=64), dict(kcore0=17), dict(kcore0=0xffff),
    dict(narrow=1), dict(narrow=1, row0=0, kcore0=25)])
def test_tasks_that_do_not_are_refused(lib, change):
    assert not _in_bounds(lib, dict(UNIT, **change), UNIT_BYTES)


@pytest.mark.parametrize("change", [dict(codes=1024), dict(out_val=1040), dict(out_val=0xfffffff0), dict(n_out=1), dict(codes=-512)])
def test_uncompressed_tasks_that_do_not_are_refused(lib, change):
    assert not _in_bounds(lib, dict(RAW, **change), 32 * 1024)
