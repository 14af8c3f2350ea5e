"""How calls are cut (csrc/tiling.h), compiled for the host: the buffer of partial sums holds the planes of every call that a
context takes, and a matrix has one place in the working buffer whatever a layer keeps."""
import ctypes as C
import subprocess

import pytest

from paper_2207_05022_b200 import build

SOURCE = """
#include "tiling.h"
using namespace sti;
static Tiling tiling(int hidden, int slice, long long max_tokens, const int* tune) {
  Tiling t;
  t.hidden = hidden; t.slice = slice; t.max_tokens = max_tokens;
  t.attn_weights = 4 * 64 * hidden; t.ffn_weights = 2 * slice * hidden;
  t.tune.qkv_n = t.tune.f1_n = t.tune.o_n = t.tune.f2_n = 64;       // as a plan has them
  t.tune.o_group = tune[0]; t.tune.wide_min_tokens = tune[1]; t.tune.cta_budget = tune[2];
  return t;
}
// The first token count whose planes do not fit what is allocated; 0: none.
extern "C" long long overflow(int hidden, int slice, int heads, int slices, long long max_tokens, const int* tune) {
  const Tiling t = tiling(hidden, slice, max_tokens, tune);
  const size_t rows = partial_rows(t, heads, slices);
  for (long long tokens = 1; tokens <= max_tokens; ++tokens) {
    const SumPlanes p = sum_planes(t, heads, slices, tokens);
    if (static_cast<size_t>(tokens) * std::max(p.o, p.f2) > rows) return tokens;
  }
  return 0;
}
extern "C" size_t rows(int hidden, int slice, int heads, int slices, long long max_tokens, const int* tune) {
  return partial_rows(tiling(hidden, slice, max_tokens, tune), heads, slices);
}
extern "C" int wide(int hidden, int slice, int heads, int slices, long long tokens, const int* tune) {
  return use_wide(tiling(hidden, slice, tokens, tune), heads, slices, tokens);
}
// Rows of 128 bytes: where each of the four matrices begins, where what is written of it ends, and the buffer's.
extern "C" unsigned place(int hidden, int slice, const int* units, unsigned* at) {
  const int tune[3] = {8, -1, 148};
  WideMatrix wide[4];
  const unsigned rows = place_wide(tiling(hidden, slice, 1, tune), units[0], units[1], units[2], units[3], wide);
  for (int m = 0; m < 4; ++m) {
    at[2 * m] = wide[m].row0;
    at[2 * m + 1] = wide[m].row0 + (wide[m].n + 255) / 256 * 256 * wide[m].k_chunks;      // a 256-wide tile's boxes reach so far
  }
  return rows;
}
"""
MODELS = {"base": (768, 256, 12), "large": (1024, 256, 16)}
DEFAULT = (8, -1, 148)                           # heads per K group, the rule's own threshold, CTAs


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("tiling")
    (d / "probe.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", build.CSRC, str(d / "probe.cpp"), "-o", str(d / "probe.so")], check=True)
    so = C.CDLL(str(d / "probe.so"))
    args = [C.c_int] * 4 + [C.c_longlong, C.POINTER(C.c_int)]
    so.overflow.argtypes, so.overflow.restype = args, C.c_longlong
    so.rows.argtypes, so.rows.restype = args, C.c_size_t
    so.wide.argtypes = args
    so.place.argtypes = [C.c_int, C.c_int, C.POINTER(C.c_int), C.POINTER(C.c_uint)]
    return so


def _tune(values=DEFAULT):
    return (C.c_int * 3)(*values)


# one sequence of each length class, a few of them, odd and whole numbers of tiles, the largest
@pytest.mark.parametrize("context", [1, 77, 385, 400, 512, 513, 1000, 2048, 1757, 4095, 4096, 32 * 512])
@pytest.mark.parametrize("model", sorted(MODELS))
def test_every_call_s_partial_sums_fit(lib, model, context):
    hidden, slice_, n = MODELS[model]
    for heads in range(n + 1):
        for slices in range(n + 1):
            assert lib.overflow(hidden, slice_, heads, slices, context, _tune()) == 0, (heads, slices)


@pytest.mark.parametrize("tune", [(8, 0, 148), (8, 1, 148), (8, 390, 148), (1, 700, 148), (8, -1, 16), (8, -1, 132)])
def test_whatever_the_settings(lib, tune):
    for heads, slices in ((16, 16), (12, 12), (14, 14), (3, 16), (16, 1)):
        for context in (512, 1500, 4096):
            assert lib.overflow(1024, 256, heads, slices, context, _tune(tune)) == 0, (heads, slices, context)


def test_planes_are_asked_for_where_calls_have_them(lib):
    """The check above is not an empty one: calls of more than one plane, on either side of the working buffer's threshold."""
    assert lib.rows(1024, 256, 12, 12, 384, _tune()) > 384 and not lib.wide(1024, 256, 12, 12, 384, _tune())
    assert lib.rows(1024, 256, 12, 12, 512, _tune()) > 512 and lib.wide(1024, 256, 12, 12, 400, _tune())


@pytest.mark.parametrize("model", sorted(MODELS))
def test_a_matrix_never_stands_where_another_layer_has_a_different_one(lib, model):
    hidden, slice_, n = MODELS[model]
    for most_heads in range(n + 1):
        for most_slices in (0, 1, 5, n):
            places = set()
            for heads in range(most_heads + 1):
                for slices in range(most_slices + 1):
                    at = (C.c_uint * 8)()
                    rows = lib.place(hidden, slice_, (C.c_int * 4)(heads, slices, most_heads, most_slices), at)
                    begin, end = list(at)[0::2], list(at)[1::2]
                    places.add(tuple(begin) + (rows,))
                    assert begin[0] == 0 and all(b % 128 == 0 for b in begin)
                    assert all(e <= limit for e, limit in zip(end, begin[1:] + [rows]))
            assert len(places) == 1
