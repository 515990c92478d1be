"""The FP32 sums of csrc/sums.cuh, compiled for the host: their error against exact sums,
and what they do with overflows and NaN."""
import ctypes as C
import math
import os
import subprocess

import numpy as np
import pytest

from conftest import ROOT

SRC = r"""
#include "sums.cuh"
extern "C" double sum2(const float* v, int n) {  // one after the other, as rows and tiles
  Sum2 a = {0.f, 0.f};
  for (int i = 0; i < n; ++i) sum2_add(a, v[i]);
  return sum2_value(a);
}
extern "C" double lanes(const float* v) {  // the exchange pattern of warp_sum(Sum2)
  Sum2 a[32], b[32];
  for (int i = 0; i < 32; ++i) a[i] = {v[i], 0.f};
  for (int o = 16; o > 0; o >>= 1) {
    for (int i = 0; i < 32; ++i) { b[i] = a[i]; sum2_add(b[i], a[i ^ o]); }
    for (int i = 0; i < 32; ++i) a[i] = b[i];
  }
  return sum2_value(a[0]);
}
extern "C" int depth(int n) { return tree_depth(n); }
template <int N> float tree(const float* v) {
  float t[N];
  for (int i = 0; i < N; ++i) t[i] = v[i];
  tree_sum(t, [](float x, float y) { return x + y; });
  return t[0];
}
extern "C" float trees(int n, const float* v) {
  return n == 1 ? tree<1>(v) : n == 2 ? tree<2>(v) : n == 3 ? tree<3>(v) : n == 4 ? tree<4>(v) : n == 6 ? tree<6>(v) : tree<32>(v);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("sums")
    (d / "s.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-D__host__=", "-D__device__=",
                    "-D__forceinline__=inline", "-Wno-unknown-pragmas", "-I",
                    os.path.join(ROOT, "paper_2606_17850_gb300", "csrc"), str(d / "s.cpp"), "-o", str(d / "s.so")],
                   check=True)
    lib = C.CDLL(str(d / "s.so"))
    fp = C.POINTER(C.c_float)
    lib.sum2.argtypes, lib.sum2.restype = [fp, C.c_int], C.c_double
    lib.lanes.argtypes, lib.lanes.restype = [fp], C.c_double
    lib.trees.argtypes, lib.trees.restype = [C.c_int, fp], C.c_float
    return lib


def _p(v):
    return v.ctypes.data_as(C.POINTER(C.c_float))


U = 2.0 ** -24


def _sets(n):
    rng = np.random.default_rng(n)
    small = np.full(n, 2.0 ** -25.5, np.float32)
    small[0] = 1.0                                    # every later term is lost by a plain sum
    return {"small": small, "same": np.full(n, 1.0 / 3, np.float32),
            "squares": (rng.standard_normal(n) ** 2).astype(np.float32),
            "signed": (rng.standard_normal(n) * 10.0 ** rng.uniform(-6, 6, n)).astype(np.float32)}


@pytest.mark.parametrize("n", [1, 2, 12, 32, 100, 256, 1024])
def test_long_sums_keep_their_rounding_errors(lib, n):
    """Error at most (n u)^2 sum |v| (the FP32 sum of n errors of at most u times a partial
    sum each) plus one FP64 rounding; a plain FP32 sum is far outside on the small terms."""
    for name, v in _sets(n).items():
        exact, mag = math.fsum(v.tolist()), math.fsum(np.abs(v).tolist())
        bound = (n * U) ** 2 * mag + 2.0 ** -52 * mag
        assert abs(lib.sum2(_p(v), n) - exact) <= bound, name
        if n == 32:
            assert abs(lib.lanes(_p(v)) - exact) <= bound, name
        if name == "small" and n >= 12:
            plain = np.float32(0)
            for x in v:
                plain = np.float32(plain + x)
            assert abs(float(plain) - exact) > 100 * bound


@pytest.mark.parametrize("n", [1, 2, 3, 4, 6, 32])
def test_tree_of_a_column(lib, n):
    """At most ceil(log2 n) roundings on the way of any term (tree_depth)."""
    v = _sets(n)["signed"]
    exact, mag = math.fsum(v.tolist()), math.fsum(np.abs(v).tolist())
    assert lib.depth(n) == math.ceil(math.log2(n))
    assert abs(lib.trees(n, _p(v)) - exact) <= 1.01 * math.ceil(math.log2(n)) * U * mag


def test_overflow_and_nan_stay(lib):
    v = np.zeros(32, np.float32)
    v[3] = v[9] = 3e38
    assert lib.sum2(_p(v), 32) == math.inf and lib.lanes(_p(v)) == math.inf
    v[9] = np.inf
    assert lib.sum2(_p(v), 32) == math.inf and lib.lanes(_p(v)) == math.inf
    v[20] = np.nan
    assert math.isnan(lib.lanes(_p(v))) and math.isnan(lib.sum2(_p(v), 32))
