"""The buckets of the ranking kernels (bucket_map.cuh), every layout there is, on the CPU: the header is plain C++."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = r"""
#include "bucket_map.cuh"
using namespace madakv;
// Buckets of the layout of `rows` window rows whose fine part begins at t0 that do not hold exactly the keys between their start
// and the next one's, or whose start does not follow from that of their group of eight.
extern "C" int misplaced(uint32_t t0, int rows) {
  const BucketMap g = bucket_map_from(t0, rows);
  int bad = map_bucket(g, 0u) != 0u || map_bucket(g, kTopKey) != (uint32_t)kBuckets - 1u;
  for (int b = 0; b < kBuckets; ++b) {
    const BucketStart s = bucket_start(g, b), first = bucket_start(g, b & ~7);
    const uint32_t end = b + 1 < kBuckets ? bucket_start(g, b + 1).t : kTopKey + 1u;
    bool ok = s.t < end && map_bucket(g, s.t) == (uint32_t)b && map_bucket(g, end - 1u) == (uint32_t)b;
    ok = ok && map_bucket(g, s.t + (end - s.t) / 2u) == (uint32_t)b;
    ok = ok && (b == 0 || map_bucket(g, s.t - 1u) == (uint32_t)b - 1u);
    ok = ok && s.shift == first.shift && s.t == first.t + ((uint32_t)(b & 7) << s.shift);
    ok = ok && (b + 1 == kBuckets || end == s.t + (1u << s.shift));
    bad += !ok;
  }
  return bad;
}
extern "C" uint32_t t_of(float score) {
  union { float f; uint32_t u; } x = {score};
  return kTopKey - x.u;
}
extern "C" float top_of(int rows) { return fine_top(rows); }
"""


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    at = tmp_path_factory.mktemp("bucket_map")
    src, out = at / "shim.cpp", at / "shim.so"
    src.write_text(SHIM)
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-fPIC", "-shared", "-I",
                           os.path.join(ROOT, "paper_2506_15724_b200", "csrc"), "-o", str(out), str(src)])
    lib = ctypes.CDLL(str(out))
    lib.t_of.restype, lib.t_of.argtypes = ctypes.c_uint32, [ctypes.c_float]
    lib.top_of.restype, lib.top_of.argtypes = ctypes.c_float, [ctypes.c_int]
    lib.misplaced.argtypes = [ctypes.c_uint32, ctypes.c_int]
    return lib


# up to 127 window rows and from 128 on the fine buckets are differently wide
@pytest.mark.parametrize("rows", [1, 8, 64, 127, 128, 255, 256, 257, 1024, 4096])
def test_every_bucket_holds_the_keys_between_its_edges(shim, rows):
    """A key is counted in the bucket whose range it is later looked for in. The fine part of a layout begins at a multiple of a
    quarter octave; all of them from the mean of one token to that of 2^20, and a bit beyond on both sides."""
    first, last = shim.t_of(rows * 3.0), shim.t_of(rows * 0.5 / (1 << 20))
    layouts = 0
    for t0 in range(first & ~((1 << 21) - 1), last + (1 << 21), 1 << 21):
        assert shim.misplaced(t0, rows) == 0, (rows, hex(t0))
        layouts += 1
    assert layouts > 80
