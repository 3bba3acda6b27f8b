"""The buckets of the ranking kernels (bucket_map.cuh), every layout there is, on the CPU: the header is plain C++."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = r"""
#include <initializer_list>
#include "bucket_map.cuh"
using namespace madakv;
// Buckets of the layout of `rows` window rows whose fine part begins at t0 that do not hold exactly the keys between their start
// and the next one's, or whose start does not follow from that of their group of eight. (0 rows: of the plain layout.)
template <typename Map>
static int misplaced_in(const Map& g) {
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
extern "C" int misplaced(uint32_t t0, int rows) { return rows ? misplaced_in(bucket_map_from(t0, rows)) : misplaced_in(PlainMap()); }
// Buckets whose mass does not come out right from the words of its keys, for as many keys as mass_known() takes, or that take
// fewer than they have to: one key of any score, and of scores from 2^-9 on as many as 2^32 over the bucket's width. Of a
// layout over [t, t + 2^(11 + shift)) too.
static int wrong(const BucketStart& s, int x, int b) {
  const uint32_t first = s.t + ((uint32_t)x << s.shift), last = bucket_last(s, x, b), at[3] = {first, last, first + (last - first) / 3u};
  const MassRule rule = mass_rule(s.t);
  int bad = mass_rule(last).up != rule.up || mass_rule(last).linear != rule.linear || !mass_known(rule, 1, first, last);
  uint32_t most = 1;
  while (most < (1u << 20) && mass_known(rule, 2 * most, first, last)) most *= 2;
  for (uint32_t step = most / 4; step > 0; step /= 2)
    if (mass_known(rule, most + step, first, last)) most += step;
  if (rule.linear && most < (1u << (31 - s.shift)) && most < (1u << 20)) ++bad;
  for (uint32_t c : {1u, 2u, most}) {
    if (!mass_known(rule, c, first, last)) continue;
    for (int kind = 0; kind < 7; ++kind) {  // all alike, two values half and half, all three
      uint32_t n[3] = {0, 0, 0}, sum = 0;
      unsigned long long want = 0;
      if (kind < 3) n[kind] = c;
      else if (kind < 6) n[kind - 3] = c / 2, n[(kind - 2) % 3] = c - c / 2;
      else n[0] = c / 3, n[1] = c / 3, n[2] = c - 2 * (c / 3);
      for (int k = 0; k < 3; ++k) {
        sum += n[k] * mass_word(at[k]);
        want += n[k] * (unsigned long long)((double)score_of(at[k]) * 4294967296.0);
      }
      bad += mass_sum(rule, c, sum, last) << rule.up != want;
    }
  }
  return bad;
}
extern "C" int wrong_masses(uint32_t t0, int rows) {
  const BucketMap g = bucket_map_from(t0, rows);
  int bad = 0;
  for (int b = 1; b < kBuckets; ++b) bad += wrong(bucket_start(g, b & ~7), b & 7, b);
  for (int b = 1; b < kBuckets - 1; b += 13) {
    const BucketStart s = bucket_start(g, b);
    for (int x : {0, 8, 1024, 2040}) {
      const BucketStart in = {s.t + ((uint32_t)x << (s.shift - 11)), s.shift - 11, false};
      for (int k = 0; k < 8; ++k) bad += wrong(in, k, x + k);
    }
  }
  return bad;
}
// Is the mass of n keys known if all of them lie in the last bucket?
extern "C" int known_at_the_end(int rows, int n) {
  const float top = (float)rows / (float)n * fine_top(rows);
  uint32_t key;
  memcpy(&key, &top, 4);
  for (int x = -1; x <= 1; ++x) {  // (the quotient may be off by two places)
    const BucketMap g = bucket_map_from(kTopKey - key + 2 * x, rows);
    const BucketStart last = bucket_start(g, kBuckets - 1);
    if (!mass_known(mass_rule(last.t), n, last.t, kTopKey)) return 0;
  }
  return 1;
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
    lib.misplaced.argtypes = lib.wrong_masses.argtypes = [ctypes.c_uint32, ctypes.c_int]
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


def test_every_bucket_of_the_plain_layout_holds_the_keys_between_its_edges(shim):
    assert shim.misplaced(0, 0) == 0


@pytest.mark.parametrize("rows", [8, 127, 128, 4096])
def test_masses_of_buckets_are_exact(shim, rows):
    """The mass of a bucket follows exactly from the sum of its keys' words, for one key of any score below the last 512 and for as many
    equal or spread ones as the layout says it does."""
    for t0 in range(shim.t_of(rows * 3.0) & ~((1 << 21) - 1), shim.t_of(rows * 0.5 / (1 << 20)) + (1 << 21), 1 << 21):
        assert shim.wrong_masses(t0, rows) == 0, (rows, hex(t0))


def test_keys_that_all_lie_in_the_last_bucket(shim):
    """However many window rows and tokens there are, the mass of keys that all lie below the layout is known without exact
    sweeps (which 290 rows and more needed at four to sixteen tokens per row)."""
    rows = sorted({int(1.17 ** x) for x in range(53)} | {127, 128, 255, 256, 257, 288, 289, 448, 2048, 4095, 4096})
    lengths = sorted({int(1.07 ** x) for x in range(205)} | {(1 << x) + y for x in range(21) for y in (-1, 0, 1)} - {0, (1 << 20) + 1})
    assert max(lengths) == 1 << 20
    for r in rows:
        for n in lengths:
            assert shim.known_at_the_end(r, n), (r, n)
