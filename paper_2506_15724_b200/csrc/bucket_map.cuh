// The buckets that allocation and selection sort a unit's keys into (see rank_common.cuh). Plain integer and float arithmetic that a
// C++ compiler for the host takes too, so that the layouts can be checked one by one without a GPU.
#pragma once

#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define MADAKV_HD __host__ __device__ __forceinline__
#else
#define MADAKV_HD inline
#endif

namespace madakv {
namespace {

constexpr uint32_t kTopKey = 0x7fffffffu;  // t = kTopKey - key: ascending t is descending importance, octaves begin at multiples of 2^23

// The first layout of the buckets depends on a sequence's length and the window only, so that no sweep has to find the range of
// the keys before. The scores of a unit add up to its window rows, so their mean is known; sums of many rows crowd around
// it or, where a few tokens hold much of the mass, somewhat below (half of the keys of a grouped-query unit lie within a
// twelfth of an octave). 768 buckets cover 1.5 octaves there, for fewer than 128 rows three; 64 or, for small means, 32 per
// octave lie above, up to 512.0, and 64 below; the first and the last one take what lies outside. (64 buckets per octave
// throughout: 1000 candidates for 32768 keys of 224 rows and a sweep more for 131072 keys of 256 rows, 3400 in one
// bucket; and atomics on few addresses. One octave: 64 units of 3688 keys, 256 rows, whose keys lie half an octave below
// the mean, 60 us for the three steps after scoring instead of 50.)
// The last bucket has to begin so low that the mass of a unit's keys is known if all of them lie there (mass_known), as nearly all
// do in a unit whose mass one token holds: n keys below 1 / n. 832 buckets above leave seven octaves below the fine ones,
// enough for 256 rows, 576 leave eleven, enough for the most rows there can be (4096). (With 832 for any number, 4 units of
// 8192 keys, 448 rows, all but a two-thousandth of the mass in one key: allocation 23.8 us, with 576 15.5.)
constexpr int kBuckets = 2048, kDig = 11, kMidBuckets = 768;
constexpr int kMidRows = 128;              // from this many window rows on: 1.5 octaves
constexpr uint32_t kMapTop = 0x3c000000u;  // t of the largest score below 512.0
constexpr int kLowShift = 17;
struct BucketMap {
  uint32_t mid;              // where the fine buckets start
  int mid_shift, high_shift; // values of t per bucket there and above, as shifts; below it is kLowShift
  int c1, b0, c3;            // bucket of t above: (t >> high_shift) - c1; first fine bucket; below: (t >> kLowShift) + c3
};
// t0: t of the largest score that the fine buckets are for.
MADAKV_HD BucketMap bucket_map_from(uint32_t t0, int rows) {
  BucketMap g;
  g.mid_shift = rows >= kMidRows ? 14 : 15;
  // (aligned so that eight buckets from a multiple of eight on are equally wide)
  const uint32_t first = kMapTop + (8u << 18), mid = t0 & ~((8u << 18) - 1u);
  g.mid = mid > first ? mid : first;
  g.high_shift = (g.mid - kMapTop) >> 17 <= (rows <= 256 ? 832u : 576u) ? 17 : 18;
  g.c1 = (int)(kMapTop >> g.high_shift);
  g.b0 = (int)(g.mid >> g.high_shift) - g.c1;
  g.c3 = g.b0 + kMidBuckets - (int)((g.mid + ((uint32_t)kMidBuckets << g.mid_shift)) >> kLowShift);
  return g;
}
// The factor between the mean score and the largest one that the fine buckets are for.
MADAKV_HD float fine_top(int rows) { return rows >= kMidRows ? 1.23f : 2.2f; }
// The fine buckets' line is steeper than the two others: before them it runs below the upper line, behind them above the lower
// one. What of the two others lies on the far side of the fine buckets decides nothing (with 32 buckets per octave above, the
// lower line, carried on that far, would cross the upper one).
MADAKV_HD uint32_t map_bucket(const BucketMap& g, uint32_t t) {
  const int high = (int)(t >> g.high_shift) - g.c1, fine = ((int)(t - g.mid) >> g.mid_shift) + g.b0, low = (int)(t >> kLowShift) + g.c3;
  const int below = fine < low ? fine : low, at = high > below ? high : below, last = at < kBuckets - 1 ? at : kBuckets - 1;
  return (uint32_t)(last > 0 ? last : 0);
}
// Where bucket b starts (t; the first one: where it would) and, as a shift, the width of it and of its neighbours up to the next
// multiple of eight.
struct BucketStart {
  uint32_t t;
  int shift;
  bool ends;  // (of the layout) the first bucket takes all that lies before it, too, the last one all behind it
};
MADAKV_HD BucketStart bucket_start(const BucketMap& g, int b) {
  if (b < g.b0) return {(uint32_t)(b + g.c1) << g.high_shift, g.high_shift, true};
  if (b < g.b0 + kMidBuckets) return {g.mid + ((uint32_t)(b - g.b0) << g.mid_shift), g.mid_shift, true};
  return {(uint32_t)(b - g.c3) << kLowShift, kLowShift, true};
}
// The last t of the bucket x places behind the one that b starts with, which is bucket `at` then.
MADAKV_HD uint32_t bucket_last(const BucketStart& b, int x, int at) {
  const uint32_t last = b.t + ((uint32_t)(x + 1) << b.shift) - 1u;
  return (b.ends && at == kBuckets - 1) || last > kTopKey ? kTopKey : last;
}

// The plain layout, the same for all sequences: 64 buckets per octave from 512 down to 2^-23, for half the instructions per key.
struct PlainMap {};
MADAKV_HD uint32_t map_bucket(const PlainMap&, uint32_t t) {
  const int b = (int)(t >> 17) - (int)(kMapTop >> 17), last = b < kBuckets - 1 ? b : kBuckets - 1;
  return (uint32_t)(last > 0 ? last : 0);
}
MADAKV_HD BucketStart bucket_start(const PlainMap&, int b) { return {kMapTop + ((uint32_t)b << 17), 17, true}; }

// The mass of a bucket, exactly, from its keys' count and the sum modulo 2^32 of a word per key. Scores from 2^-9 on are multiples
// of 2^-32 and those of a bucket lie in one octave, so that q = floor(x * 2^32) is linear in the key: their word is the key itself,
// and what it tells is exact however large the scores are (as long as they are fewer than 2^32 / width: 16384 for the widest buckets).
// The word of smaller scores is q, above a constant; all of them lie between the bucket's edges, so that the sum is known
// where count * (distance of the edges) is below 2^32. (With q modulo 2^32 for all scores one key of 32 or more, an attention sink
// as many prompts have one, sent its unit through some thirty exact sweeps: 8 units of 32768 keys, 128 rows, half of
// the mass in one key, allocation 65.8 us instead of 12.0.)
constexpr uint32_t kLinearEnd = 0x45000000u;  // t of the largest score below 2^-9
constexpr uint32_t kLowBias = 0x3b000000u;    // the bits of 2^-9
MADAKV_HD float score_of(uint32_t t) {  // t <= kTopKey
  const uint32_t key = kTopKey - t;
  float x;
  memcpy(&x, &key, 4);
  return x;
}
// (The sum with 2^-9, rounded towards zero, has floor(x * 2^32) in the low bits of its significand. The conversion to an integer
// runs at a small fraction of the rate of additions.)
MADAKV_HD uint32_t mass_word(uint32_t t) {
#ifdef __CUDA_ARCH__
  float w;  // (a predicated addition instead of a choice between two results)
  asm("{.reg .pred small;\n\tsetp.lt.f32 small, %1, 0f3b000000;\n\tmov.f32 %0, %1;\n\t@small add.rz.f32 %0, %1, 0f3b000000;}" : "=f"(w) : "f"(score_of(t)));
  return __float_as_uint(w);
#else
  return t < kLinearEnd ? kTopKey - t : kLowBias + (uint32_t)((double)score_of(t) * 4294967296.0);
#endif
}
// Buckets of one octave (eight of them from a multiple of eight on are), of which t is any key's: how their masses are found.
struct MassRule {
  bool linear;
  int up;  // their sums are in units of 2^up
};
MADAKV_HD MassRule mass_rule(uint32_t t) {
  const bool linear = t < kLinearEnd;
  return {linear, linear ? (int)((kTopKey - t) >> 23) - (int)(kLowBias >> 23) : 0};
}
// Mass of c keys whose words add up to sum, in a bucket whose smallest key is `last`.
MADAKV_HD unsigned long long mass_sum(const MassRule& r, uint32_t c, uint32_t sum, uint32_t last) {
  const uint32_t w = mass_word(last), least = r.linear ? (w & 0x7fffffu) | 0x800000u : w - kLowBias;
  return (unsigned long long)c * least + (sum - c * w);
}
// Is that exact, for a bucket from first to last? (For small scores a little is left for the rounding.)
MADAKV_HD bool mass_known(const MassRule& r, uint32_t c, uint32_t first, uint32_t last) {
  if (r.linear) return (unsigned long long)c * (last - first) <= 0xffffffffull;
  return (float)c * (score_of(first) - score_of(last)) < 0.999f;
}

}  // namespace
}  // namespace madakv
