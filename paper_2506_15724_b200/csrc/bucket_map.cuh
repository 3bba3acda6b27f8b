// The buckets that allocation and selection sort a unit's keys into (see rank_common.cuh). Plain integer and float arithmetic that a
// C++ compiler for the host takes too, so that the layouts can be checked one by one without a GPU.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define MADAKV_HD __host__ __device__ __forceinline__
#else
#define MADAKV_HD inline
#endif

namespace madakv {
namespace {

constexpr uint32_t kTopKey = 0x7f81ffffu;  // t = kTopKey - key: ascending t is descending importance

// The first layout of the buckets depends on a sequence's length and the window only, so that no sweep has to find the range of
// the keys before. The scores of a unit add up to its window rows, so their mean is known; sums of many rows crowd around
// it or, where a few tokens hold much of the mass, somewhat below (half of the keys of a grouped-query unit lie within a
// twelfth of an octave). 768 buckets cover 1.5 octaves there, for fewer than 128 rows three; 64 or, for small means, 32 per
// octave lie above, up to 512.0, and 64 below; the first and the last one take what lies outside. (64 buckets per octave
// throughout: 1000 candidates for 32768 keys of 224 rows and a sweep more for 131072 keys of 256 rows, 3400 in one
// bucket; and atomics on few addresses. One octave: 64 units of 3688 keys, 256 rows, whose keys lie half an octave below
// the mean, 60 us for the three steps after scoring instead of 50.)
constexpr int kBuckets = 2048, kDig = 11, kMidBuckets = 768;
constexpr int kMidRows = 128;              // from this many window rows on: 1.5 octaves
constexpr uint32_t kMapTop = 0x3b800000u;  // t of 512.0, rounded down to where a bucket starts
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
  g.high_shift = (g.mid - kMapTop) >> 17 <= 832u ? 17 : 18;
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
};
MADAKV_HD BucketStart bucket_start(const BucketMap& g, int b) {
  if (b < g.b0) return {(uint32_t)(b + g.c1) << g.high_shift, g.high_shift};
  if (b < g.b0 + kMidBuckets) return {g.mid + ((uint32_t)(b - g.b0) << g.mid_shift), g.mid_shift};
  return {(uint32_t)(b - g.c3) << kLowShift, kLowShift};
}

}  // namespace
}  // namespace madakv
