// Shared pieces of the two ranking kernels (Eq. 9's count in allocate.cu, the top-budget selection in select.cu): the
// keys of one unit, spread over a team of 1-8 blocks, and the narrowing of a threshold to a short list of candidates.
//
// A unit's keys sit in registers (KPT consecutive positions per thread); a long unit in a call with few units is spread over
// a thread-block cluster, whose blocks exchange their partial results through distributed shared memory, and a unit
// longer than its blocks' registers is read twice by a kernel of its own (see rank_shape). The threshold (the budget-th
// largest key, or the key at which a mass is reached) is found in few steps. Two things bound these kernels: the integer
// instructions per key in calls with many units (an SM has some 230 000 keys of 256 units of 131072 keys to handle), and the
// fixed latency of a step (barriers, walking the buckets) in calls with few.
//   buckets  a count (and for Eq. 9 a mass, see allocate.cu) per key into 2048 buckets by shared atomics without a result
//            (bucket_map); a walk of the buckets narrows the range that the threshold can lie in to one bucket, usually
//            some tens of keys
//   list     the keys of the narrowed range are collected in shared memory and compared with one another (more than 64
//            of them: after half of a block's threads per modality have laid buckets over them once more)
// A team's blocks meet twice. Every block sums its buckets up to 32 coarse ones and pushes those to all; behind the first
// barrier a warp per modality of every block finds the coarse bucket, reads its 64 buckets from all blocks and finds the
// bucket, the same in every block, with the places of all blocks' keys in the list; the keys are pushed there before the
// second barrier. (With a share of all buckets per block, read from all others, their totals and the bucket announced and
// the lists gathered, five barriers in all, allocation and selection of 4 units of 32768 keys, 224 rows, took 17.1 and 10.2 us;
// now 11.9 and 7.6, one call after the other.)
// Buckets over the range of each unit's keys needed a sweep for that range before; without it, and with long units read
// twice instead of three (allocation) or four times (selection), allocation + selection + compaction went from 602 to 483 us
// on 256 units of 131072 keys, from 618 to 523 on 1600 of 13411, from 213 to 161 on 3360 of 471, from 31 to 26 on 200 of 772.
// (The same in four or five passes of a plain radix descent: 750 us on the first of these.)
// Keys that crowd (many ties, a few values far away from all others) make the list overflow; then the buckets are laid
// over the narrowed range once more, and after that the range is bisected with exact sweeps over all keys, which ends
// for any input, at the latest when the range holds one value.
#pragma once

#include "bucket_map.cuh"
#include "common.cuh"

namespace madakv {
namespace {

constexpr unsigned int kFull = 0xffffffffu;
constexpr int kRankThreads = 512;
constexpr int kRankWarps = kRankThreads / 32;
constexpr int kHalf = kRankThreads / 2;        // threads per modality in the walks
constexpr int kListCap = 1024;                 // candidates per modality at most
// Candidates that are compared with one another, which takes instructions in proportion to their square; more are sorted into
// buckets once more before, some 1500 clocks. (With up to 256 compared, 8 x 4 units of 8192 keys, 224 rows, one key with nine
// tenths of the mass or two heaps of scores, 110-280 candidates: allocation 20.4 and 22.5 us, selection 13.2 and 16.2; with 64,
// 10.8, 11.3, 9.9, 10.0. With 96 and 128 the same within 3 %.)
constexpr uint32_t kFewCap = 64;
constexpr int kMaxTeam = 8;
constexpr uint32_t kNoKey = 0xffffffffu;       // t of a slot without a key
constexpr uint32_t kNowhere = 0xfffffffeu;     // start of a range that holds no t at all (t < 2^31)
typedef unsigned long long u64;

// ---- the blocks of a unit: a cluster, or one block on its own
__device__ __forceinline__ uint32_t team_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
template <int TEAM>
__device__ __forceinline__ void team_sync() {
  if (TEAM > 1)
    asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
  else
    __syncthreads();
}
// The two halves of a first barrier: no block of a cluster touches another's shared memory before that one has started.
template <int TEAM>
__device__ __forceinline__ void team_started() {
  if (TEAM > 1) asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");
}
template <int TEAM>
__device__ __forceinline__ void team_wait_started() {
  if (TEAM > 1) asm volatile("barrier.cluster.wait;" ::: "memory");
}
__device__ __forceinline__ uint32_t peer_addr(const void* local, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(local)), "r"(rank));
  return r;
}
template <int TEAM>
__device__ __forceinline__ uint32_t peer_load(const uint32_t* local, uint32_t rank) {
  if (TEAM == 1) return *local;
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(peer_addr(local, rank)));
  return v;
}
template <int TEAM>
__device__ __forceinline__ u64 peer_load(const u64* local, uint32_t rank) {
  if (TEAM == 1) return *local;
  u64 v;
  asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(peer_addr(local, rank)));
  return v;
}
template <int TEAM>
__device__ __forceinline__ void peer_store(uint32_t* local, uint32_t rank, uint32_t v) {
  if (TEAM == 1) *local = v;
  else asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(peer_addr(local, rank)), "r"(v) : "memory");
}
template <int TEAM>
__device__ __forceinline__ void peer_store(u64* local, uint32_t rank, u64 v) {
  if (TEAM == 1) *local = v;
  else asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(peer_addr(local, rank)), "l"(v) : "memory");
}

template <int TEAM>
__device__ __forceinline__ void peer_store(uint4* local, uint32_t rank, uint4 v) {
  if (TEAM == 1) *local = v;
  else asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(peer_addr(local, rank)), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

// ---- sums over a warp
// 64-bit sum (modulo 2^64) through three 32-bit reductions: 22 + 22 + 20 bits, 32 of which cannot overflow 32 bits
__device__ __forceinline__ u64 warp_sum64(u64 v) {
  const uint32_t a = __reduce_add_sync(kFull, (uint32_t)v & 0x3fffffu);
  const uint32_t b = __reduce_add_sync(kFull, (uint32_t)(v >> 22) & 0x3fffffu);
  const uint32_t c = __reduce_add_sync(kFull, (uint32_t)(v >> 44));
  return (u64)a + ((u64)b << 22) + ((u64)c << 44);
}
__device__ __forceinline__ uint32_t warp_scan32(uint32_t v) {  // inclusive
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t t = __shfl_up_sync(kFull, v, off);
    if ((int)(threadIdx.x & 31) >= off) v += t;
  }
  return v;
}
__device__ __forceinline__ u64 warp_scan64(u64 v) {
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const u64 t = __shfl_up_sync(kFull, v, off);
    if ((int)(threadIdx.x & 31) >= off) v += t;
  }
  return v;
}

// ---- loads: KPT consecutive positions from pos0 (a multiple of KPT) of a unit's scores and of its sequence's mask, as far
// as the row goes (n_max positions; what lies beyond the sequence's own length is sorted out by the caller, so that the
// loads need not wait for the length).
// Rows of odd lengths start anywhere: scores are read in aligned 16-byte pieces and moved down by `mis` elements
// (the same for the whole unit), mask bytes in aligned words and funnel shifts; only threads at the ends of a row go
// element by element.
// A score's order-preserving key is its bits where it is positive, else (NaN too) 0; kept is t, its distance from kTopKey.
__device__ __forceinline__ uint32_t score_t(float x) { return kTopKey - __float_as_uint(fmaxf(x, 0.0f)); }
// The loads are issued apart from their use, so that scores, mask, length and budgets are all on their way together (one after
// the other, as the branches had them, they took two or three latencies of the memory: 5000 of a block's 16000 clocks).
template <int KPT>
struct RawScores {
  float4 v[KPT / 4 + 1];
  int down;  // elements to move down
};
template <int KPT>
__device__ __forceinline__ void issue_scores(const float* row, int mis, int n_max, int pos0, RawScores<KPT>& raw) {
  raw.down = 0;
  raw.v[KPT / 4] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (mis == 0 && pos0 + KPT <= n_max) {
#pragma unroll
    for (int j = 0; j < KPT / 4; ++j) raw.v[j] = __ldg(reinterpret_cast<const float4*>(row + pos0) + j);
  } else if (mis != 0 && pos0 + KPT + 4 <= n_max) {
    // (a misaligned row has a unit before it: the pieces start inside the array; they end inside the row)
#pragma unroll
    for (int j = 0; j < KPT / 4 + 1; ++j) raw.v[j] = __ldg(reinterpret_cast<const float4*>(row + pos0 - mis) + j);
    raw.down = mis;
  } else {
    auto one = [&](int x) { return pos0 + x < n_max ? __ldg(row + pos0 + x) : 0.f; };
#pragma unroll
    for (int j = 0; j < KPT / 4; ++j) raw.v[j] = make_float4(one(4 * j), one(4 * j + 1), one(4 * j + 2), one(4 * j + 3));
  }
}
template <int KPT>
__device__ __forceinline__ void take_scores(const RawScores<KPT>& raw, int mis, uint32_t (&t)[KPT]) {
  float f[KPT + 4];
#pragma unroll
  for (int j = 0; j < KPT / 4 + 1; ++j) {
    f[4 * j] = raw.v[j].x;
    f[4 * j + 1] = raw.v[j].y;
    f[4 * j + 2] = raw.v[j].z;
    f[4 * j + 3] = raw.v[j].w;
  }
  if (mis) {  // (the same for the whole unit)
#pragma unroll
    for (int j = 0; j < KPT + 3; ++j) f[j] = (raw.down & 1) ? f[j + 1] : f[j];
#pragma unroll
    for (int j = 0; j < KPT; ++j) f[j] = (raw.down & 2) ? f[j + 2] : f[j];
  }
#pragma unroll
  for (int j = 0; j < KPT; ++j) t[j] = score_t(f[j]);
}
template <int KPT>
__device__ __forceinline__ void load_scores(const float* row, int mis, int n_max, int pos0, uint32_t (&t)[KPT]) {
  RawScores<KPT> raw;
  issue_scores<KPT>(row, mis, n_max, pos0, raw);
  take_scores<KPT>(raw, mis, t);
}
template <int KPT>
struct RawMask {
  uint32_t w[KPT / 4 + 1];
  uint32_t shift;  // bits to move down
  uint32_t bits;   // of positions that were read one by one
};
template <int KPT>
__device__ __forceinline__ void issue_mask(const uint8_t* row, int n_max, int pos0, RawMask<KPT>& raw) {
  const uintptr_t at = reinterpret_cast<uintptr_t>(row + pos0);
  raw.shift = raw.bits = 0;
#pragma unroll
  for (int j = 0; j < KPT / 4 + 1; ++j) raw.w[j] = 0;
  if (pos0 + KPT <= n_max && (at & (KPT - 1)) == 0) {
    if (KPT == 8) {
      const uint2 v = __ldg(reinterpret_cast<const uint2*>(row + pos0));
      raw.w[0] = v.x;
      raw.w[1] = v.y;
    } else {
#pragma unroll
      for (int j = 0; j < KPT / 16; ++j) {
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(row + pos0) + j);
        raw.w[4 * j] = v.x;
        raw.w[4 * j + 1] = v.y;
        raw.w[4 * j + 2] = v.z;
        raw.w[4 * j + 3] = v.w;
      }
    }
  } else if (pos0 >= 4 && pos0 + KPT + 4 <= n_max) {
    const uint32_t* src = reinterpret_cast<const uint32_t*>(at & ~(uintptr_t)3);
    raw.shift = (uint32_t)(at & 3) * 8;
#pragma unroll
    for (int j = 0; j < KPT / 4 + 1; ++j) raw.w[j] = __ldg(src + j);
  } else {
#pragma unroll
    for (int j = 0; j < KPT; ++j)
      if (pos0 + j < n_max && __ldg(row + pos0 + j)) raw.bits |= 1u << j;
  }
}
template <int KPT>
__device__ __forceinline__ uint32_t take_mask(const RawMask<KPT>& raw) {  // bit j: position pos0 + j is visual
  uint32_t vis = raw.bits;
#pragma unroll
  for (int j = 0; j < KPT / 4; ++j) vis |= nonzero_bytes(__funnelshift_r(raw.w[j], raw.w[j + 1], raw.shift)) << (4 * j);
  return vis;
}
template <int KPT>
__device__ __forceinline__ uint32_t load_mask(const uint8_t* row, int n_max, int pos0) {
  RawMask<KPT> raw;
  issue_mask<KPT>(row, n_max, pos0, raw);
  return take_mask<KPT>(raw);
}
// Bits of a long unit in shared memory, one per position of the block: word w sits at w + w / 32, so that threads that walk
// several consecutive words each hit different banks. A thread's 16 positions of round r are half a word.
__device__ __forceinline__ int bits_slot(int w) { return w + (w >> 5); }
__device__ __forceinline__ uint16_t& bits_of_thread(uint32_t* words, int r) {
  const int half = r * kRankThreads + threadIdx.x;
  return reinterpret_cast<uint16_t*>(words)[2 * bits_slot(half >> 1) + (half & 1)];
}
template <int KPT>
__device__ __forceinline__ uint32_t valid_bits(int n, int pos0) {  // bit j: position pos0 + j lies inside the sequence
  const int k = min(max(n - pos0, 0), KPT);
  return k == 32 ? 0xffffffffu : (1u << k) - 1u;
}

// The first layout for a sequence of n tokens (bucket_map.cuh).
__device__ __forceinline__ BucketMap bucket_map(int rows, int n) {
  return bucket_map_from(kTopKey - __float_as_uint(__fdividef((float)rows, (float)max(n, 1)) * fine_top(rows)), rows);
}

// ---- shared memory of a block
// What a walk finds for a modality.
struct Found {
  u64 mass, above_q;                   // mass of all its keys (allocation); mass before the bucket
  uint32_t total, hit, at, above, in;  // its keys; whether what is needed is reached; the bucket; keys before it and in it
  uint32_t before;                     // of the keys before the bucket (of all, if it is not reached) those of the blocks before this one
  uint32_t inexact;                    // masses are not known exactly
  uint32_t seg[kMaxTeam + 1];          // places of each block's keys of the bucket
};
constexpr int kCoarse = kBuckets / 64;
template <int TEAM, int WORDS>  // WORDS: count, or count and mass, per bucket
struct RankShared {
  static constexpr int kStride = kBuckets;
  static constexpr int kCap = TEAM > 1 && WORDS == 2 ? kListCap / 2 : kListCap;  // (allocation's teams have no room for more)
  // the buckets' counts; once they are walked, the buckets of the finish (count, mass low, mass high; one per thread and
  // modality) and the keys that are compared with one another, with their masses, take their place
  alignas(16) uint32_t cnt[2 * WORDS * kStride];
  uint4 coarse[2][TEAM][TEAM > 1 ? kCoarse : 1];  // every block's sums of 64 buckets: count, mass (low, high), inexact
  alignas(16) uint32_t list[2][kCap];           // candidates of the team (allocation: in block 0)
  Found found[2];
  u64 wsum[2][kRankWarps];                      // per warp: masses (allocation)
  u64 slice_q[2][kMaxTeam];
  u64 wscan_q[kRankWarps];
  u64 want[2];                                  // walk: what is to be reached
  u64 fin_m[2];                                 // finish: mass before the range
  uint32_t slice_c[2][kMaxTeam];
  uint32_t wscan_c[kRankWarps], wcnt[2][kRankWarps];
  uint32_t few_n[2];
  uint32_t fin_c[2], fin_lo[2], fin_in[2], fin_more[2];
  uint32_t list_n;                              // candidates of this block: visual | text << 16
  __device__ uint32_t* fin_bucket(int m, int k) { return cnt + (m * 3 + k) * kHalf; }
  __device__ uint32_t* few(int m) { return cnt + (6 + m) * kHalf; }
  __device__ u64* few_mass(int m) { return reinterpret_cast<u64*>(cnt + (8 + 2 * m) * kHalf); }
  static_assert((WORDS == 2 ? 12 : 8) * kHalf <= 2 * WORDS * kStride, "room for the finish");
};

// What is known of modality m's threshold: t lies in [lo, lo + span], `in` keys of the modality do, `above` keys lie
// before lo. Identical in every thread of the team.
struct RankRange {
  uint32_t lo, span, in, above;
};
__device__ __forceinline__ int range_shift(uint32_t span, int dig) { return max(32 - __clz((int)span) - dig, 0); }

// The range of t of bucket `at`, of the first layout or of one over g with 2^shift values of t per bucket.
template <typename Map>
__device__ __forceinline__ void bucket_range(RankRange& g, const Map* map, uint32_t at, int shift) {
  if (map) {
    const BucketStart s = bucket_start(*map, (int)at);
    g.lo = at ? s.t : 0u;
    g.span = (at < kBuckets - 1 ? s.t + (1u << s.shift) - 1u : kTopKey) - g.lo;
  } else {
    const uint32_t cut = at << shift;
    g.span = min(g.span - cut, (1u << shift) - 1u);
    g.lo += cut;
  }
}
// (Without a barrier: the caller has one before the buckets are used.)
template <int TEAM, int WORDS>
__device__ __forceinline__ void zero_buckets(RankShared<TEAM, WORDS>& sh) {
  for (int x = threadIdx.x; x < 2 * WORDS * RankShared<TEAM, WORDS>::kStride / 4; x += kRankThreads)
    reinterpret_cast<uint4*>(sh.cnt)[x] = make_uint4(0, 0, 0, 0);
  if (threadIdx.x == 0) sh.list_n = 0;
}

// Walk of the buckets, filled in by all threads of the block: start(m, b) tells where bucket b of modality m starts,
// need(m, mass) what is to be reached, a mass (WORDS = 2) or a count; 0: nothing. Leaves `found`, the same in every block
// (but for `before`). Ends with a barrier of the block.
template <int TEAM, int WORDS, typename Start, typename Need>
__device__ __forceinline__ void walk(RankShared<TEAM, WORDS>& sh, uint32_t rank, Start start, Need need) {
  constexpr bool kMass = WORDS == 2;
  constexpr int kStride = RankShared<TEAM, WORDS>::kStride;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  __syncthreads();
  {  // eight buckets per thread
    const int m = tid / kHalf, i = tid % kHalf, b0 = i * 8;
    const uint4* w = reinterpret_cast<const uint4*>(sh.cnt + m * kStride + b0);
    const uint4 v0 = w[0], v1 = w[1];
    uint32_t lc = ((v0.x + v0.y) + (v0.z + v0.w)) + ((v1.x + v1.y) + (v1.z + v1.w));
    const uint32_t c[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
    u64 lq = 0;
    bool bad = false;
    if (kMass && lc) {  // (the buckets of most threads are empty)
      const uint4 s0 = w[2 * kStride / 4], s1 = w[2 * kStride / 4 + 1];
      const uint32_t s[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
      const BucketStart at = start(m, b0);
      const MassRule rule = mass_rule(at.t);
      uint32_t most = 0;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        lq += mass_sum(rule, c[k], s[k], bucket_last(at, k, b0 + k));
        most = max(most, c[k]);
      }
      lq <<= rule.up;
      // (the eight are equally wide, but for what the first and the last one of a layout take besides)
      bad = !mass_known(rule, most, at.t, bucket_last(at, 0, b0));
      if (at.ends && b0 == 0) bad = bad || c[0];
      if (at.ends && b0 == kBuckets - 8) bad = bad || !mass_known(rule, c[7], at.t + (7u << at.shift), kTopKey);
    }
    const uint32_t bads = kMass ? __ballot_sync(kFull, bad) : 0u;
    if (TEAM == 1) {  // a block on its own: every thread learns what lies before its buckets
      uint32_t ic = warp_scan32(lc);
      u64 iq = kMass ? warp_scan64(lq) : 0ull;
      Found& f = sh.found[m];
      if (lane == 31) {
        sh.wscan_c[warp] = ic;
        if (kMass) {
          sh.wscan_q[warp] = iq;
          sh.wcnt[0][warp] = bads;
        }
      }
      __syncthreads();
      if (i < 32) {  // a warp per modality: what lies before each of its warps, and what is needed
        const bool here = lane / (kRankWarps / 2) == m;
        const uint32_t wc = here ? sh.wscan_c[lane] : 0u, before_c = warp_scan32(wc) - wc;
        const u64 wq = kMass && here ? sh.wscan_q[lane] : 0ull, before_q = kMass ? warp_scan64(wq) - wq : 0ull;
        const uint32_t inexact = kMass ? __any_sync(kFull, lane < kRankWarps && sh.wcnt[0][lane]) : 0u;
        if (here) {
          sh.wscan_c[lane] = before_c;
          if (kMass) sh.wscan_q[lane] = before_q;
        }
        if (lane == (m + 1) * (kRankWarps / 2) - 1) {
          const u64 all = before_q + wq;
          f.total = before_c + wc;
          f.mass = all;
          f.inexact = inexact;
          f.hit = 0;
          f.seg[0] = 0;
          sh.want[m] = need(m, all);
        }
      }
      __syncthreads();
      ic += sh.wscan_c[warp];
      if (kMass) iq += sh.wscan_q[warp];
      const u64 want = sh.want[m];
      if (want && (kMass ? iq - lq < want && iq >= want : ic - lc < want && ic >= want)) {
        uint32_t run = ic - lc, at = 0, at_c = 0, at_in = 0;
        u64 run_q = iq - lq, at_q = 0;
        BucketStart first = {};
        MassRule rule = {};
        if (kMass) {
          first = start(m, b0);
          rule = mass_rule(first.t);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          if (kMass ? run_q < want : run < want) {
            at = b0 + k;
            at_c = run;
            at_in = c[k];
            at_q = run_q;
          }
          run += c[k];
          if (kMass) run_q += mass_sum(rule, c[k], sh.cnt[(2 + m) * kStride + b0 + k], bucket_last(first, k, b0 + k)) << rule.up;
        }
        f.hit = 1;
        f.at = at;
        f.above = at_c;
        f.in = at_in;
        f.above_q = at_q;
      }
      __syncthreads();
      return;
    }
    // eight threads per coarse bucket
#pragma unroll
    for (int off = 1; off < 8; off <<= 1) {
      lc += __shfl_xor_sync(kFull, lc, off);
      if (kMass) lq += __shfl_xor_sync(kFull, lq, off);
    }
    if ((lane & 7) < TEAM)
      peer_store<TEAM>(&sh.coarse[m][rank][i >> 3], lane & 7, make_uint4(lc, (uint32_t)lq, (uint32_t)(lq >> 32), (bads >> (lane & 24)) & 0xffu));
  }
  team_sync<TEAM>();
  if (warp < 2) {
    const int m = warp;
    uint32_t c = 0, mine = 0, bad = 0;  // mine: of the blocks before this one
    u64 q = 0;
#pragma unroll
    for (int r = 0; r < TEAM; ++r) {
      const uint4 e = sh.coarse[m][r][lane];
      c += e.x;
      if (r < (int)rank) mine += e.x;
      q += ((u64)e.z << 32) | e.y;
      bad |= e.w;
    }
    const uint32_t ic = warp_scan32(c);
    const u64 iq = kMass ? warp_scan64(q) : 0ull;
    const u64 all_q = kMass ? __shfl_sync(kFull, iq, 31) : 0ull, want = need(m, all_q);
    const uint32_t at_coarse = __ballot_sync(kFull, want && (kMass ? iq - q < want && iq >= want : ic - c < want && ic >= want));
    Found& f = sh.found[m];
    bad = kMass ? __any_sync(kFull, bad) : 0u;
    if (lane == 31) {
      f.total = ic;
      f.mass = iq;
      f.hit = at_coarse ? 1u : 0u;
      f.inexact = bad;
    }
    if (!at_coarse) {
      if (!kMass) {
        mine = __reduce_add_sync(kFull, mine);
        if (lane == 0) f.before = want ? mine : 0u;
      }
    } else {
      const int who = __ffs((int)at_coarse) - 1, b = who * 64 + 2 * lane;
      u64 pair[TEAM], sums[TEAM];
      const uint32_t* w = sh.cnt + m * kStride + b;
#pragma unroll
      for (int r = 0; r < TEAM; ++r) {
        pair[r] = peer_load<TEAM>(reinterpret_cast<const u64*>(w), r);
        if (kMass) sums[r] = peer_load<TEAM>(reinterpret_cast<const u64*>(w + 2 * kStride), r);
      }
      uint32_t last0 = 0, last1 = 0;
      MassRule rule = {};
      if (kMass) {
        const BucketStart at = start(m, b);
        rule = mass_rule(at.t);
        last0 = bucket_last(at, 0, b);
        last1 = bucket_last(at, 1, b + 1);
      }
      uint32_t c0 = 0, c1 = 0, m0 = 0, m1 = 0;
      u64 q0 = 0, q1 = 0;
#pragma unroll
      for (int r = 0; r < TEAM; ++r) {
        const uint32_t x = (uint32_t)pair[r], y = (uint32_t)(pair[r] >> 32);
        c0 += x;
        c1 += y;
        if (r < (int)rank) m0 += x, m1 += y;
        if (kMass) {
          q0 += mass_sum(rule, x, (uint32_t)sums[r], last0);
          q1 += mass_sum(rule, y, (uint32_t)(sums[r] >> 32), last1);
        }
      }
      if (kMass) {
        q0 <<= rule.up;
        q1 <<= rule.up;
      }
      const uint32_t run_c = __shfl_sync(kFull, ic - c, who) + warp_scan32(c0 + c1) - (c0 + c1);
      const u64 run_q = kMass ? __shfl_sync(kFull, iq - q, who) + warp_scan64(q0 + q1) - (q0 + q1) : 0ull;
      const uint32_t here = __ballot_sync(kFull, kMass ? run_q < want && run_q + q0 + q1 >= want : run_c < want && run_c + c0 + c1 >= want);
      const int at = here ? __ffs((int)here) - 1 : 31;  // (none only where the masses are not exact)
      const bool second = kMass ? run_q + q0 < want : run_c + c0 < want;
      uint32_t before = 0;
      if (!kMass)
        before = __reduce_add_sync(kFull, (lane < who ? mine : 0u) + (lane < at ? m0 + m1 : 0u) + (lane == at && second ? m0 : 0u));
      if (lane == at) {
        f.at = b + (second ? 1 : 0);
        f.above = run_c + (second ? c0 : 0u);
        f.in = second ? c1 : c0;
        f.above_q = run_q + (second ? q0 : 0ull);
        f.before = before;
        uint32_t place = 0;
#pragma unroll
        for (int r = 0; r < TEAM; ++r) {
          f.seg[r] = place;
          place += second ? (uint32_t)(pair[r] >> 32) : (uint32_t)pair[r];
        }
        f.seg[TEAM] = place;
      }
    }
  }
  __syncthreads();
}

// The places of the blocks' candidates in the list where no walk has told them (after exact sweeps): c0 and c1 are the
// numbers in this thread's hands. Barriers of the team.
template <int TEAM, int WORDS>
__device__ __forceinline__ void find_places(RankShared<TEAM, WORDS>& sh, uint32_t rank, uint32_t c0, uint32_t c1) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  c0 = __reduce_add_sync(kFull, c0);
  c1 = __reduce_add_sync(kFull, c1);
  __syncthreads();
  if (lane == 0) {
    sh.wcnt[0][warp] = c0;
    sh.wcnt[1][warp] = c1;
  }
  __syncthreads();
  if (warp < 2) {
    const uint32_t n = __reduce_add_sync(kFull, lane < kRankWarps ? sh.wcnt[warp][lane] : 0u);
    if (lane < TEAM) peer_store<TEAM>(&sh.slice_c[warp][rank], lane, n);
  }
  team_sync<TEAM>();
  if (threadIdx.x < 2) {
    uint32_t place = 0;
    for (int r = 0; r < TEAM; ++r) {
      sh.found[threadIdx.x].seg[r] = place;
      place += sh.slice_c[threadIdx.x][r];
    }
  }
  __syncthreads();
}

// A candidate of modality m into the list, at place x: of block 0, or (kAll) of all blocks.
template <int TEAM, int WORDS, bool kAll>
__device__ __forceinline__ void put(RankShared<TEAM, WORDS>& sh, int m, uint32_t x, uint32_t v) {
  uint32_t* at = &sh.list[m][x];
#pragma unroll
  for (int r = 0; r < (kAll ? TEAM : 1); ++r) peer_store<TEAM>(at, r, v);
}
// A warp's candidates into the list, as offsets from lo0 / lo1: bit j of in0 / in1 is set where the thread's j-th key belongs to
// the list of modality 0 / 1. One atomic per warp; candidates are few, so a thread picks them one by one.
template <int TEAM, int WORDS, int KPT, bool kAll>
__device__ __forceinline__ void append(RankShared<TEAM, WORDS>& sh, uint32_t rank, uint32_t in0, uint32_t in1, const uint32_t (&key)[KPT],
                                       uint32_t lo0, uint32_t lo1) {
  if (!__any_sync(kFull, (in0 | in1) != 0)) return;
  const int lane = threadIdx.x & 31;
  const uint32_t mine = __popc(in0) | (__popc(in1) << 16), incl = warp_scan32(mine);
  uint32_t base = 0;
  if (lane == 31) base = atomicAdd(&sh.list_n, incl);
  base = __shfl_sync(kFull, base, 31) + incl - mine;
  uint32_t o0 = (base & 0xffffu) + sh.found[0].seg[rank], o1 = (base >> 16) + sh.found[1].seg[rank];
  for (uint32_t left = in0 | in1; left; left &= left - 1) {
    const int j = __ffs(left) - 1;
    uint32_t k = key[0];
#pragma unroll
    for (int x = 1; x < KPT; ++x) k = x == j ? key[x] : k;
    const bool first = (in0 >> j) & 1u;
    put<TEAM, WORDS, kAll>(sh, first ? 0 : 1, first ? o0++ : o1++, k - (first ? lo0 : lo1));
  }
}

// The same for a unit that is not in registers: positions instead of keys, into lists of the block's own (the keys are read
// again when those are complete).
template <int TEAM, int WORDS>
__device__ __forceinline__ void append_positions(RankShared<TEAM, WORDS>& sh, uint32_t* pos0, uint32_t* pos1, uint32_t in0, uint32_t in1, int at) {
  if (!__any_sync(kFull, (in0 | in1) != 0)) return;
  const int lane = threadIdx.x & 31;
  const uint32_t mine = __popc(in0) | (__popc(in1) << 16), incl = warp_scan32(mine);
  uint32_t base = 0;
  if (lane == 31) base = atomicAdd(&sh.list_n, incl);
  base = __shfl_sync(kFull, base, 31) + incl - mine;
  uint32_t o0 = base & 0xffffu, o1 = base >> 16;
  for (; in0; in0 &= in0 - 1) pos0[o0++] = (uint32_t)(at + __ffs(in0) - 1);
  for (; in1; in1 &= in1 - 1) pos1[o1++] = (uint32_t)(at + __ffs(in1) - 1);
}

// The whole block: where among the candidates (offsets into the ranges; r0.in and r1.in of them) the thresholds lie, half of
// the threads per modality. need: a mass (with kMass; `before` is the exact mass before the range) or a count. Leaves in
// shared memory, per modality: fin_lo (the smallest t up to which the threshold is reached), fin_c and fin_m (count and mass
// before it), fin_in (candidates that equal it). A modality that is not `on` is left out. The lists are complete behind a
// barrier; ends with a barrier of the block.
template <int TEAM, int WORDS, bool kMass>
__device__ __forceinline__ void finish_lists(RankShared<TEAM, WORDS>& sh, const RankRange& r0, const RankRange& r1, bool on0, bool on1,
                                             u64 need0, u64 need1, u64 before0, u64 before1) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, m = tid / kHalf, i = tid % kHalf;
  const uint32_t n = m ? r1.in : r0.in, base = m ? r1.lo : r0.lo;
  const bool on = m ? on1 : on0;
  const u64 need = m ? need1 : need0;
  const uint32_t* list = sh.list[m];
  uint32_t in = n, above_c = m ? r1.above : r0.above;
  u64 above = m ? before1 : before0;
  auto mass = [&](uint32_t x) { return psi_fix(kTopKey - (base + x)); };
  const bool many0 = on0 && r0.in > kFewCap && r0.span > 0, many1 = on1 && r1.in > kFewCap && r1.span > 0;
  if (many0 || many1) {  // (the same in all threads)
    uint32_t lo = 0, span = m ? r1.span : r0.span;
    uint32_t *fc = sh.fin_bucket(m, 0), *flo = sh.fin_bucket(m, 1), *fhi = sh.fin_bucket(m, 2);
    for (;;) {
      const bool more = on && in > kFewCap && span > 0;
      if (i == 0) {
        sh.fin_more[m] = more ? 1u : 0u;
        sh.few_n[m] = 0;
      }
      fc[i] = 0;
      if (kMass) flo[i] = fhi[i] = 0;
      __syncthreads();
      if (!(sh.fin_more[0] | sh.fin_more[1])) break;
      const int shift = range_shift(span, 8);
      if (more) {
        for (uint32_t x = i; x < n; x += kHalf) {
          const uint32_t d = list[x] - lo;
          if (d <= span) {
            const uint32_t b = d >> shift;
            atomicAdd(&fc[b], 1u);
            if (kMass) {
              const u64 q = mass(list[x]);
              const uint32_t add = (uint32_t)q, old = atomicAdd(&flo[b], add);
              const uint32_t hi = (uint32_t)(q >> 32) + ((uint32_t)(old + add) < old ? 1u : 0u);
              if (hi) atomicAdd(&fhi[b], hi);
            }
          }
        }
      }
      __syncthreads();
      const uint32_t c = fc[i];
      uint32_t ic = warp_scan32(c);
      u64 q = 0, iq = 0;
      if (kMass) {
        q = ((u64)fhi[i] << 32) | flo[i];
        iq = warp_scan64(q);
      }
      if (lane == 31) {
        sh.wscan_c[warp] = ic;
        if (kMass) sh.wscan_q[warp] = iq;
      }
      __syncthreads();
      const bool lower = lane >= m * (kRankWarps / 2) && lane < warp;
      ic += above_c + __reduce_add_sync(kFull, lower ? sh.wscan_c[lane] : 0u);
      if (kMass) iq += above + warp_sum64(lower ? sh.wscan_q[lane] : 0ull);
      if (more && (kMass ? iq - q < need && iq >= need : ic - c < need && ic >= need)) {
        sh.fin_lo[m] = i;
        sh.fin_in[m] = c;
        sh.fin_c[m] = ic - c;
        if (kMass) sh.fin_m[m] = iq - q;
      }
      __syncthreads();
      if (more) {
        const uint32_t cut = sh.fin_lo[m] << shift;
        lo += cut;
        span = min(span - cut, (1u << shift) - 1u);
        in = sh.fin_in[m];
        above_c = sh.fin_c[m];
        if (kMass) above = sh.fin_m[m];
      }
    }
    if (on)
      for (uint32_t x = i; x < n; x += kHalf) {
        const uint32_t v = list[x];
        if (v - lo <= span) {
          const uint32_t s = atomicAdd(&sh.few_n[m], 1u);
          if (s < kFewCap) sh.few(m)[s] = v;  // (more than kFewCap are left only if all are alike)
        }
      }
    __syncthreads();
    list = sh.few(m);
  }
  // The keys left, compared with one another, four threads per key. The threshold's keys are those that what is needed is
  // reached with, but not before. (Keys that crowd are all alike: one of them is enough.)
  constexpr uint32_t kPer = kHalf / kFewCap;
  const uint32_t k = !on ? 0u : in > kFewCap ? 1u : in;
  if (kMass) {
    if ((uint32_t)i < k) sh.few_mass(m)[i] = mass(list[i]);
    __syncthreads();
  }
  if (((uint32_t)i & ~31u) / kPer < k) {  // (the other warps have no key)
    const uint32_t x = (uint32_t)i / kPer, part = (uint32_t)i % kPer, v = list[min(x, k - 1u)];
    uint32_t lt_c = 0, eq_c = 0;
    u64 lt = 0;
#pragma unroll 1
    for (uint32_t j = 4 * part; j < k; j += 4 * kPer) {  // (four at a time; behind the last one none counts)
      const uint4 o4 = *reinterpret_cast<const uint4*>(list + j);
      const uint32_t o[4] = {o4.x, j + 1 < k ? o4.y : kNoKey, j + 2 < k ? o4.z : kNoKey, j + 3 < k ? o4.w : kNoKey};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (o[e] < v) {
          ++lt_c;
          if (kMass) lt += sh.few_mass(m)[j + e];
        }
        if (o[e] == v) ++eq_c;
      }
    }
#pragma unroll
    for (int off = 1; off < (int)kPer; off <<= 1) {
      lt_c += __shfl_xor_sync(kFull, lt_c, off);
      eq_c += __shfl_xor_sync(kFull, eq_c, off);
      if (kMass) lt += __shfl_xor_sync(kFull, lt, off);
    }
    if (k < in) eq_c = in;
    const bool here = kMass ? above + lt < need && above + lt + eq_c * mass(v) >= need : above_c + lt_c < need && above_c + lt_c + eq_c >= need;
    if (x < k && part == 0 && here) {  // (all that write write the same)
      sh.fin_lo[m] = base + v;
      sh.fin_in[m] = eq_c;
      sh.fin_c[m] = above_c + lt_c;
      if (kMass) sh.fin_m[m] = above + lt;
    }
  }
  __syncthreads();
}

// ---- host: how a unit's keys are spread
struct RankShape {
  int kpt, team;  // keys per thread, blocks per unit
};
// A call with a unit or more per SM gets one block per unit, which reads the keys of a long unit in every sweep (kpt = 0, the
// "long" kernels): spread over 2, 4 and 8 blocks such a call was slower the more blocks there were (256 units of 131072 keys:
// allocation 156, 167, 174, 228 us, selection 219, 223, 240, 297 us), because every block pays for the fixed steps. With
// fewer units a team of up to 8 blocks per unit brings the call to about a block per SM, and a call with a few units (one
// layer), which is bound by the latency of its blocks, takes 8 keys per thread instead of 16. Measured, allocation + selection
// in us: 4 units of 32768 keys 11.9 + 7.6 with 8 blocks of 8 keys, 12.8 + 8.2 with 4 of 16; 32 of 8192, batch of 8, 9.7 + 8.8 with
// 2 of 8, 10.7 + 9.6 with one of 16; 4 of 8192, 448 rows, 9.7 + 6.6 and 10.8 + 7.6. Where 8 keys per thread make more than
// two blocks per SM, 16 would be as good or better: 40 units of 16384 13.9 + 9.7 with 4 of 8, 13.0 + 8.5 with 2 of 16; 80 of
// 5000 11.6 + 9.9 and 11.1 + 8.8; 16 of 20000 12.8 + 10.7 and 12.2 + 9.2. Teams that bring a call to half a block per SM instead
// of one: 32 of 65536 19.5 + 15.4 instead of 21.7 + 13.9, 112 of 12000 17.8 + 11.2 and 19.2 + 10.8; to two: 112 of 12000 24.2 + 16.2,
// 256 of 32768 42.8 + 33.3 instead of 35.0 + 24.5, 256 of 131072 122 + 85 instead of 101 + 85.
constexpr int kLongKeys = 262144;  // keys per block that a long kernel has bits for in shared memory
inline RankShape rank_shape(long long units, int n_max) {
  const int cap16 = kRankThreads * 16, cap8 = kRankThreads * 8;
  if (n_max <= cap8) return {8, 1};
  int team = 1, fit16 = 1, fit8 = 1;
  while (fit8 < kMaxTeam && (long long)fit8 * cap8 < n_max) fit8 *= 2;
  while (fit16 < kMaxTeam && (long long)fit16 * cap16 < n_max) fit16 *= 2;
  while (team < kMaxTeam && units * team < 148) team *= 2;
  if (team >= fit8 && (long long)fit8 * cap8 >= n_max) return {8, fit8};
  if (team >= fit16 && (long long)fit16 * cap16 >= n_max) return {16, fit16};
  while (team < kMaxTeam && (long long)team * kLongKeys < n_max) team *= 2;
  return {0, team < fit16 ? team : fit16};
}
// Words of shared memory that a block of a long kernel needs per kind of bit.
inline int long_words(int n_max, int team) {
  const int round = kRankThreads * 16 * team;
  return (n_max + round - 1) / round * (kRankThreads * 16 / 32 + kRankThreads * 16 / 1024);
}

// Launch of `units` teams, with programmatic stream serialisation (see launch_pdl).
template <typename... KArgs, typename... Args>
inline void launch_team(void (*kernel)(KArgs...), int units, int team, size_t smem, cudaStream_t st, Args... args) {
  launch_ex(kernel, dim3((unsigned)units * (unsigned)team), dim3(kRankThreads), smem, st, team, KArgs(args)...);
}

}  // namespace
}  // namespace madakv
