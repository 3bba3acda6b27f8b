// Shared pieces of the two ranking kernels (Eq. 9's count in allocate.cu, the top-budget selection in select.cu): the
// keys of one unit, spread over a team of 1-8 blocks, and the narrowing of a threshold to a short list of candidates.
//
// A unit's keys sit in registers (KPT consecutive positions per thread); a long unit in a call with few units is spread over
// a thread-block cluster, whose blocks exchange their partial results through distributed shared memory, and a unit
// longer than its blocks' registers is read twice by a kernel of its own (see rank_shape). The threshold (the budget-th
// largest key, or the key at which a mass is reached) is found in few steps. Two things bound these kernels: the integer
// instructions per key in calls with many units (an SM has some 230 000 keys of 256 units of 131072 keys to handle), and the
// fixed latency of a step (barriers, walking the buckets) in calls with few.
//   buckets  a count (and for Eq. 9 a mass, see allocate.cu) per key into 2048 buckets that are the same for all units, by
//            shared atomics without a result; a walk of the buckets narrows the range that the threshold can lie in to one
//            bucket, usually some tens of keys
//   list     the keys of the narrowed range are collected in shared memory, where half of a block's threads per modality
//            lay buckets over them once more; the few keys left are compared with one another
// Buckets over the range of each unit's keys needed a sweep for that range before; without it, and with long units read
// twice instead of three (allocation) or four times (selection), allocation + selection + compaction went from 602 to 483 us
// on 256 units of 131072 keys, from 618 to 523 on 1600 of 13411, from 213 to 161 on 3360 of 471, from 31 to 26 on 200 of 772.
// (The same in four or five passes of a plain radix descent: 750 us on the first of these.)
// Keys that crowd (many ties, a few values far away from all others) make the list overflow; then the buckets are laid
// over the narrowed range once more, and after that the range is bisected with exact sweeps over all keys, which ends
// for any input, at the latest when the range holds one value.
#pragma once

#include "common.cuh"

namespace madakv {
namespace {

constexpr unsigned int kFull = 0xffffffffu;
constexpr int kRankThreads = 512;
constexpr int kRankWarps = kRankThreads / 32;
constexpr int kHalf = kRankThreads / 2;        // threads per modality in the walks
constexpr int kListCap = 1024;                 // candidates per modality
constexpr int kFewCap = 32;                    // candidates compared with one another
constexpr int kMaxTeam = 8;
constexpr uint32_t kTopKey = 0x7f81ffffu;      // t = kTopKey - key: ascending t is descending importance
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
template <int KPT>
__device__ __forceinline__ void load_scores(const float* row, int mis, int n_max, int pos0, uint32_t (&t)[KPT]) {
  if (mis == 0 && pos0 + KPT <= n_max) {
#pragma unroll
    for (int j = 0; j < KPT; j += 4) {
      const float4 v = __ldg(reinterpret_cast<const float4*>(row + pos0 + j));
      t[j] = score_t(v.x);
      t[j + 1] = score_t(v.y);
      t[j + 2] = score_t(v.z);
      t[j + 3] = score_t(v.w);
    }
  } else if (mis != 0 && pos0 + KPT + 4 <= n_max) {
    // (a misaligned row has a unit before it: the pieces start inside the array; they end inside the row)
    float f[KPT + 4];
    const float4* src = reinterpret_cast<const float4*>(row + pos0 - mis);
#pragma unroll
    for (int j = 0; j < KPT + 4; j += 4) {
      const float4 v = __ldg(src + j / 4);
      f[j] = v.x;
      f[j + 1] = v.y;
      f[j + 2] = v.z;
      f[j + 3] = v.w;
    }
#pragma unroll
    for (int j = 0; j < KPT + 3; ++j) f[j] = (mis & 1) ? f[j + 1] : f[j];
#pragma unroll
    for (int j = 0; j < KPT; ++j) t[j] = score_t((mis & 2) ? f[j + 2] : f[j]);
  } else {
#pragma unroll
    for (int j = 0; j < KPT; ++j) t[j] = pos0 + j < n_max ? score_t(__ldg(row + pos0 + j)) : kTopKey;
  }
}
template <int KPT>
__device__ __forceinline__ uint32_t load_mask(const uint8_t* row, int n_max, int pos0) {  // bit j: position pos0 + j is visual
  const uintptr_t at = reinterpret_cast<uintptr_t>(row + pos0);
  uint32_t vis = 0;
  if (pos0 + KPT <= n_max && (at & (KPT - 1)) == 0) {
    uint32_t w[KPT / 4];
    if (KPT == 8) {
      const uint2 v = __ldg(reinterpret_cast<const uint2*>(row + pos0));
      w[0] = v.x;
      w[1] = v.y;
    } else {
#pragma unroll
      for (int j = 0; j < KPT / 16; ++j) {
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(row + pos0) + j);
        w[4 * j] = v.x;
        w[4 * j + 1] = v.y;
        w[4 * j + 2] = v.z;
        w[4 * j + 3] = v.w;
      }
    }
#pragma unroll
    for (int j = 0; j < KPT / 4; ++j) vis |= nonzero_bytes(w[j]) << (4 * j);
  } else if (pos0 >= 4 && pos0 + KPT + 4 <= n_max) {
    const uint32_t* src = reinterpret_cast<const uint32_t*>(at & ~(uintptr_t)3);
    const uint32_t sh = (uint32_t)(at & 3) * 8;
    uint32_t w = __ldg(src);
#pragma unroll
    for (int j = 0; j < KPT / 4; ++j) {
      const uint32_t nx = __ldg(src + j + 1);
      vis |= nonzero_bytes(__funnelshift_r(w, nx, sh)) << (4 * j);
      w = nx;
    }
  } else {
#pragma unroll
    for (int j = 0; j < KPT; ++j)
      if (pos0 + j < n_max && __ldg(row + pos0 + j)) vis |= 1u << j;
  }
  return vis;
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

// The first layout of the buckets is the same for all units, so that no sweep has to find the range of the keys before: 64
// buckets per octave from 512 down to 2^-23, the first and the last one take what lies outside. It is as fine as a
// layout over the range of importance values is (they spread over some twenty octaves).
constexpr int kMapShift = 17, kMapFirst = 7616;  // t >> 17 of the values from 512 up
constexpr int kDig = 11, kBuckets = 1 << kDig;

// ---- shared memory of a block
template <int TEAM, int WORDS>  // WORDS: count, or count and mass, per bucket
struct RankShared {
  static constexpr int kPer = kBuckets / (kHalf * TEAM);  // buckets per thread of the walk: 8, 4, 2, 1
  static constexpr int kStride = kBuckets;
  // the buckets' counts; once they are walked, the candidates of the whole team and the buckets of the finish (count,
  // mass low, mass high; one per thread and modality) take their place
  static constexpr int kFinish = 2 * kListCap + 6 * kHalf;
  static constexpr int kArea = 2 * WORDS * kStride > kFinish ? 2 * WORDS * kStride : kFinish;
  alignas(16) uint32_t cnt[kArea];
  uint32_t list[2][kListCap];                   // this block's candidates
  u64 wsum[2][kRankWarps];                      // per warp: masses (allocation)
  u64 slice_q[2][kMaxTeam];
  u64 wscan_q[kRankWarps], wscan_r[kRankWarps];
  u64 few_m[2][kFewCap];
  u64 first[2], last[2], first_q[2];            // walk: (count before << 32) | bucket, its count, mass before
  u64 fin_m[2];                                 // finish: mass before the range
  uint32_t slice_c[2][kMaxTeam];
  uint32_t wscan_c[kRankWarps], wcnt[2][kRankWarps], inexact;
  uint32_t few[2][kFewCap], few_n[2];
  uint32_t fin_c[2], fin_lo[2], fin_in[2], fin_more[2];
  uint32_t list_n;                              // candidates of this block: visual | text << 16
  uint32_t res[2][2];                           // selection: threshold, ties still wanted
  __device__ uint32_t* all(int m) { return cnt + m * kListCap; }  // the team's candidates
  __device__ uint32_t* fin_bucket(int m, int k) { return cnt + 2 * kListCap + (m * 3 + k) * kHalf; }
  __device__ uint32_t* candidates(int m) { return TEAM > 1 ? all(m) : list[m]; }
};

// What is known of modality m's threshold: t lies in [lo, lo + span], `in` keys of the modality do, `above` keys lie
// before lo. Identical in every thread of the team.
struct RankRange {
  uint32_t lo, span, in, above;
};
__device__ __forceinline__ int range_shift(uint32_t span, int dig) { return max(32 - __clz((int)span) - dig, 0); }

__device__ __forceinline__ uint32_t map_bucket(uint32_t t) {
  return (uint32_t)max(min((int)(t >> kMapShift) - kMapFirst, kBuckets - 1), 0);
}
// The range of t of bucket `at`, of the first layout or of one over g with 2^shift values of t per bucket.
__device__ __forceinline__ void bucket_range(RankRange& g, bool first, uint32_t at, int shift) {
  if (first) {
    g.lo = at ? (kMapFirst + at) << kMapShift : 0u;
    g.span = (at < kBuckets - 1 ? ((kMapFirst + at + 1) << kMapShift) - 1u : kTopKey) - g.lo;
  } else {
    const uint32_t cut = at << shift;
    g.span = min(g.span - cut, (1u << shift) - 1u);
    g.lo += cut;
  }
}
template <int TEAM, int WORDS>
__device__ __forceinline__ void zero_buckets(RankShared<TEAM, WORDS>& sh) {
  for (int x = threadIdx.x; x < 2 * WORDS * RankShared<TEAM, WORDS>::kStride / 4; x += kRankThreads)
    reinterpret_cast<uint4*>(sh.cnt)[x] = make_uint4(0, 0, 0, 0);
  if (threadIdx.x == 0) sh.list_n = 0;
  __syncthreads();
}

// This thread's words of the buckets, from word `at` on, added up over all blocks (the loads from distributed shared memory are
// in flight together).
template <int TEAM, int WORDS>
__device__ __forceinline__ void bucket_counts(const RankShared<TEAM, WORDS>& sh, uint32_t at,
                                              uint32_t (&c)[RankShared<TEAM, WORDS>::kPer]) {
  constexpr int kPer = RankShared<TEAM, WORDS>::kPer;
  const uint32_t* w = sh.cnt + at;
  if (TEAM == 1) {
#pragma unroll
    for (int k = 0; k < kPer; k += 4) {
      const uint4 v = *reinterpret_cast<const uint4*>(w + k);
      c[k] = v.x;
      c[(k + 1) % kPer] = v.y;
      c[(k + 2) % kPer] = v.z;
      c[(k + 3) % kPer] = v.w;
    }
  } else if (kPer == 1) {
    uint32_t v[TEAM];
#pragma unroll
    for (int r = 0; r < TEAM; ++r) v[r] = peer_load<TEAM>(w, r);
    c[0] = 0;
#pragma unroll
    for (int r = 0; r < TEAM; ++r) c[0] += v[r];
  } else {
    u64 v[TEAM][kPer / 2 + (kPer == 1)];
#pragma unroll
    for (int r = 0; r < TEAM; ++r)
#pragma unroll
      for (int k = 0; k < kPer / 2; ++k) v[r][k] = peer_load<TEAM>(reinterpret_cast<const u64*>(w) + k, r);
#pragma unroll
    for (int k = 0; k < kPer; ++k) c[k] = 0;
#pragma unroll
    for (int r = 0; r < TEAM; ++r)
#pragma unroll
      for (int k = 0; k < kPer / 2; ++k) {
        c[2 * k] += (uint32_t)v[r][k];
        c[(2 * k + 1) % kPer] += (uint32_t)(v[r][k] >> 32);
      }
  }
}

// A warp's candidates into the block's lists, as offsets from lo0 / lo1: bit j of in0 / in1 is set where the thread's j-th
// key belongs to the list of modality 0 / 1. One atomic per warp; candidates are few, so a thread picks them one by one.
template <int TEAM, int WORDS, int KPT>
__device__ __forceinline__ void append(RankShared<TEAM, WORDS>& sh, uint32_t in0, uint32_t in1, const uint32_t (&key)[KPT],
                                       uint32_t lo0, uint32_t lo1) {
  if (!__any_sync(kFull, (in0 | in1) != 0)) return;
  const int lane = threadIdx.x & 31;
  const uint32_t mine = __popc(in0) | (__popc(in1) << 16), incl = warp_scan32(mine);
  uint32_t base = 0;
  if (lane == 31) base = atomicAdd(&sh.list_n, incl);
  base = __shfl_sync(kFull, base, 31) + incl - mine;
  uint32_t o0 = base & 0xffffu, o1 = base >> 16;
  for (uint32_t left = in0 | in1; left; left &= left - 1) {
    const int j = __ffs(left) - 1;
    uint32_t k = key[0];
#pragma unroll
    for (int x = 1; x < KPT; ++x) k = x == j ? key[x] : k;
    if ((in0 >> j) & 1u) sh.list[0][o0++] = k - lo0;
    else sh.list[1][o1++] = k - lo1;
  }
}

// The same for a unit that is not in registers: positions instead of keys (the keys are read again when the list is complete).
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

// All blocks' candidates into this block (warp r copies block r's); returns their number, visual | text << 16. A block on
// its own has them already. Ends with a barrier of the block.
template <int TEAM, int WORDS>
__device__ __forceinline__ uint32_t gather_lists(RankShared<TEAM, WORDS>& sh) {
  if (TEAM == 1) return sh.list_n;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t n = lane < TEAM ? peer_load<TEAM>(&sh.list_n, lane) : 0u;
  const uint32_t incl = warp_scan32(n), total = __shfl_sync(kFull, incl, 31);
  if (warp < TEAM) {
    const uint32_t k = __shfl_sync(kFull, n, warp), to = __shfl_sync(kFull, incl, warp) - k;
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      const uint32_t km = m ? k >> 16 : k & 0xffffu, at = m ? to >> 16 : to & 0xffffu;
      for (uint32_t x = lane; x < km; x += 32) sh.all(m)[at + x] = peer_load<TEAM>(&sh.list[m][x], warp);
    }
  }
  __syncthreads();
  return total;
}

// The whole block: where among the candidates (offsets into rg[m]) the thresholds lie, half of the threads per modality. need: a
// mass (with kMass; `before` is the exact mass before the range) or a count. Leaves in shared memory, per modality: fin_lo
// (the smallest t up to which the threshold is reached), fin_c and fin_m (count and mass before it), fin_in (candidates
// that equal it). A modality that is not `on` is left out. Ends with a barrier of the block.
template <int TEAM, int WORDS, bool kMass>
__device__ __forceinline__ void finish_lists(RankShared<TEAM, WORDS>& sh, const RankRange& r0, const RankRange& r1, uint32_t got, bool on0,
                                             bool on1, u64 need0, u64 need1, u64 before0, u64 before1) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, m = tid / kHalf, i = tid % kHalf;
  const uint32_t n = m ? got >> 16 : got & 0xffffu, base = m ? r1.lo : r0.lo;
  const bool on = m ? on1 : on0;
  const u64 need = m ? need1 : need0;
  const uint32_t* list = sh.candidates(m);
  uint32_t lo = 0, span = m ? r1.span : r0.span, in = n, above_c = m ? r1.above : r0.above;
  u64 above = m ? before1 : before0;
  uint32_t *fc = sh.fin_bucket(m, 0), *flo = sh.fin_bucket(m, 1), *fhi = sh.fin_bucket(m, 2);
  auto mass = [&](uint32_t x) { return psi_fix(kTopKey - (base + x)); };
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
  // the keys left, compared with one another by one warp per modality
  if (on && span > 0)
    for (uint32_t x = i; x < n; x += kHalf) {
      const uint32_t v = list[x];
      if (v - lo <= span) {
        const uint32_t s = atomicAdd(&sh.few_n[m], 1u);
        if (s < kFewCap) {
          sh.few[m][s] = v;
          if (kMass) sh.few_m[m][s] = mass(v);
        }
      }
    }
  __syncthreads();
  if (on && i < 32) {
    uint32_t at = lo, equal = in;
    if (span > 0) {
      const uint32_t v = lane < (int)in ? sh.few[m][lane] : kNoKey;
      uint32_t lt_c = 0, eq_c = 0;
      u64 lt = 0, eq = 0;
#pragma unroll 4
      for (uint32_t j = 0; j < in; ++j) {
        const uint32_t o = sh.few[m][j];
        if (o < v) ++lt_c;
        if (o == v) ++eq_c;
        if (kMass) {
          const u64 q = sh.few_m[m][j];
          if (o < v) lt += q;
          if (o == v) eq += q;
        }
      }
      const bool ok = lane < (int)in && (kMass ? above + lt + eq >= need : above_c + lt_c + eq_c >= need);
      at = __reduce_min_sync(kFull, ok ? v : kNoKey);
      const int who = max(__ffs(__ballot_sync(kFull, ok && v == at)) - 1, 0);
      equal = __shfl_sync(kFull, eq_c, who);
      above_c += __shfl_sync(kFull, lt_c, who);
      if (kMass) above += __shfl_sync(kFull, lt, who);
    }
    if (lane == 0) {
      sh.fin_lo[m] = base + at;
      sh.fin_in[m] = equal;
      sh.fin_c[m] = above_c;
      if (kMass) sh.fin_m[m] = above;
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
// layer), which is bound by the latency of its blocks, takes 8 keys per thread instead of 16 (4 units of 32768 keys: 12.8 +
// 10.9 us with 8 blocks of 8 keys, 15.5 + 13.7 with 4 blocks of 16, 30 + 54 with one block per unit).
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
