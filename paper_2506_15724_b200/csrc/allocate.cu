// Stages 2-3: modality masses and preference (Eq. 6, Eq. 8), sparsity counts (Eq. 9), layer compensation
// (Eq. 10-11) and the integer per-head, per-modality budgets.
//
// All sums of psi are exact: psi is mapped to 2^-32 fixed point (psi_fix) and added as 64-bit integers, so the
// results do not depend on the order of summation or on the launch shape. Eq. 9 is a "top-p" count: the number of
// largest keys whose mass reaches theta * W_m. The layer recurrence is a scalar fp64 scan per sequence with
// explicitly rounded operations (no FMA contraction), so it is reproducible bit for bit.
#include "rank_common.cuh"

namespace madakv {
namespace {

struct AllocParams {
  const float* psi;
  const uint8_t* mask;
  const int32_t* seq_len;
  const int32_t* budget;
  double* mass;
  double* pref;
  int32_t* demand;
  double* phi;
  int32_t* budgets;
  int L, Hkv, n_max, mpa, hcc_mode, keep_window, window, rows;  // rows: window rows per KV head
  u64 theta_fix;  // floor(theta * 2^32)
  unsigned* counter;  // one per sequence, zero between calls: the units that are done; null: masses and demands only
  int depth, layer;   // one layer of a pass over `depth` layers (the arrays hold that layer, L = 1), or layer = -1: all layers
};

// Visual tokens among the first n of a sequence, counted by the whole block into *s_nv (which the caller has zeroed
// behind a barrier); the caller synchronises before reading it.
__device__ __forceinline__ void count_visual(const uint8_t* mask, int n, int* s_nv) {
  int c = 0;
  if ((reinterpret_cast<uintptr_t>(mask) & 15) == 0) {  // 16 tokens per load
    const int n16 = n >> 4;
#pragma unroll 4
    for (int i = threadIdx.x; i < n16; i += blockDim.x) {
      const uint4 v = __ldg(reinterpret_cast<const uint4*>(mask) + i);
      const uint32_t w4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int k = 0; k < 4; ++k)  // a byte counts if it is not zero
        c += __popc(((w4[k] | (w4[k] >> 1) | (w4[k] >> 2) | (w4[k] >> 3) | (w4[k] >> 4) | (w4[k] >> 5) | (w4[k] >> 6) |
                      (w4[k] >> 7)) & 0x01010101u));
    }
#pragma unroll 1
    for (int i = (n16 << 4) + threadIdx.x; i < n; i += blockDim.x) c += mask[i] ? 1 : 0;
  } else {
#pragma unroll 1
    for (int i = threadIdx.x; i < n; i += blockDim.x) c += mask[i] ? 1 : 0;
  }
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) c += __shfl_xor_sync(0xffffffffu, c, off);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(s_nv, c);
}
// The layer's integer budget Phi^l from phi^l, and phi^{l+1} (Eq. 10-11); l counts from 1, the update exists for l < L.
__device__ __forceinline__ double rounded_budget(double ph, double lo, double hi) {
  return fmin(fmax(floor(__dadd_rn(ph, 0.5)), lo), hi);
}
// The divisor of Eq. 11 for the step from layer l (0 for a mode without one) and its correctly rounded reciprocal: both
// are known before the recurrence starts.
__device__ __forceinline__ double phi_divisor(int Hkv, int L, int l, int hcc_mode) {
  if (hcc_mode == MADAKV_HCC_PAPER || hcc_mode == MADAKV_HCC_DEMAND) return (double)((long long)Hkv * (L - l));  // per-head units
  return hcc_mode == MADAKV_HCC_LITERAL ? (double)(L - l) : 0.0;  // Eq. 11 as printed
}
// K / div rounded to nearest, with the reciprocal at hand: the quotient of the product is within one unit in the last
// place, and one correction by the exact remainder makes it the correctly rounded one (Markstein, "Computation of
// elementary functions on the IBM RISC System/6000 processor", 1990). Three dependent operations instead of a division in
// a chain that is one layer after the other (llava: 11.8 us for the 32 layers with divisions).
__device__ __forceinline__ double next_phi(double ph, double dem, int Hkv, double div, double rcp, double lo, double hi) {
  const double K = __dsub_rn(dem, __dmul_rn((double)Hkv, ph));  // Eq. 10
  const double q = __dmul_rn(K, rcp);
  const double quot = __fma_rn(__fma_rn(-q, div, K), rcp, q);
  const double next = div > 0.0 ? __dsub_rn(ph, quot) : ph;  // Eq. 11
  return next < lo ? lo : (next > hi ? hi : next);  // (never NaN; both comparisons at once)
}
// Eq. 8 integerised for one head: the visual share rounded half up, the rest to text, surplus of a modality with too
// few tokens passed to the other. With `keep_demand` (mode DEMAND, every layer but the last) the head keeps what
// Eq. 9 asked for instead. lo_v, lo_t: the proxy tokens of each modality when they are retained unconditionally
// (cfg->keep_window), else 0: budgets are floored at them, the head's total at their sum.
__device__ __forceinline__ void split_budget(const AllocParams& p, int64_t u, double pref_v, int2 dem, double Phi, int n, int n_v, int n_t,
                                             int lo_v, int lo_t, bool keep_demand) {
  if (keep_demand) {
    p.budgets[u * 2] = p.mpa ? max(dem.x, lo_v) : 0;
    p.budgets[u * 2 + 1] = p.mpa ? max(dem.y, lo_t) : min(max(dem.x + dem.y, lo_v + lo_t), n);
    return;
  }
  const int P = max((int)Phi, lo_v + lo_t);
  int bv, bt;
  if (p.mpa) {
    bv = (int)floor(__dadd_rn(__dmul_rn(pref_v, Phi), 0.5));  // Eq. 8, rounded half up
    bv = min(max(bv, lo_v), P - lo_t);
    bt = P - bv;
    if (bv > n_v) { bt += bv - n_v; bv = n_v; }
    if (bt > n_t) { bv = min(n_v, bv + (bt - n_t)); bt = n_t; }
  } else {
    bv = 0;
    bt = min(P, n);
  }
  p.budgets[u * 2] = bv;
  p.budgets[u * 2 + 1] = bt;
}

// What is left once all units of sequence b have their masses and demands, by one block: Eq. 10-11 as a scalar scan over the
// layers (or one step of it), then Eq. 8 integerised for every (layer, head). n_v: the sequence's visual tokens; ph: phi of the
// first layer. What bounds it is a chain of latencies, so demands and preferences are read together, before anything else,
// and the scan finds its operands converted and a layer ahead. (Read where they were used, with the scan's conversions
// in its chain, 11700 clocks for 2 layers of 4 heads, a whole all-layer call of 32 layers 10.7 us.)
constexpr int kLayerChunk = 512;
constexpr int kUnitChunk = 2048;  // units whose demands are summed from shared memory
constexpr int kBudgetBytes = 4 * (kLayerChunk + 1) * 8 + kUnitChunk * 4;
__device__ __forceinline__ double first_phi(const AllocParams& p, int b) {
  return p.layer > 0 ? p.phi[(int64_t)b * p.depth + p.layer] : (double)p.budget[b];
}
__device__ __noinline__ void sequence_budgets(const AllocParams& p, int b, int n, int n_v, double ph, double* s_phi) {
  __shared__ int s_wv;
  double *s_rcp = s_phi + kLayerChunk + 1, *s_div = s_rcp + kLayerChunk + 1, *s_dem = s_div + kLayerChunk + 1;
  int* s_unit = reinterpret_cast<int*>(s_dem + kLayerChunk + 1);
  constexpr int U = 2;  // units per thread whose demand and preference stay in registers
  const int tid = threadIdx.x, nt = blockDim.x;
  const int wlen = p.keep_window ? min(p.window, n) : 0;  // proxy tokens retained unconditionally
  const double lo = n >= 1 ? 1.0 : 0.0, hi = (double)n;
  const int depth = p.depth, first = max(p.layer, 0);  // the layers of the arrays: first .. first + L - 1 of depth
  const int chunk = min(kLayerChunk, max(1, kUnitChunk / p.Hkv));
  for (int l0 = 0; l0 < p.L; l0 += chunk) {
    const int ln = min(chunk, p.L - l0), units = ln * p.Hkv;
    const int64_t u0 = ((int64_t)b * p.L + l0) * p.Hkv;
    auto unit_demand = [&](int x) { return __ldcg(reinterpret_cast<const int2*>(p.demand) + u0 + x); };
    double pref[U];
    int2 dem[U];
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const int x = tid + j * nt;
      pref[j] = 0.0;
      dem[j] = make_int2(0, 0);
      if (x < units) {
        pref[j] = __ldcg(p.pref + (u0 + x) * 2);
        dem[j] = unit_demand(x);
      }
    }
    if (l0 == 0 && tid == 0) s_wv = 0;
#pragma unroll 1
    for (int l = tid; l < ln; l += nt) {
      const double div = first + l0 + l + 1 < depth ? phi_divisor(p.Hkv, depth, first + l0 + l + 1, p.hcc_mode) : 0.0;
      s_div[l] = div;
      s_rcp[l] = div > 0.0 ? __drcp_rn(div) : 0.0;
    }
    const bool in_shared = units <= kUnitChunk;
    if (in_shared) {
#pragma unroll
      for (int j = 0; j < U; ++j)
        if (tid + j * nt < units) s_unit[tid + j * nt] = dem[j].x + dem[j].y;
#pragma unroll 1
      for (int x = tid + U * nt; x < units; x += nt) {
        const int2 d = unit_demand(x);
        s_unit[x] = d.x + d.y;
      }
    }
    __syncthreads();
    if (l0 == 0 && wlen > 0) count_visual(p.mask + (int64_t)b * p.n_max + (n - wlen), wlen, &s_wv);
    // Eq. 10's sum over heads (integers: any order gives the same sum)
    if (in_shared) {
#pragma unroll 1
      for (int l = tid; l < ln; l += nt) {
        long long sum = 0;
#pragma unroll 4
        for (int h = 0; h < p.Hkv; ++h) sum += s_unit[l * p.Hkv + h];
        s_dem[l] = (double)sum;
      }
    } else if (tid < 32) {  // one layer of very many heads
      long long sum = 0;
#pragma unroll 1
      for (int x = tid; x < units; x += 32) {
        const int2 d = unit_demand(x);
        sum += (long long)d.x + d.y;
      }
#pragma unroll
      for (int off = 16; off >= 1; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
      if (tid == 0) s_dem[0] = (double)sum;
    }
    __syncthreads();
    if (tid == 0) {
      double rcp = s_rcp[0], div = s_div[0], dm = s_dem[0];
#pragma unroll 1
      for (int l = 0; l < ln; ++l) {
        const double r1 = s_rcp[l + 1], d1 = s_div[l + 1], m1 = s_dem[l + 1];  // (the last ones are not used)
        s_phi[l] = ph;
        if (first + l0 + l + 1 < depth) ph = next_phi(ph, dm, p.Hkv, div, rcp, lo, hi);  // (the paper counts layers from 1)
        rcp = r1;
        div = d1;
        dm = m1;
      }
      if (p.layer >= 0 && first + 1 < depth) p.phi[(int64_t)b * depth + first + 1] = ph;
    }
    __syncthreads();
    const int n_t = n - n_v;
    const int lo_v = p.mpa ? s_wv : 0, lo_t = wlen - lo_v;
#pragma unroll 1
    for (int l = tid; l < ln; l += nt)
      if (p.layer <= 0) p.phi[(int64_t)b * depth + l0 + l] = s_phi[l];
#pragma unroll 1
    for (int x = tid; x < units; x += nt) {  // (one copy of the code: it is run once)
      const bool again = x >= U * nt;
      const bool second = x >= nt;
      const double pv = again ? __ldcg(p.pref + (u0 + x) * 2) : second ? pref[1] : pref[0];
      const int2 d = again ? unit_demand(x) : second ? dem[1] : dem[0];
      const int l = x / p.Hkv;
      split_budget(p, u0 + x, pv, d, rounded_budget(s_phi[l], lo, hi), n, n_v, n_t, lo_v, lo_t,
                   p.hcc_mode == MADAKV_HCC_DEMAND && first + l0 + l + 1 < depth);
    }
    __syncthreads();
  }
}

// The ranges Eq. 9's two thresholds can lie in, with the exact masses before them, the masses to reach and the modalities' own.
template <int CAP>  // candidates that fit the list
struct MassRanges {
  RankRange r0, r1;
  u64 above0, above1, need0, need1, W0, W1;
  bool exact;
  uint32_t n_vis;  // visual tokens
  __device__ __forceinline__ bool listed() const { return r0.in <= CAP && r1.in <= CAP; }
  __device__ __forceinline__ bool crowded0() const { return r0.in > CAP && r0.span > 0; }
  __device__ __forceinline__ bool crowded1() const { return r1.in > CAP && r1.span > 0; }
};
// The mass to reach, Eq. 9: theta_fix * W has 96 bits; the prefix test  prefix * 2^32 >= theta_fix * W  is
// prefix >= ceil(theta_fix * W / 2^32)
__device__ __forceinline__ u64 mass_target(u64 theta_fix, u64 W) {
  const u64 hi = __umul64hi(theta_fix, W), lo = theta_fix * W;
  return (hi << 32) + (lo >> 32) + ((lo & 0xffffffffull) ? 1ull : 0ull);
}

// A bucket holds a count and the sum of a word per key, two shared atomics without a result, which is enough for the exact mass
// (bucket_map.cuh). A unit with a bucket for which it is not (mass_known: ten thousands of nearly equal scores), or with scores of
// 512 and more, goes the slow way: exact sweeps that halve the range.
// (Exact 64-bit masses by atomics that return the old word, to detect carries: alloc 52 us on llava.)
template <int TEAM>
__device__ __forceinline__ void add_key(uint32_t* at, uint32_t t) {
  atomicAdd(at, 1u);
  atomicAdd(at + 2 * RankShared<TEAM, 2>::kStride, mass_word(t));
}
template <int KPT, int TEAM>
__device__ __forceinline__ void add_first(RankShared<TEAM, 2>& sh, const BucketMap& map, const uint32_t (&t)[KPT], uint32_t vis, uint32_t valid) {
  constexpr int kStride = RankShared<TEAM, 2>::kStride;
  if (valid == valid_bits<KPT>(KPT, 0)) {
#pragma unroll
    for (int j = 0; j < KPT; ++j) add_key<TEAM>(sh.cnt + ((vis >> j) & 1u ? 0 : kStride) + map_bucket(map, t[j]), t[j]);
  } else {
#pragma unroll
    for (int j = 0; j < KPT; ++j)
      if ((valid >> j) & 1u) add_key<TEAM>(sh.cnt + ((vis >> j) & 1u ? 0 : kStride) + map_bucket(map, t[j]), t[j]);
  }
}
template <int KPT, int TEAM>
__device__ __forceinline__ void add_again(RankShared<TEAM, 2>& sh, const MassRanges<RankShared<TEAM, 2>::kCap>& g, const uint32_t (&t)[KPT], uint32_t vis, int shift0,
                                          int shift1) {
#pragma unroll
  for (int j = 0; j < KPT; ++j) {
    const bool v = (vis >> j) & 1u;
    const uint32_t x = t[j] - (v ? g.r0.lo : g.r1.lo);
    if (x <= (v ? g.r0.span : g.r1.span)) add_key<TEAM>(sh.cnt + (v ? 0 : RankShared<TEAM, 2>::kStride) + (x >> (v ? shift0 : shift1)), t[j]);
  }
}

// Walk of the buckets (of the first layout, `map`, or of one over the ranges): the ranges shrink to the buckets in which the
// masses are reached (if all sums are exact).
template <int TEAM>
__device__ __forceinline__ void mass_walk(RankShared<TEAM, 2>& sh, uint32_t rank, const BucketMap* map, u64 theta_fix,
                                          MassRanges<RankShared<TEAM, 2>::kCap>& g, int shift0, int shift1) {
  walk<TEAM, 2>(
      sh, rank,
      [&](int m, int b) {
        const int shift = m ? shift1 : shift0;
        return map ? bucket_start(*map, b) : BucketStart{(m ? g.r1.lo : g.r0.lo) + ((uint32_t)b << shift), shift, false};
      },
      [&](int m, u64 W) { return map ? mass_target(theta_fix, W) : (m ? g.need1 - g.above1 : g.need0 - g.above0); });
  g.exact = !(sh.found[0].inexact | sh.found[1].inexact);
  if (map) {
    g.n_vis = sh.found[0].total;
    g.W0 = sh.found[0].mass;
    g.W1 = sh.found[1].mass;
    g.need0 = mass_target(theta_fix, g.W0);
    g.need1 = mass_target(theta_fix, g.W1);
  }
  auto narrow = [&](RankRange& r, u64& above, u64 need, const Found& f, int shift) {
    if (!need) {  // nothing to reach
      r = RankRange{kNowhere, 0u, 0u, 0u};
      return;
    }
    bucket_range(r, map, f.at, shift);
    r.above += f.above;
    r.in = f.in;
    above += f.above_q;
  };
  if (g.exact) {
    narrow(g.r0, g.above0, g.need0, sh.found[0], shift0);
    narrow(g.r1, g.above1, g.need1, sh.found[1], shift1);
  }
}

// (Rare) too many keys in a range, or sums that were not exact: halve it with exact sweeps until its keys fit the list or
// are all alike. `sweep` calls its argument with the keys of the thread, some at a time.
template <int TEAM, typename Sweep>
__device__ __forceinline__ void mass_bisect(RankShared<TEAM, 2>& sh, uint32_t rank, u64 theta_fix,
                                            MassRanges<RankShared<TEAM, 2>::kCap>& g, Sweep sweep) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // sums over the team, into every thread (of values that are already summed up over the warp)
  auto team_sums = [&](u64& a0, u64& a1) {
    __syncthreads();
    if (lane == 0) {
      sh.wsum[0][warp] = a0;
      sh.wsum[1][warp] = a1;
    }
    __syncthreads();
    if (warp == 0) {
      const u64 t0 = warp_sum64(lane < kRankWarps ? sh.wsum[0][lane] : 0ull);
      const u64 t1 = warp_sum64(lane < kRankWarps ? sh.wsum[1][lane] : 0ull);
      if (lane < TEAM) {
        peer_store<TEAM>(&sh.slice_q[0][rank], lane, t0);
        peer_store<TEAM>(&sh.slice_q[1][rank], lane, t1);
      }
    }
    team_sync<TEAM>();
    a0 = warp_sum64(lane < TEAM ? sh.slice_q[0][lane] : 0ull);
    a1 = warp_sum64(lane < TEAM ? sh.slice_q[1][lane] : 0ull);
    team_sync<TEAM>();
  };
  if (!g.exact) {
    u64 W0 = 0, W1 = 0;
    uint32_t c0 = 0, c1 = 0;
    sweep([&](uint32_t t, bool v) {
      if (t != kNoKey) {
        const u64 q = psi_fix(kTopKey - t);
        if (v) { W0 += q; ++c0; } else { W1 += q; ++c1; }
      }
    });
    W0 = warp_sum64(W0);
    W1 = warp_sum64(W1);
    team_sums(W0, W1);
    u64 n0 = __reduce_add_sync(kFull, c0), n1 = __reduce_add_sync(kFull, c1);
    team_sums(n0, n1);
    g.n_vis = (uint32_t)n0;
    g.W0 = W0;
    g.W1 = W1;
    g.need0 = mass_target(theta_fix, W0);
    g.need1 = mass_target(theta_fix, W1);
    g.r0 = g.need0 ? RankRange{0u, kTopKey, (uint32_t)n0, 0u} : RankRange{kNowhere, 0u, 0u, 0u};
    g.r1 = g.need1 ? RankRange{0u, kTopKey, (uint32_t)n1, 0u} : RankRange{kNowhere, 0u, 0u, 0u};
    g.above0 = g.above1 = 0;
  }
  while (g.crowded0() || g.crowded1()) {
    const bool on0 = g.crowded0(), on1 = g.crowded1();
    const uint32_t mid0 = g.r0.lo + (g.r0.span >> 1), mid1 = g.r1.lo + (g.r1.span >> 1);
    u64 a0 = 0, a1 = 0;
    uint32_t c0 = 0, c1 = 0;
    sweep([&](uint32_t t, bool v) {
      if ((v ? on0 : on1) && t >= (v ? g.r0.lo : g.r1.lo) && t <= (v ? mid0 : mid1)) {
        const u64 q = psi_fix(kTopKey - t);
        if (v) { a0 += q; ++c0; } else { a1 += q; ++c1; }
      }
    });
    a0 = warp_sum64(a0);
    a1 = warp_sum64(a1);
    team_sums(a0, a1);
    u64 n0 = __reduce_add_sync(kFull, c0), n1 = __reduce_add_sync(kFull, c1);
    team_sums(n0, n1);
    auto halve = [](RankRange& r, u64& above, u64 need, u64 a, uint32_t c) {
      const uint32_t half = r.span >> 1;
      if (above + a >= need) {
        r.span = half;
        r.in = c;
      } else {
        above += a;
        r.above += c;
        r.in -= c;
        r.lo += half + 1;
        r.span -= half + 1;
      }
    };
    if (on0) halve(g.r0, g.above0, g.need0, a0, (uint32_t)n0);
    if (on1) halve(g.r1, g.above1, g.need1, a1, (uint32_t)n1);
  }
}

// With all candidates on their way to block 0's list: it finds the counts and writes the unit's results; the unit that is
// done last goes on with its sequence (ph: phi of its first layer).
template <int TEAM>
__device__ __forceinline__ void mass_finish(RankShared<TEAM, 2>& sh, const AllocParams& p, uint32_t rank, int u, int b, int n, double ph,
                                            const MassRanges<RankShared<TEAM, 2>::kCap>& g) {
  constexpr uint32_t kCap = RankShared<TEAM, 2>::kCap;
  const int tid = threadIdx.x;
  team_sync<TEAM>();  // (the last access to another block's shared memory)
  if (rank != 0) return;
  const bool on0 = g.need0 && g.r0.in <= kCap, on1 = g.need1 && g.r1.in <= kCap;
  finish_lists<TEAM, 2, true>(sh, g.r0, g.r1, on0, on1, g.need0, g.need1, g.above0, g.above1);
  if (tid < 2) {
    const u64 need = tid ? g.need1 : g.need0;
    uint32_t count = 0;
    if (need) {
      // every key left has the value kTopKey - t: as few of them as reach the threshold
      const RankRange my = tid ? g.r1 : g.r0;
      const bool listed = tid ? on1 : on0;
      uint32_t take = listed ? sh.fin_in[tid] : my.in;
      if (take > 1) {
        const u64 above = listed ? sh.fin_m[tid] : (tid ? g.above1 : g.above0);
        const u64 each = psi_fix(kTopKey - (listed ? sh.fin_lo[tid] : my.lo));
        if (each > 0) {
          const u64 k = (need - above + each - 1) / each;
          if (k < (u64)take) take = (uint32_t)k;
        }
      }
      count = (listed ? sh.fin_c[tid] : my.above) + take;
    }
    p.demand[(int64_t)u * 2 + tid] = (int32_t)count;
  } else if (tid >= 32 && tid < 34) {
    const int m = tid - 32;
    const u64 W = m ? g.W1 : g.W0, tot = g.W0 + g.W1;
    p.mass[(int64_t)u * 2 + m] = __ull2double_rn(W) / 4294967296.0;
    p.pref[(int64_t)u * 2 + m] = tot ? __ddiv_rn(__ull2double_rn(W), __ull2double_rn(tot)) : 0.0;
  }
  if (!p.counter) return;
  __shared__ unsigned s_last;
  __syncthreads();
  if (tid == 0) s_last = arrive_inc(p.counter + b, (unsigned)(p.L * p.Hkv) - 1u);  // (wraps to 0: ready for the next call)
  __syncthreads();
  if (s_last != (unsigned)(p.L * p.Hkv) - 1u) return;
  static_assert(sizeof(sh.cnt) >= kBudgetBytes, "the scan reuses the buckets");
  sequence_budgets(p, b, n, (int)g.n_vis, ph, reinterpret_cast<double*>(sh.cnt));
}

// t of KPT consecutive positions (kNoKey outside the sequence); returns those that are inside.
template <int KPT>
__device__ __forceinline__ uint32_t take_valid(const RawScores<KPT>& raw, int mis, int n, int pos0, uint32_t (&t)[KPT]) {
  take_scores<KPT>(raw, mis, t);
  const uint32_t valid = valid_bits<KPT>(n, pos0);
  if (valid != valid_bits<KPT>(KPT, 0)) {
#pragma unroll
    for (int j = 0; j < KPT; ++j)
      if (!((valid >> j) & 1u)) t[j] = kNoKey;
  }
  return valid;
}
template <int KPT>
__device__ __forceinline__ uint32_t load_valid(const float* psi, int mis, int n_max, int n, int pos0, uint32_t (&t)[KPT]) {
  RawScores<KPT> raw;
  issue_scores<KPT>(psi, mis, n_max, pos0, raw);
  return take_valid<KPT>(raw, mis, n, pos0, t);
}

// Masses, preference and Eq. 9's counts of one unit whose keys fit the registers of its team (see rank_common.cuh). (A
// team clears its buckets, and its blocks learn of one another, under the kernel before; blocks on their own, which may be
// several rounds of them, while their loads are on the way.)
template <int KPT, int TEAM>
__global__ void __launch_bounds__(kRankThreads, 2) alloc_unit_kernel(const __grid_constant__ AllocParams p) {
  constexpr uint32_t kCap = RankShared<TEAM, 2>::kCap;
  __shared__ RankShared<TEAM, 2> sh;
  team_started<TEAM>();
  if (TEAM > 1) zero_buckets<TEAM, 2>(sh);
  pdl_wait();
  pdl_go();
  const uint32_t rank = TEAM > 1 ? team_rank() : 0u;
  const int u = blockIdx.x / TEAM, b = u / (p.Hkv * p.L);
  const int pos0 = (int)rank * kRankThreads * KPT + threadIdx.x * KPT;  // a block owns consecutive positions
  const int mis = (int)(((int64_t)u * p.n_max) & 3);
  RawScores<KPT> raw;
  RawMask<KPT> raw_mask;
  issue_scores<KPT>(p.psi + (int64_t)u * p.n_max, mis, p.n_max, pos0, raw);
  issue_mask<KPT>(p.mask + (int64_t)b * p.n_max, p.n_max, pos0, raw_mask);
  if (TEAM == 1) zero_buckets<TEAM, 2>(sh);
  const int n = clamped_len(p.seq_len, b, p.n_max);
  const double ph = p.counter ? first_phi(p, b) : 0.0;
  uint32_t t[KPT];
  const uint32_t valid = take_valid<KPT>(raw, mis, n, pos0, t), vis = take_mask<KPT>(raw_mask);
  const BucketMap map = bucket_map(p.rows, n);
  __syncthreads();
  add_first<KPT, TEAM>(sh, map, t, vis, valid);
  MassRanges<kCap> g = {};
  team_wait_started<TEAM>();
  mass_walk<TEAM>(sh, rank, &map, p.theta_fix, g, 0, 0);
  bool swept = false;
  if (!g.exact || !g.listed()) {
    if (g.exact) {
      const int shift0 = range_shift(g.r0.span, kDig), shift1 = range_shift(g.r1.span, kDig);
      team_sync<TEAM>();
      zero_buckets<TEAM, 2>(sh);
      __syncthreads();
      add_again<KPT, TEAM>(sh, g, t, vis, shift0, shift1);
      mass_walk<TEAM>(sh, rank, nullptr, p.theta_fix, g, shift0, shift1);
    }
    if (!g.exact || g.crowded0() || g.crowded1()) {
      mass_bisect<TEAM>(sh, rank, p.theta_fix, g, [&](auto each) {
#pragma unroll
        for (int j = 0; j < KPT; ++j) each(t[j], (vis >> j) & 1u);
      });
      swept = true;
    }
  }
  uint32_t in = 0;
#pragma unroll
  for (int j = 0; j < KPT; ++j) {
    const bool v = (vis >> j) & 1u;
    if (t[j] - (v ? g.r0.lo : g.r1.lo) <= (v ? g.r0.span : g.r1.span)) in |= 1u << j;
  }
  const uint32_t in0 = g.r0.in <= kCap ? in & vis : 0u, in1 = g.r1.in <= kCap ? in & ~vis : 0u;
  if (swept) find_places<TEAM, 2>(sh, rank, __popc(in0), __popc(in1));
  append<TEAM, 2, KPT, false>(sh, rank, in0, in1, t, g.r0.lo, g.r1.lo);
  mass_finish<TEAM>(sh, p, rank, u, b, n, ph, g);
}

// The same for a longer unit, which is read twice, for the buckets and for the candidates (listed as positions); the mask is
// kept as bits in shared memory. (256 units of 131072 keys: 111 us; 153 with three sweeps over keys and mask.)
template <int TEAM>
__global__ void __launch_bounds__(kRankThreads, 2) alloc_long_kernel(const __grid_constant__ AllocParams p) {
  constexpr int KPT = 16, kRound = kRankThreads * KPT;
  constexpr uint32_t kCap = RankShared<TEAM, 2>::kCap;
  __shared__ RankShared<TEAM, 2> sh;
  extern __shared__ __align__(16) uint32_t bits[];
  team_started<TEAM>();
  zero_buckets<TEAM, 2>(sh);
  pdl_wait();
  pdl_go();
  const uint32_t rank = TEAM > 1 ? team_rank() : 0u;
  const int tid = threadIdx.x, u = blockIdx.x / TEAM, b = u / (p.Hkv * p.L);
  const int n = clamped_len(p.seq_len, b, p.n_max);
  const double ph = p.counter ? first_phi(p, b) : 0.0;
  const float* psi = p.psi + (int64_t)u * p.n_max;
  const int mis = (int)(((int64_t)u * p.n_max) & 3);
  const uint8_t* mask = p.mask + (int64_t)b * p.n_max;
  uint32_t *pos0 = bits, *pos1 = bits + kListCap, *vis_w = bits + 2 * kListCap;
  const int rounds = (n + kRound * TEAM - 1) / (kRound * TEAM);
  const int start = (int)rank * rounds * kRound;  // a block owns consecutive positions
  const BucketMap map = bucket_map(p.rows, n);
  __syncthreads();
#pragma unroll 1
  for (int r = 0; r < rounds; ++r) {
    const int at = start + r * kRound + tid * KPT;
    uint32_t t[KPT];
    const uint32_t valid = load_valid<KPT>(psi, mis, p.n_max, n, at, t);
    const uint32_t vis = load_mask<KPT>(mask, p.n_max, at);
    bits_of_thread(vis_w, r) = (uint16_t)vis;
    add_first<KPT, TEAM>(sh, map, t, vis, valid);
  }
  MassRanges<kCap> g = {};
  team_wait_started<TEAM>();
  mass_walk<TEAM>(sh, rank, &map, p.theta_fix, g, 0, 0);
  bool swept = false;
  if (!g.exact || !g.listed()) {
    if (g.exact) {
      const int shift0 = range_shift(g.r0.span, kDig), shift1 = range_shift(g.r1.span, kDig);
      team_sync<TEAM>();
      zero_buckets<TEAM, 2>(sh);
      __syncthreads();
#pragma unroll 1
      for (int r = 0; r < rounds; ++r) {
        uint32_t t[KPT];
        load_valid<KPT>(psi, mis, p.n_max, n, start + r * kRound + tid * KPT, t);
        add_again<KPT, TEAM>(sh, g, t, bits_of_thread(vis_w, r), shift0, shift1);
      }
      mass_walk<TEAM>(sh, rank, nullptr, p.theta_fix, g, shift0, shift1);
    }
    if (!g.exact || g.crowded0() || g.crowded1()) {
      mass_bisect<TEAM>(sh, rank, p.theta_fix, g, [&](auto each) {
#pragma unroll 1
        for (int r = 0; r < rounds; ++r) {
          uint32_t t[KPT];
          load_valid<KPT>(psi, mis, p.n_max, n, start + r * kRound + tid * KPT, t);
          const uint32_t vis = bits_of_thread(vis_w, r);
#pragma unroll
          for (int j = 0; j < KPT; ++j) each(t[j], (vis >> j) & 1u);
        }
      });
      swept = true;
    }
  }
  const bool on0 = g.r0.in <= kCap, on1 = g.r1.in <= kCap;
#pragma unroll 1
  for (int r = 0; r < rounds; ++r) {
    const int at = r * kRound + tid * KPT;
    uint32_t t[KPT];
    load_valid<KPT>(psi, mis, p.n_max, n, start + at, t);
    const uint32_t vis = bits_of_thread(vis_w, r);
    uint32_t in = 0;
#pragma unroll
    for (int j = 0; j < KPT; ++j) {
      const bool v = (vis >> j) & 1u;
      if (t[j] - (v ? g.r0.lo : g.r1.lo) <= (v ? g.r0.span : g.r1.span)) in |= 1u << j;
    }
    append_positions<TEAM, 2>(sh, pos0, pos1, on0 ? in & vis : 0u, on1 ? in & ~vis : 0u, at);
  }
  __syncthreads();
  const uint32_t listed = sh.list_n;
  if (swept) find_places<TEAM, 2>(sh, rank, tid == 0 ? listed & 0xffffu : 0u, tid == 0 ? listed >> 16 : 0u);
  const int m = tid / kHalf, mine_n = m ? listed >> 16 : listed & 0xffffu;
  for (int i = tid % kHalf; i < mine_n; i += kHalf)
    put<TEAM, 2, false>(sh, m, sh.found[m].seg[rank] + i, score_t(__ldg(psi + start + (m ? pos1 : pos0)[i])) - (m ? g.r1.lo : g.r0.lo));
  mass_finish<TEAM>(sh, p, rank, u, b, n, ph, g);
}

// The same as a kernel of its own, one block per sequence: for the budgets of one layer whose masses and demands are given
// (madakv_demand_layer), and after alloc_unit_kernel in calls of many units. `after_units`: the kernel before this one is that
// one, which has waited for all kernels before it, so the tokens can be counted before the wait for its results.
__global__ void __launch_bounds__(1024) alloc_seq_kernel(const __grid_constant__ AllocParams p, int after_units) {
  __shared__ int s_nv;
  __shared__ __align__(16) double s_phi[kBudgetBytes / 8];
  if (!after_units) pdl_wait();
  const int b = blockIdx.x;
  const int n = clamped_len(p.seq_len, b, p.n_max);
  const double ph = first_phi(p, b);
  if (threadIdx.x == 0) s_nv = 0;
  __syncthreads();
  count_visual(p.mask + (int64_t)b * p.n_max, n, &s_nv);
  __syncthreads();
  if (after_units) pdl_wait();
  pdl_go();
  sequence_budgets(p, b, n, s_nv, ph, s_phi);
}

template <int TEAM>
void launch_alloc_long(const AllocParams& p, int units, cudaStream_t st) {
  auto kern = alloc_long_kernel<TEAM>;
  // (the largest of any call, so that threads with calls of different sizes do not take the room from one another; a failure
  // shows at the launch)
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (2 * kListCap + long_words(kLongKeys, 1)) * 4);
  launch_team(kern, units, TEAM, (size_t)(2 * kListCap + long_words(p.n_max, TEAM)) * 4, st, p);
}
void launch_alloc_units(const madakv_config& c, const AllocParams& p, int units, cudaStream_t st) {
  const RankShape s = rank_shape(units, c.max_seq_len);
  switch (s.kpt * 16 + s.team) {
    case 8 * 16 + 1: launch_team(alloc_unit_kernel<8, 1>, units, 1, 0, st, p); break;
    case 8 * 16 + 2: launch_team(alloc_unit_kernel<8, 2>, units, 2, 0, st, p); break;
    case 8 * 16 + 4: launch_team(alloc_unit_kernel<8, 4>, units, 4, 0, st, p); break;
    case 8 * 16 + 8: launch_team(alloc_unit_kernel<8, 8>, units, 8, 0, st, p); break;
    case 16 * 16 + 1: launch_team(alloc_unit_kernel<16, 1>, units, 1, 0, st, p); break;
    case 16 * 16 + 2: launch_team(alloc_unit_kernel<16, 2>, units, 2, 0, st, p); break;
    case 16 * 16 + 4: launch_team(alloc_unit_kernel<16, 4>, units, 4, 0, st, p); break;
    case 16 * 16 + 8: launch_team(alloc_unit_kernel<16, 8>, units, 8, 0, st, p); break;
    case 1: launch_alloc_long<1>(p, units, st); break;
    case 2: launch_alloc_long<2>(p, units, st); break;
    case 4: launch_alloc_long<4>(p, units, st); break;
    default: launch_alloc_long<8>(p, units, st); break;
  }
}

// Masses, demands and, with p.budgets, what follows from them. In a call of fewer units than SMs the last unit of a
// sequence goes on with it (a kernel for that cost 2 us on the host and 4-6 on the GPU); in a larger one the fences and
// counters of all units cost more than the kernel (256 units of 131072 keys: 606 us with them for the three steps after scoring,
// 597 without).
void launch_alloc(const madakv_config& c, AllocParams p, void* ws, cudaStream_t st) {
  const int units = c.batch * p.L * p.Hkv;
  p.counter = p.budgets && units < 148 ? reinterpret_cast<unsigned*>((char*)ws + kHeaderBytes) : nullptr;
  launch_alloc_units(c, p, units, st);
  if (p.budgets && !p.counter) launch_pdl(alloc_seq_kernel, dim3(c.batch), dim3(1024), 0, st, p, 1);
}

AllocParams alloc_params(const madakv_config& c, int layers, const float* psi, const uint8_t* mask, const int32_t* seq_len,
                         double* mass, double* pref, int32_t* demand) {
  AllocParams p = {};
  p.psi = psi;
  p.mask = mask;
  p.seq_len = seq_len;
  p.mass = mass;
  p.pref = pref;
  p.demand = demand;
  p.L = layers;
  p.Hkv = c.n_kv_heads;
  p.n_max = c.max_seq_len;
  p.mpa = c.mpa;
  p.hcc_mode = c.hcc_mode;
  p.keep_window = c.keep_window;
  p.window = c.window;
  p.rows = c.n_q_heads / c.n_kv_heads * c.window;
  p.theta_fix = (u64)((double)c.theta * 4294967296.0);
  p.depth = c.n_layers;
  p.layer = -1;
  return p;
}

}  // namespace

int launch_allocate(const madakv_config& c, const float* psi, const uint8_t* mask, const int32_t* seq_len,
                    const int32_t* budget, double* mass, double* pref, int32_t* demand, double* phi, int32_t* budgets,
                    void* ws, cudaStream_t st) {
  AllocParams p = alloc_params(c, c.n_layers, psi, mask, seq_len, mass, pref, demand);
  p.budget = budget;
  p.phi = phi;
  p.budgets = budgets;
  launch_alloc(c, p, ws, st);
  return launch_status();
}

int launch_allocate_layer(const madakv_config& c, int layer, const float* psi, const uint8_t* mask,
                          const int32_t* seq_len, const int32_t* budget, double* mass, double* pref, int32_t* demand,
                          double* phi, int32_t* budgets, void* ws, cudaStream_t st) {
  AllocParams p = alloc_params(c, 1, psi, mask, seq_len, mass, pref, demand);  // the per-layer arrays hold one layer
  p.budget = budget;
  p.phi = phi;
  p.budgets = budgets;
  p.layer = layer;
  if (psi) launch_alloc(c, p, ws, st);
  else launch_pdl(alloc_seq_kernel, dim3(c.batch), dim3(1024), 0, st, p, 0);  // masses and demands come from launch_demand_layer
  return launch_status();
}

int launch_demand_layer(const madakv_config& c, const float* psi, const uint8_t* mask, const int32_t* seq_len,
                        double* mass, double* pref, int32_t* demand, void* ws, cudaStream_t st) {
  launch_alloc(c, alloc_params(c, 1, psi, mask, seq_len, mass, pref, demand), ws, st);
  return launch_status();
}

}  // namespace madakv
