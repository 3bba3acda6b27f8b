// Stage 4a: per-head, per-modality top-budget selection (Section 3.3, the eviction step after Eq. 8).
//
//   seg_scan     (large calls only) one block: visual-token count of every sequence, kept_len[u] = b_v + b_t and the exclusive
//                scan seg_off (rows, with headroom)
//   select_unit  a team of blocks per unit (rank_common.cuh) finds, for both modalities at once, the budget-th largest
//                value and how many of its ties are still needed; an ordered sweep then emits the kept positions in
//                ascending order, giving ties to the lowest positions (prefix sums over the team provide the tie ranks
//                and the output slots). It runs beside seg_scan and waits for the segment offsets only before it emits.
// Two options outside the paper: with pooling the ranking key of a position is the maximum of the keys of the
// positions around it (a maximum of fp32 values is exact, so nothing changes for the integer results); with
// forced retention the proxy tokens are emitted by the sweep without taking part in the ranking, and the wanted
// counts shrink by their number.
// Integer work only: results are bit-exact functions of (psi bits, mask, budgets).
#include "rank_common.cuh"

namespace madakv {
namespace {

struct SelParams {
  const float* psi;
  const uint8_t* mask;
  const int32_t* seq_len;
  const int32_t* budgets;
  int32_t* kept_len;
  int64_t* seg_off;
  int32_t* kept_idx;
  int64_t capacity;
  void* ws;
  int32_t* seq_nv;  // ws: visual-token count of every sequence
  int32_t* seq_wv;  // ws: visual tokens among the proxy tokens of every sequence (forced retention)
  int units, B, L, Hkv, n_max, mpa, headroom, keep_window, window, pool_r;  // pool_r: (pool_kernel - 1) / 2
  int rows;   // window rows per KV head
  int words;  // of bits, per kind of bit and block (long kernels)
  int alone;  // no seg_scan before: every unit adds up the segments before its own
};

// Segment of a unit with these budgets: its visual and text tokens, those of them that are kept anyway.
__device__ __forceinline__ int segment_length(const SelParams& p, int2 bud, int n, int n_v, int lo_v, int lo_t) {
  return (p.mpa ? min(max(bud.x, lo_v), n_v) : 0) + min(max(bud.y, lo_t), n - n_v);
}

// A warp's part (of `parts`) of the visual tokens among the first n of a sequence (c), and of those from wfrom on (cw); sums of
// the warp.
__device__ __forceinline__ void count_tokens(const uint8_t* mask, int n, int wfrom, int part, int parts, int& c, int& cw) {
  const int lane = threadIdx.x & 31;
  c = cw = 0;
  // whole 16-byte pieces of the row by vector loads, its ends by bytes
  const int lead = min(n, (int)((16 - (reinterpret_cast<uintptr_t>(mask) & 15)) & 15));
  const int n16 = (n - lead) >> 4;
  for (int i = part * 32 + lane; i < n16; i += parts * 32) {
    const uint4 v = __ldg(reinterpret_cast<const uint4*>(mask + lead) + i);
    c += __popc(nonzero_bytes(v.x) | (nonzero_bytes(v.y) << 4) | (nonzero_bytes(v.z) << 8) | (nonzero_bytes(v.w) << 12));
  }
  if (part == 0) {
    if (lane < lead) c += mask[lane] ? 1 : 0;
    const int i = lead + (n16 << 4) + lane;
    if (i < n) c += mask[i] ? 1 : 0;
  }
  for (int i = wfrom + part * 32 + lane; i < n; i += parts * 32) cw += mask[i] ? 1 : 0;  // (no proxy tokens: wfrom = n)
  c = __reduce_add_sync(kFull, c);
  cw = __reduce_add_sync(kFull, cw);
}

// One block. The visual tokens are counted by warps that share the sequences (several warps per sequence when there are
// fewer sequences than warps), then the segments are scanned, 1024 units at a time.
__global__ void __launch_bounds__(1024) seg_scan_kernel(SelParams p) {
  __shared__ long long warp_tot[32];
  __shared__ long long carry;
  __shared__ int s_cnt[32], s_wcnt[32];
  pdl_wait();
  pdl_go();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // visual tokens among the first seq_len[b] positions of every sequence
  const int share = p.B >= 32 ? 1 : 32 / p.B;  // warps per sequence
  for (int b0 = 0; b0 < p.B; b0 += 32 / share) {
    if (warp == 0) s_cnt[lane] = s_wcnt[lane] = 0;
    __syncthreads();
    const int slot = warp / share, b = b0 + slot, part = warp % share;
    if (slot < 32 / share && b < p.B) {
      const int n = clamped_len(p.seq_len, b, p.n_max);
      const uint8_t* mask = p.mask + (int64_t)b * p.n_max;
      const int wfrom = p.keep_window ? max(n - p.window, 0) : n;  // first proxy token retained unconditionally
      int c = 0, cw = 0;                                           // visual tokens, visual proxy tokens
      if (p.mpa) count_tokens(mask, n, wfrom, part, share, c, cw);
      if (lane == 0 && c) atomicAdd(&s_cnt[slot], c);
      if (lane == 0 && cw) atomicAdd(&s_wcnt[slot], cw);
    }
    __syncthreads();
    if (warp == 0 && lane < 32 / share && b0 + lane < p.B) {
      p.seq_nv[b0 + lane] = s_cnt[lane];
      p.seq_wv[b0 + lane] = s_wcnt[lane];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();  // also orders the seq_nv stores before the loads below (same block)
  for (int base = 0; base < p.units; base += 1024) {
    const int u = base + threadIdx.x;
    long long v = 0;
    if (u < p.units) {
      const int b = u / (p.Hkv * p.L);
      const int n = clamped_len(p.seq_len, b, p.n_max);
      const int n_v = p.seq_nv[b];
      const int lo_v = p.seq_wv[b], lo_t = (p.keep_window ? min(p.window, n) : 0) - lo_v;  // proxy tokens kept anyway
      const int len = segment_length(p, make_int2(p.budgets[2 * u], p.budgets[2 * u + 1]), n, n_v, lo_v, lo_t);
      p.kept_len[u] = len;
      v = (long long)len + p.headroom;
    }
    long long incl = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const long long t = __shfl_up_sync(kFull, incl, off);
      if ((threadIdx.x & 31) >= off) incl += t;
    }
    if ((threadIdx.x & 31) == 31) warp_tot[threadIdx.x >> 5] = incl;
    __syncthreads();
    long long wbase = 0;
    for (int i = 0; i < (int)(threadIdx.x >> 5); ++i) wbase += warp_tot[i];
    const long long excl = carry + wbase + incl - v;
    if (u < p.units) p.seg_off[u] = excl;
    __syncthreads();
    if (threadIdx.x == 1023) carry = excl + v;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    p.seg_off[p.units] = carry;
    if (carry > p.capacity) set_status(p.ws, MADAKV_ECAPACITY);
  }
}

// Keys of the two options: the maximum over the 2 * pool_r + 1 positions around each of KPT consecutive ones (pool_r may
// be 0; positions outside the sequence do not count). The largest score is the smallest t.
constexpr int kMaxPoolR = 7;  // pool_kernel <= 15
template <int KPT>
__device__ __forceinline__ void load_pooled(const float* row, int mis, int n, int pos0, int pool_r, uint32_t (&t)[KPT]) {
  uint32_t e[KPT + 16];  // t of positions pos0 - 8 .. pos0 + KPT + 7
  if (mis == 0 && pos0 >= 8 && pos0 + KPT + 8 <= n) {
#pragma unroll
    for (int x = 0; x < KPT + 16; x += 4) {
      const float4 v = __ldg(reinterpret_cast<const float4*>(row + pos0 - 8 + x));
      e[x] = score_t(v.x);
      e[x + 1] = score_t(v.y);
      e[x + 2] = score_t(v.z);
      e[x + 3] = score_t(v.w);
    }
  } else {
#pragma unroll
    for (int x = 0; x < KPT + 16; ++x) {
      const int pos = pos0 - 8 + x;
      e[x] = (pos >= 0 && pos < n) ? score_t(__ldg(row + pos)) : kTopKey;
    }
  }
#pragma unroll
  for (int j = 0; j < KPT; ++j) {
    uint32_t m = e[j + 8];
#pragma unroll
    for (int d = 1; d <= kMaxPoolR; ++d)
      if (d <= pool_r) m = min(m, min(e[j + 8 - d], e[j + 8 + d]));
    t[j] = m;
  }
}

// What a call without seg_scan knows of the sequences before a block's own: their visual tokens, all and among the proxy tokens.
constexpr int kAloneSeqs = 64, kAloneTokens = 65536;
struct SeqCounts {
  int nv[kAloneSeqs], wv[kAloneSeqs];
};

// A unit of a block, and what is wanted of it.
template <bool kPool>
struct SelUnit {
  const float* psi;
  const uint8_t* mask;
  int u, b, mis, n, wfrom, lo_v, lo_t;
  uint32_t want0, want1;
  int2 bud;         // the unit's budgets
  int2 before_bud;  // p.alone: budgets of unit threadIdx.x, if that comes before this one, its sequence and that one's length
  int before_b, before_n;
  __device__ __forceinline__ SelUnit(const SelParams& p, int unit) {
    u = unit;
    b = u / (p.Hkv * p.L);
    psi = p.psi + (int64_t)u * p.n_max;
    mis = (int)(((int64_t)u * p.n_max) & 3);
    mask = p.mask + (int64_t)b * p.n_max;
  }
  __device__ __forceinline__ void set_up(const SelParams& p) {
    if (p.alone && (int)threadIdx.x < u) {
      before_b = threadIdx.x / (p.Hkv * p.L);
      before_bud = __ldg(reinterpret_cast<const int2*>(p.budgets) + threadIdx.x);
      before_n = clamped_len(p.seq_len, before_b, p.n_max);
    }
    n = clamped_len(p.seq_len, b, p.n_max);
    // proxy tokens retained unconditionally (none without cfg->keep_window): they are emitted by the sweep and the
    // ranking only has to find the rest of each modality's budget
    wfrom = kPool && p.keep_window ? max(n - p.window, 0) : n;
    if (kPool) pdl_wait();  // (the forced tokens' counts are seg_scan's)
    lo_v = 0;
    if (kPool && !p.alone) lo_v = p.seq_wv[b];
    if (kPool && p.alone && p.mpa)  // (a window has at most 1024 tokens)
      for (int x = wfrom; x < n; x += kRankThreads)
        lo_v += __syncthreads_count(x + (int)threadIdx.x < n && mask[x + threadIdx.x] != 0);
    lo_t = (n - wfrom) - lo_v;
    bud = __ldg(reinterpret_cast<const int2*>(p.budgets) + u);
    want0 = (uint32_t)(p.mpa ? max(bud.x - lo_v, 0) : 0);
    want1 = (uint32_t)max(bud.y - lo_t, 0);
  }
  // p.alone: the tokens of the sequences before this one (behind a barrier after the counts were cleared)
  __device__ __forceinline__ void count_before(const SelParams& p, SeqCounts& s) const {
    if (!p.mpa) return;
    const int warp = threadIdx.x >> 5, parts = max(1, kRankWarps / b);
    for (int x = warp; x < b * parts; x += kRankWarps) {
      const int b2 = x / parts, n2 = clamped_len(p.seq_len, b2, p.n_max);
      int c, cw;
      count_tokens(p.mask + (int64_t)b2 * p.n_max, n2, p.keep_window ? max(n2 - p.window, 0) : n2, x % parts, parts, c, cw);
      if ((threadIdx.x & 31) == 0) {
        atomicAdd(&s.nv[b2], c);
        atomicAdd(&s.wv[b2], cw);
      }
    }
  }
  // t of KPT consecutive positions; returns those that are ranked, `forced`: those that are kept without
  template <int KPT>
  __device__ __forceinline__ uint32_t load(const SelParams& p, int pos0, uint32_t (&t)[KPT], uint32_t& forced) const {
    RawScores<KPT> raw;
    if (!kPool) issue_scores<KPT>(psi, mis, p.n_max, pos0, raw);
    return take(p, raw, pos0, t, forced);
  }
  template <int KPT>  // (raw: not used with pooling, which does not know its neighbours' bounds before the length)
  __device__ __forceinline__ uint32_t take(const SelParams& p, const RawScores<KPT>& raw, int pos0, uint32_t (&t)[KPT], uint32_t& forced) const {
    if (kPool) load_pooled<KPT>(psi, mis, n, pos0, p.pool_r, t);
    else take_scores<KPT>(raw, mis, t);
    uint32_t valid = valid_bits<KPT>(n, pos0);
    forced = 0;
    if (kPool) {
      forced = valid & ~valid_bits<KPT>(wfrom, pos0);
      valid &= ~forced;
    }
    if (valid != valid_bits<KPT>(KPT, 0)) {
#pragma unroll
      for (int j = 0; j < KPT; ++j)
        if (!((valid >> j) & 1u)) t[j] = kNoKey;
    }
    return valid;
  }
  __device__ __forceinline__ uint32_t load_one(const SelParams& p, int pos) const {  // the same of one ranked position
    if (!kPool) return score_t(__ldg(psi + pos));
    uint32_t m = kTopKey;
    for (int x = max(pos - p.pool_r, 0); x <= min(pos + p.pool_r, n - 1); ++x) m = min(m, score_t(__ldg(psi + x)));
    return m;
  }
};

// The ranges the two thresholds can lie in. short: the modality has no more keys than are wanted, all of them are kept.
template <int CAP>  // candidates that fit the list
struct SelRanges {
  RankRange r0, r1;
  bool short0, short1;
  uint32_t n_vis;   // visual tokens in the ranking
  uint32_t before;  // keys before their ranges in the blocks before this one
  __device__ __forceinline__ bool crowded0() const { return r0.in > CAP && r0.span > 0; }
  __device__ __forceinline__ bool crowded1() const { return r1.in > CAP && r1.span > 0; }
};

// Blocks on their own, whose calls are bound by instructions per key, take the plain layout of the buckets: of the finer one they
// have fewer candidates but no shorter steps (1024 units of 8192 keys 33.0 us with it, 31.4 without; 896 of 16384, 224
// rows, 47.1 and 44.9, and 50.4 and 47.5 with nine tenths of the mass in one key; 256 of 131072, 256 rows, 82.3 and 84.7,
// 88.2 and 83.5). Teams, whose steps grow with the candidates, take the finer one.
template <int TEAM>
struct SelectMap {
  using Map = BucketMap;
  static __device__ __forceinline__ Map of(int rows, int n) { return bucket_map(rows, n); }
};
template <>
struct SelectMap<1> {
  using Map = PlainMap;
  static __device__ __forceinline__ Map of(int, int) { return {}; }
};
template <int KPT, int TEAM, typename Map>
__device__ __forceinline__ void count_first(RankShared<TEAM, 1>& sh, const Map& map, const uint32_t (&t)[KPT], uint32_t vis, uint32_t valid) {
  constexpr int kStride = RankShared<TEAM, 1>::kStride;
  if (valid == valid_bits<KPT>(KPT, 0)) {
#pragma unroll
    for (int j = 0; j < KPT; ++j) atomicAdd(sh.cnt + ((vis >> j) & 1u ? 0 : kStride) + map_bucket(map, t[j]), 1u);
  } else {
#pragma unroll
    for (int j = 0; j < KPT; ++j)
      if ((valid >> j) & 1u) atomicAdd(sh.cnt + ((vis >> j) & 1u ? 0 : kStride) + map_bucket(map, t[j]), 1u);
  }
}
template <int KPT, int TEAM>
__device__ __forceinline__ void count_again(RankShared<TEAM, 1>& sh, const SelRanges<RankShared<TEAM, 1>::kCap>& g, const uint32_t (&t)[KPT], uint32_t vis, int shift0, int shift1) {
#pragma unroll
  for (int j = 0; j < KPT; ++j) {
    const bool v = (vis >> j) & 1u;
    const uint32_t x = t[j] - (v ? g.r0.lo : g.r1.lo);
    if (x <= (v ? g.r0.span : g.r1.span)) atomicAdd(sh.cnt + (v ? 0 : RankShared<TEAM, 1>::kStride) + (x >> (v ? shift0 : shift1)), 1u);
  }
}

// Walk of the buckets (of the first layout, `map`, or of one over the ranges): the ranges shrink to the buckets with the wanted
// keys.
template <int TEAM, typename Map>
__device__ __forceinline__ void select_walk(RankShared<TEAM, 1>& sh, uint32_t rank, const Map* map, uint32_t want0, uint32_t want1,
                                            SelRanges<RankShared<TEAM, 1>::kCap>& g, int shift0, int shift1) {
  walk<TEAM, 1>(
      sh, rank, [](int, int) { return BucketStart{0u, 0, false}; },
      [&](int m, u64) -> u64 { return m ? (g.short1 || !want1 ? 0u : want1 - g.r1.above) : (g.short0 || !want0 ? 0u : want0 - g.r0.above); });
  if (map) g.n_vis = sh.found[0].total;
  auto narrow = [&](RankRange& r, bool& is_short, const Found& f, int shift) {
    if (TEAM > 1) g.before += f.before;
    if (!f.hit) {  // the modality has no more keys than wanted
      is_short = true;
      r = RankRange{kNowhere, 0u, 0u, 0u};
      return;
    }
    bucket_range(r, map, f.at, shift);
    r.above += f.above;
    r.in = f.in;
  };
  if (want0 && !g.short0) narrow(g.r0, g.short0, sh.found[0], shift0);
  if (want1 && !g.short1) narrow(g.r1, g.short1, sh.found[1], shift1);
}

// (Rare) too many keys in a range: halve it with exact sweeps until they fit the list or are all alike. `sweep` calls its
// argument with the keys of the thread, some at a time.
template <int TEAM, typename Sweep>
__device__ __forceinline__ void select_bisect(RankShared<TEAM, 1>& sh, uint32_t want0, uint32_t want1,
                                              SelRanges<RankShared<TEAM, 1>::kCap>& g, Sweep sweep) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  while (g.crowded0() || g.crowded1()) {
    const bool on0 = g.crowded0(), on1 = g.crowded1();
    const uint32_t mid0 = g.r0.lo + (g.r0.span >> 1), mid1 = g.r1.lo + (g.r1.span >> 1);
    uint32_t c0 = 0, c1 = 0;
    sweep([&](uint32_t t, bool v) {
      if ((v ? on0 : on1) && t >= (v ? g.r0.lo : g.r1.lo) && t <= (v ? mid0 : mid1)) {
        if (v) ++c0; else ++c1;
      }
    });
    c0 = __reduce_add_sync(kFull, c0);
    c1 = __reduce_add_sync(kFull, c1);
    if (lane == 0) {
      sh.wcnt[0][warp] = c0;
      sh.wcnt[1][warp] = c1;
    }
    team_sync<TEAM>();
    c0 = c1 = 0;
#pragma unroll 1
    for (uint32_t r = 0; r < TEAM; ++r)
#pragma unroll 1
      for (int w = 0; w < kRankWarps; ++w) {
        c0 += peer_load<TEAM>(&sh.wcnt[0][w], r);
        c1 += peer_load<TEAM>(&sh.wcnt[1][w], r);
      }
    auto halve = [](RankRange& r, uint32_t want, uint32_t c) {
      const uint32_t half = r.span >> 1;
      if (r.above + c >= want) {
        r.span = half;
        r.in = c;
      } else {
        r.above += c;
        r.in -= c;
        r.lo += half + 1;
        r.span -= half + 1;
      }
    };
    if (on0) halve(g.r0, want0, c0);
    if (on1) halve(g.r1, want1, c1);
    team_sync<TEAM>();
  }
}

// With the candidates of all blocks in their lists: the smallest t up to which the wanted number of keys lies, and how many keys
// of exactly that t are still wanted, found by every block for itself. (Nothing wanted: nothing lies before 0 and no tie is
// kept; all wanted: everything lies before kNowhere.)
struct Thresholds {
  uint32_t thr0, thr1, ties0, ties1;
};
template <int TEAM>
__device__ __forceinline__ Thresholds select_thresholds(RankShared<TEAM, 1>& sh, uint32_t want0, uint32_t want1,
                                                        const SelRanges<RankShared<TEAM, 1>::kCap>& g) {
  constexpr uint32_t kCap = RankShared<TEAM, 1>::kCap;
  team_sync<TEAM>();  // (the last access to another block's shared memory, but for counts_before() after exact sweeps)
  const bool on0 = want0 && !g.short0 && g.r0.in <= kCap, on1 = want1 && !g.short1 && g.r1.in <= kCap;
  finish_lists<TEAM, 1, false>(sh, g.r0, g.r1, on0, on1, want0, want1, 0ull, 0ull);
  Thresholds h;
  h.thr0 = !want0 ? 0u : (g.short0 ? kNowhere : (on0 ? sh.fin_lo[0] : g.r0.lo));
  h.thr1 = !want1 ? 0u : (g.short1 ? kNowhere : (on1 ? sh.fin_lo[1] : g.r1.lo));
  h.ties0 = !want0 || g.short0 ? 0u : want0 - (on0 ? sh.fin_c[0] : g.r0.above);
  h.ties1 = !want1 || g.short1 ? 0u : want1 - (on1 ? sh.fin_c[1] : g.r1.above);
  return h;
}

// Counts of (ties v, ties t, kept outright) travel as one 3 x 21-bit word. What lies before this thread's positions, from its
// own counts.
__device__ __forceinline__ u64 emit_counts(uint32_t gt, uint32_t eq, uint32_t vis) {
  return (u64)__popc(eq & vis) | ((u64)__popc(eq & ~vis) << 21) | ((u64)__popc(gt) << 42);
}
// The blocks before this one: their keys before the ranges are known from the walk, those of them in the ranges from the list,
// where every block's keys have places of their own. After exact sweeps (`swept`) the blocks exchange their totals instead.
template <int TEAM>
__device__ __forceinline__ u64 counts_before(RankShared<TEAM, 1>& sh, uint32_t rank, u64 mine, const Thresholds& h, uint32_t want0, uint32_t want1,
                                             const SelRanges<RankShared<TEAM, 1>::kCap>& g, uint32_t forced_before, bool swept) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const u64 incl = warp_scan64(mine);
  if (lane == 31) sh.wscan_q[warp] = incl;
  u64 before = 0;
  if (TEAM > 1 && !swept) {
    const int m = threadIdx.x / kHalf;
    const RankRange r = m ? g.r1 : g.r0;
    const bool ranked = m ? want1 && !g.short1 : want0 && !g.short0;
    const uint32_t thr = m ? h.thr1 : h.thr0, mine_n = ranked ? sh.found[m].seg[rank] : 0u;
    uint32_t lt = 0, eq = 0;
    if (r.in <= RankShared<TEAM, 1>::kCap) {
      for (uint32_t x = threadIdx.x % kHalf; x < mine_n; x += kHalf) {
        const uint32_t v = r.lo + sh.list[m][x];
        lt += v < thr ? 1u : 0u;
        eq += v == thr ? 1u : 0u;
      }
    } else if (threadIdx.x % kHalf == 0) {  // all keys of the range are alike
      eq = mine_n;
    }
    lt = __reduce_add_sync(kFull, lt);
    eq = __reduce_add_sync(kFull, eq);
    if (lane == 0) sh.wsum[0][warp] = ((u64)eq << (m ? 21 : 0)) | ((u64)lt << 42);
  }
  __syncthreads();
  if (TEAM > 1 && !swept) {
    before = warp_sum64(lane < kRankWarps ? sh.wsum[0][lane] : 0ull) + ((u64)(g.before + forced_before) << 42);
  } else if (TEAM > 1) {
    if (warp == 0) {
      const u64 tot = warp_sum64(lane < kRankWarps ? sh.wscan_q[lane] : 0ull);
      if (lane < TEAM) peer_store<TEAM>(&sh.slice_q[0][rank], lane, tot);
    }
    team_sync<TEAM>();
    before = warp_sum64(lane < (int)rank ? sh.slice_q[0][lane] : 0ull);
  }
  return before + incl - mine + warp_sum64(lane < warp ? sh.wscan_q[lane] : 0ull);
}

// Where the unit's segment starts; -1: the cache is too small.
template <int TEAM, bool kPool>
__device__ __forceinline__ int64_t segment_start(RankShared<TEAM, 1>& sh, const SeqCounts& s, const SelParams& p, const SelUnit<kPool>& x,
                                                 uint32_t rank, uint32_t n_vis) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (p.alone) {
    // the segments' lengths follow from the budgets and the modalities' token counts, which are at hand
    const int n_v = (int)n_vis + x.lo_v;
    u64 sum = 0;
    if (tid < x.u) {
      const bool own = x.before_b == x.b;
      const int nv = own ? n_v : s.nv[x.before_b], lv = own ? x.lo_v : s.wv[x.before_b];
      const int lt = (kPool && p.keep_window ? min(p.window, x.before_n) : 0) - lv;
      sum = (u64)(segment_length(p, x.before_bud, x.before_n, nv, lv, lt) + p.headroom);
    }
    sum = warp_sum64(sum);
    __syncthreads();
    if (lane == 0) sh.wsum[1][warp] = sum;
    __syncthreads();
    const int64_t off = (int64_t)warp_sum64(lane < kRankWarps ? sh.wsum[1][lane] : 0ull);
    const int len = segment_length(p, x.bud, x.n, n_v, x.lo_v, x.lo_t);
    const int64_t end = off + len + p.headroom;
    if (rank == 0 && tid == 0) {
      p.kept_len[x.u] = len;
      p.seg_off[x.u] = off;
      if (x.u + 1 == p.units) {
        p.seg_off[p.units] = end;
        if (end > p.capacity) set_status(p.ws, MADAKV_ECAPACITY);
      }
    }
    return end > p.capacity ? -1 : off;
  }
  if (!kPool) pdl_wait();
  pdl_go();
  const int64_t off = p.seg_off[x.u];
  return off + p.kept_len[x.u] + p.headroom > p.capacity ? -1 : off;  // (seg_scan has raised MADAKV_ECAPACITY)
}

// Up to 32 consecutive positions: a key before its modality's threshold (gt) is kept, one at the threshold (eq) while its rank
// among these ties, in position order, is below the number still wanted. `ahead`: counts before these positions.
__device__ __forceinline__ void emit(int32_t* seg, const Thresholds& h, int pos0, u64 ahead, uint32_t gt, uint32_t eq, uint32_t vis) {
  const uint32_t e0 = (uint32_t)ahead & 0x1fffffu, e1 = (uint32_t)(ahead >> 21) & 0x1fffffu, g = (uint32_t)(ahead >> 42);
  int32_t* out = seg + g + min(e0, h.ties0) + min(e1, h.ties1);
  uint32_t keep = gt;
  uint32_t ev = eq & vis, et = eq & ~vis;
  for (uint32_t k = e0; k < h.ties0 && ev; ++k) {  // lowest positions first
    keep |= ev & (0u - ev);
    ev &= ev - 1;
  }
  for (uint32_t k = e1; k < h.ties1 && et; ++k) {
    keep |= et & (0u - et);
    et &= et - 1;
  }
  while (keep) {
    const int j = __ffs(keep) - 1;
    keep &= keep - 1;
    *out++ = pos0 + j;
  }
}

// A unit whose keys fit the registers of its team.
template <int KPT, int TEAM, bool kPool>
__global__ void __launch_bounds__(kRankThreads, 2) select_unit_kernel(const __grid_constant__ SelParams p) {
  using Map = typename SelectMap<TEAM>::Map;
  constexpr uint32_t kCap = RankShared<TEAM, 1>::kCap;
  __shared__ RankShared<TEAM, 1> sh;
  __shared__ SeqCounts s;
  team_started<TEAM>();
  if (TEAM > 1) zero_buckets<TEAM, 1>(sh);
  if (threadIdx.x < kAloneSeqs) s.nv[threadIdx.x] = s.wv[threadIdx.x] = 0;
  // (no wait here after seg_scan: it has waited for everything before it, so the scores, the mask and the budgets are final;
  // what seg_scan itself writes is read after the wait of segment_start)
  if (p.alone) {
    pdl_wait();
    pdl_go();
  }
  const uint32_t rank = TEAM > 1 ? team_rank() : 0u;
  SelUnit<kPool> x(p, blockIdx.x / TEAM);
  const int pos0 = (int)rank * kRankThreads * KPT + threadIdx.x * KPT;  // a block owns consecutive positions
  RawScores<KPT> raw;
  RawMask<KPT> raw_mask;
  if (!kPool) issue_scores<KPT>(x.psi, x.mis, p.n_max, pos0, raw);
  if (p.mpa) issue_mask<KPT>(x.mask, p.n_max, pos0, raw_mask);
  if (TEAM == 1) zero_buckets<TEAM, 1>(sh);
  x.set_up(p);
  uint32_t t[KPT], forced;
  const uint32_t valid = x.template take<KPT>(p, raw, pos0, t, forced), vis = p.mpa ? take_mask<KPT>(raw_mask) : 0u;
  const Map map = SelectMap<TEAM>::of(p.rows, x.n);
  __syncthreads();
  if (p.alone && x.b > 0) x.count_before(p, s);
  count_first<KPT, TEAM>(sh, map, t, vis, valid);
  SelRanges<kCap> g{{kNowhere, 0u, 0u, 0u}, {kNowhere, 0u, 0u, 0u}, false, false, 0u, 0u};
  team_wait_started<TEAM>();
  select_walk<TEAM, Map>(sh, rank, &map, x.want0, x.want1, g, 0, 0);
  bool swept = false;
  if (g.crowded0() || g.crowded1()) {
    const int shift0 = range_shift(g.r0.span, kDig), shift1 = range_shift(g.r1.span, kDig);
    team_sync<TEAM>();
    zero_buckets<TEAM, 1>(sh);
    __syncthreads();
    count_again<KPT, TEAM>(sh, g, t, vis, shift0, shift1);
    select_walk<TEAM, Map>(sh, rank, nullptr, x.want0, x.want1, g, shift0, shift1);
    if (g.crowded0() || g.crowded1()) {
      select_bisect<TEAM>(sh, x.want0, x.want1, g, [&](auto each) {
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
  if (swept) find_places<TEAM, 1>(sh, rank, __popc(in0), __popc(in1));
  append<TEAM, 1, KPT, true>(sh, rank, in0, in1, t, g.r0.lo, g.r1.lo);
  const Thresholds h = select_thresholds<TEAM>(sh, x.want0, x.want1, g);
  uint32_t eq = 0, gt = 0;
#pragma unroll
  for (int j = 0; j < KPT; ++j) {
    const uint32_t thr = (vis >> j) & 1u ? h.thr0 : h.thr1;
    if (t[j] == thr) eq |= 1u << j;
    if (t[j] < thr) gt |= 1u << j;
  }
  if (kPool) gt |= forced;
  const uint32_t forced_before = kPool ? (uint32_t)max(min((int)rank * kRankThreads * KPT, x.n) - x.wfrom, 0) : 0u;
  const u64 ahead = counts_before<TEAM>(sh, rank, emit_counts(gt, eq, vis), h, x.want0, x.want1, g, forced_before, swept);
  const int64_t off = segment_start<TEAM, kPool>(sh, s, p, x, rank, g.n_vis);
  if (off >= 0) emit(p.kept_idx + off, h, pos0, ahead, gt, eq, vis);
}

// A longer unit is read twice: once for the buckets, once to sort its keys into kept, dropped and candidates. The first two are
// three bits per key (visual, kept, candidate) in shared memory; candidates go to the list as positions, and when the
// thresholds are known their bits are put right, so that the positions are emitted from the bits. (With every sweep over the
// keys themselves, range, buckets, candidates and emission, 256 units of 131072 keys took 187 us instead of 110.)
template <int TEAM, bool kPool>
__global__ void __launch_bounds__(kRankThreads, 2) select_long_kernel(const __grid_constant__ SelParams p) {
  constexpr int KPT = 16, kRound = kRankThreads * KPT;
  using Map = typename SelectMap<TEAM>::Map;
  constexpr uint32_t kCap = RankShared<TEAM, 1>::kCap;
  __shared__ RankShared<TEAM, 1> sh;
  __shared__ SeqCounts s;
  extern __shared__ __align__(16) uint32_t bits[];
  team_started<TEAM>();
  zero_buckets<TEAM, 1>(sh);
  if (threadIdx.x < kAloneSeqs) s.nv[threadIdx.x] = s.wv[threadIdx.x] = 0;
  if (p.alone) {
    pdl_wait();
    pdl_go();
  }
  const uint32_t rank = TEAM > 1 ? team_rank() : 0u;
  const int tid = threadIdx.x;
  SelUnit<kPool> x(p, blockIdx.x / TEAM);
  x.set_up(p);
  uint32_t* cand_pos[2] = {bits, bits + kListCap};
  uint32_t* vis_w = bits + 2 * kListCap;
  uint32_t* keep_w = vis_w + p.words;
  uint32_t* cand_w = keep_w + p.words;
  const int rounds = (x.n + kRound * TEAM - 1) / (kRound * TEAM);
  const int start = (int)rank * rounds * kRound;  // a block owns consecutive positions

  const Map map = SelectMap<TEAM>::of(p.rows, x.n);
  __syncthreads();
  if (p.alone && x.b > 0) x.count_before(p, s);
#pragma unroll 1
  for (int r = 0; r < rounds; ++r) {
    const int pos0 = start + r * kRound + tid * KPT;
    uint32_t t[KPT], forced;
    const uint32_t valid = x.template load<KPT>(p, pos0, t, forced);
    const uint32_t vis = p.mpa ? load_mask<KPT>(x.mask, p.n_max, pos0) : 0u;
    bits_of_thread(vis_w, r) = (uint16_t)vis;
    count_first<KPT, TEAM>(sh, map, t, vis, valid);
  }
  SelRanges<kCap> g{{kNowhere, 0u, 0u, 0u}, {kNowhere, 0u, 0u, 0u}, false, false, 0u, 0u};
  team_wait_started<TEAM>();
  select_walk<TEAM, Map>(sh, rank, &map, x.want0, x.want1, g, 0, 0);
  bool swept = false;
  if (g.crowded0() || g.crowded1()) {
    const int shift0 = range_shift(g.r0.span, kDig), shift1 = range_shift(g.r1.span, kDig);
    team_sync<TEAM>();
    zero_buckets<TEAM, 1>(sh);
    __syncthreads();
#pragma unroll 1
    for (int r = 0; r < rounds; ++r) {
      uint32_t t[KPT], forced;
      x.template load<KPT>(p, start + r * kRound + tid * KPT, t, forced);
      count_again<KPT, TEAM>(sh, g, t, bits_of_thread(vis_w, r), shift0, shift1);
    }
    select_walk<TEAM, Map>(sh, rank, nullptr, x.want0, x.want1, g, shift0, shift1);
    if (g.crowded0() || g.crowded1()) {
      select_bisect<TEAM>(sh, x.want0, x.want1, g, [&](auto each) {
#pragma unroll 1
        for (int r = 0; r < rounds; ++r) {
          uint32_t t[KPT], forced;
          x.template load<KPT>(p, start + r * kRound + tid * KPT, t, forced);
          const uint32_t vis = bits_of_thread(vis_w, r);
#pragma unroll
          for (int j = 0; j < KPT; ++j) each(t[j], (vis >> j) & 1u);
        }
      });
      swept = true;
    }
  }

  // ---- kept and candidates. Nothing wanted: nothing lies before 0; all wanted: everything lies before kNowhere.
  const uint32_t lo0 = x.want0 ? g.r0.lo : 0u, lo1 = x.want1 ? g.r1.lo : 0u;
  const uint32_t wide0 = x.want0 && !g.short0 ? g.r0.span + 1u : 0u, wide1 = x.want1 && !g.short1 ? g.r1.span + 1u : 0u;
  const bool on0 = g.r0.in <= kCap, on1 = g.r1.in <= kCap;
#pragma unroll 1
  for (int r = 0; r < rounds; ++r) {
    const int at = r * kRound + tid * KPT;
    uint32_t t[KPT], forced;
    x.template load<KPT>(p, start + at, t, forced);
    const uint32_t vis = bits_of_thread(vis_w, r);
    uint32_t in = 0, keep = forced;
#pragma unroll
    for (int j = 0; j < KPT; ++j) {
      const bool v = (vis >> j) & 1u;
      const uint32_t lo = v ? lo0 : lo1;
      if (t[j] < lo) keep |= 1u << j;
      if (t[j] - lo < (v ? wide0 : wide1)) in |= 1u << j;
    }
    bits_of_thread(keep_w, r) = (uint16_t)keep;
    bits_of_thread(cand_w, r) = (uint16_t)in;
    append_positions<TEAM, 1>(sh, cand_pos[0], cand_pos[1], on0 ? in & vis : 0u, on1 ? in & ~vis : 0u, at);
  }
  __syncthreads();
  const uint32_t listed = sh.list_n;
  if (swept) find_places<TEAM, 1>(sh, rank, tid == 0 ? listed & 0xffffu : 0u, tid == 0 ? listed >> 16 : 0u);
  const int m = tid / kHalf, mine_n = m ? listed >> 16 : listed & 0xffffu, place = mine_n ? sh.found[m].seg[rank] : 0;
  for (int i = tid % kHalf; i < mine_n; i += kHalf)
    put<TEAM, 1, true>(sh, m, place + i, x.load_one(p, start + (int)cand_pos[m][i]) - (m ? lo1 : lo0));
  const Thresholds h = select_thresholds<TEAM>(sh, x.want0, x.want1, g);
  // ---- of the candidates, those before the threshold are kept and those at it stay candidates (ties)
  for (int i = tid % kHalf; i < mine_n; i += kHalf) {
    const uint32_t t = sh.list[m][place + i] + (m ? lo1 : lo0), thr = m ? h.thr1 : h.thr0, at = cand_pos[m][i];
    if (t < thr) atomicOr(keep_w + bits_slot(at >> 5), 1u << (at & 31));
    if (t != thr) atomicAnd(cand_w + bits_slot(at >> 5), ~(1u << (at & 31)));
  }
  __syncthreads();
  const int words = rounds * (kRound / 32), share = (words + kRankThreads - 1) / kRankThreads;  // consecutive words per thread
  const int w0 = min(tid * share, words), w1 = min(w0 + share, words);
  u64 mine = 0;
  for (int w = w0; w < w1; ++w) mine += emit_counts(keep_w[bits_slot(w)], cand_w[bits_slot(w)], vis_w[bits_slot(w)]);
  const uint32_t forced_before = kPool ? (uint32_t)max(min(start, x.n) - x.wfrom, 0) : 0u;
  u64 ahead = counts_before<TEAM>(sh, rank, mine, h, x.want0, x.want1, g, forced_before, swept);
  const int64_t off = segment_start<TEAM, kPool>(sh, s, p, x, rank, g.n_vis);
  if (off < 0) return;
  for (int w = w0; w < w1; ++w) {
    const uint32_t gt = keep_w[bits_slot(w)], eq = cand_w[bits_slot(w)], vis = vis_w[bits_slot(w)];
    emit(p.kept_idx + off, h, start + w * 32, ahead, gt, eq, vis);
    ahead += emit_counts(gt, eq, vis);
  }
}

template <int TEAM, bool kPool>
void launch_long(SelParams p, cudaStream_t st) {
  auto kern = select_long_kernel<TEAM, kPool>;
  p.words = long_words(p.n_max, TEAM);
  // (the largest of any call, so that threads with calls of different sizes do not take the room from one another; a failure
  // shows at the launch)
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (2 * kListCap + 3 * long_words(kLongKeys, 1)) * 4);
  launch_team(kern, p.units, TEAM, (size_t)(2 * kListCap + 3 * p.words) * 4, st, p);
}
template <bool kPool>
void launch_select_unit(const madakv_config& c, const SelParams& p, cudaStream_t st) {
  const RankShape s = rank_shape(p.units, c.max_seq_len);
  switch (s.kpt * 16 + s.team) {
    case 8 * 16 + 1: launch_team(select_unit_kernel<8, 1, kPool>, p.units, 1, 0, st, p); break;
    case 8 * 16 + 2: launch_team(select_unit_kernel<8, 2, kPool>, p.units, 2, 0, st, p); break;
    case 8 * 16 + 4: launch_team(select_unit_kernel<8, 4, kPool>, p.units, 4, 0, st, p); break;
    case 8 * 16 + 8: launch_team(select_unit_kernel<8, 8, kPool>, p.units, 8, 0, st, p); break;
    case 16 * 16 + 1: launch_team(select_unit_kernel<16, 1, kPool>, p.units, 1, 0, st, p); break;
    case 16 * 16 + 2: launch_team(select_unit_kernel<16, 2, kPool>, p.units, 2, 0, st, p); break;
    case 16 * 16 + 4: launch_team(select_unit_kernel<16, 4, kPool>, p.units, 4, 0, st, p); break;
    case 16 * 16 + 8: launch_team(select_unit_kernel<16, 8, kPool>, p.units, 8, 0, st, p); break;
    case 1: launch_long<1, kPool>(p, st); break;
    case 2: launch_long<2, kPool>(p, st); break;
    case 4: launch_long<4, kPool>(p, st); break;
    default: launch_long<8, kPool>(p, st); break;
  }
}

}  // namespace

int launch_select(const madakv_config& c, const float* psi, const uint8_t* mask, const int32_t* seq_len,
                  const int32_t* budgets, int32_t* kept_len, int64_t* seg_off, int32_t* kept_idx, int64_t capacity,
                  void* ws, cudaStream_t st) {
  SelParams p;
  p.psi = psi;
  p.mask = mask;
  p.seq_len = seq_len;
  p.budgets = budgets;
  p.kept_len = kept_len;
  p.seg_off = seg_off;
  p.kept_idx = kept_idx;
  p.capacity = capacity;
  p.ws = ws;
  p.units = c.batch * c.n_layers * c.n_kv_heads;
  p.B = c.batch;
  p.L = c.n_layers;
  p.Hkv = c.n_kv_heads;
  p.n_max = c.max_seq_len;
  p.mpa = c.mpa;
  p.headroom = c.max_new_tokens;
  p.seq_nv = reinterpret_cast<int32_t*>((char*)ws + ws_layout(c).seq_nv_off);
  p.seq_wv = p.seq_nv + c.batch;
  p.keep_window = c.keep_window;
  p.window = c.window;
  p.pool_r = (c.pool_kernel - 1) / 2;
  p.rows = c.n_q_heads / c.n_kv_heads * c.window;
  // Few units: no kernel of its own for the scan of the segments (2 us on the host, 3-5 on the GPU). A unit needs the visual-token
  // counts of the sequences before its own, which it takes itself as long as they are a few loads per thread; a larger call is
  // better off with a scan that runs beside the ranking. Layer by layer, where the host is the bound, a step of allocation,
  // selection and compaction takes 28.4 us without the scan and 30.4 with it (8 x 4 units of 1000 or 4000 keys, 4 x 8 of 2000,
  // 64 x 2 of 500), about the same near the limit (8 x 4 of 8000, 36.0 and 35.7); selections one after the other, which the GPU is
  // the bound of, take 0.3-1.4 us more without it up to the limit (36 x 4 of 1024 7.6 and 7.0, 8 x 4 of 8192 8.8 and 7.5) and 2-9
  // beyond (8 x 4 of 16384 10.8 and 7.7, 64 x 2 of 8192 24.2 and 15.3).
  p.alone = p.units < 148 && c.batch <= kAloneSeqs && (c.batch == 1 || (int64_t)c.batch * c.max_seq_len <= kAloneTokens);
  if (!p.alone) launch_pdl(seg_scan_kernel, dim3(1), dim3(1024), 0, st, p);
  if (c.pool_kernel > 1 || c.keep_window) launch_select_unit<true>(c, p, st);
  else launch_select_unit<false>(c, p, st);
  return launch_status();
}

}  // namespace madakv
