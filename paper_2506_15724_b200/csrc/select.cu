// Stage 4a: per-head, per-modality top-budget selection (Section 3.3, the eviction step after Eq. 8).
//
//   seg_scan     (batches only) one block: visual-token count of every sequence, kept_len[u] = b_v + b_t and the exclusive
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
  int alone;  // no seg_scan before: every unit adds up the segments before its own
};

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
      if (p.mpa) {
        // whole 16-byte pieces of the row by vector loads, its ends by bytes
        const int lead = min(n, (int)((16 - (reinterpret_cast<uintptr_t>(mask) & 15)) & 15));
        const int n16 = (n - lead) >> 4;
        for (int i = part * 32 + lane; i < n16; i += share * 32) {
          const uint4 v = __ldg(reinterpret_cast<const uint4*>(mask + lead) + i);
          c += __popc(nonzero_bytes(v.x) | (nonzero_bytes(v.y) << 4) | (nonzero_bytes(v.z) << 8) | (nonzero_bytes(v.w) << 12));
        }
        if (part == 0) {
          if (lane < lead) c += mask[lane] ? 1 : 0;
          const int i = lead + (n16 << 4) + lane;
          if (i < n) c += mask[i] ? 1 : 0;
        }
        for (int i = wfrom + part * 32 + lane; i < n; i += share * 32) cw += mask[i] ? 1 : 0;  // (no proxy tokens: wfrom = n)
      }
      c = __reduce_add_sync(kFull, c);
      cw = __reduce_add_sync(kFull, cw);
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
      const int len = (p.mpa ? min(max(p.budgets[2 * u], lo_v), n_v) : 0) + min(max(p.budgets[2 * u + 1], lo_t), n - n_v);
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
// be 0; positions outside the sequence do not count).
constexpr int kMaxPoolR = 7;  // pool_kernel <= 15
template <int KPT>
__device__ __forceinline__ void load_pooled(const float* row, int mis, int n, int pos0, int pool_r, uint32_t (&key)[KPT]) {
  uint32_t e[KPT + 16];  // keys of positions pos0 - 8 .. pos0 + KPT + 7
  if (mis == 0 && pos0 >= 8 && pos0 + KPT + 8 <= n) {
#pragma unroll
    for (int x = 0; x < KPT + 16; x += 4) {
      const float4 v = __ldg(reinterpret_cast<const float4*>(row + pos0 - 8 + x));
      e[x] = score_key(v.x);
      e[x + 1] = score_key(v.y);
      e[x + 2] = score_key(v.z);
      e[x + 3] = score_key(v.w);
    }
  } else {
#pragma unroll
    for (int x = 0; x < KPT + 16; ++x) {
      const int pos = pos0 - 8 + x;
      e[x] = (pos >= 0 && pos < n) ? score_key(__ldg(row + pos)) : 0u;
    }
  }
#pragma unroll
  for (int j = 0; j < KPT; ++j) {
    uint32_t m = e[j + 8];
#pragma unroll
    for (int d = 1; d <= kMaxPoolR; ++d)
      if (d <= pool_r) m = max(m, max(e[j + 8 - d], e[j + 8 + d]));
    key[j] = m;
  }
}

template <int KPT, int TEAM, bool kPool>
__global__ void __launch_bounds__(kRankThreads, 2) select_unit_kernel(SelParams p) {
  using SH = RankShared<TEAM, 1>;
  constexpr int kPer = SH::kPer;
  __shared__ SH sh;
  // (no wait here after seg_scan: it has waited for everything before it, so the scores, the mask and the budgets are final;
  // what seg_scan itself writes is read after the wait below)
  if (p.alone) pdl_wait();
  const uint32_t rank = TEAM > 1 ? team_rank() : 0u;
  const int u = blockIdx.x / TEAM;
  const int b = u / (p.Hkv * p.L);
  const float* psi = p.psi + (int64_t)u * p.n_max;
  const int mis = (int)(((int64_t)u * p.n_max) & 3);
  const uint8_t* mask = p.mask + (int64_t)b * p.n_max;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int kRound = kRankThreads * KPT;
  const int rounds = (p.n_max + kRound * TEAM - 1) / (kRound * TEAM);
  const int pos_first = (int)rank * rounds * kRound + tid * KPT;  // a block owns consecutive positions
  const int n = clamped_len(p.seq_len, b, p.n_max);
  // proxy tokens retained unconditionally (none without cfg->keep_window): they are emitted by the sweep and the
  // ranking only has to find the rest of each modality's budget
  const int wfrom = kPool && p.keep_window ? max(n - p.window, 0) : n;
  if (kPool) pdl_wait();  // (the forced tokens' counts are seg_scan's)
  int lo_v = 0;
  if (kPool && !p.alone) lo_v = p.seq_wv[b];
  if (kPool && p.alone && p.mpa)  // (a window has at most 1024 tokens)
    for (int x = wfrom; x < n; x += kRankThreads) lo_v += __syncthreads_count(x + tid < n && mask[x + tid] != 0);
  const int lo_t = (n - wfrom) - lo_v;
  const uint32_t want0 = (uint32_t)(p.mpa ? max(p.budgets[2 * u] - lo_v, 0) : 0),
                 want1 = (uint32_t)max(p.budgets[2 * u + 1] - lo_t, 0);

  uint32_t key[KPT], vis = 0, forced = 0;
  auto load_round = [&](int r) {
    const int pos0 = pos_first + r * kRound;
    if (kPool) load_pooled<KPT>(psi, mis, n, pos0, p.pool_r, key);
    else load_scores<KPT>(psi, mis, p.n_max, pos0, key);
    vis = p.mpa ? load_mask<KPT>(mask, p.n_max, pos0) : 0u;
    uint32_t valid = valid_bits<KPT>(n, pos0);
    if (kPool) {  // proxy tokens retained unconditionally: not ranked, always emitted
      forced = valid & ~valid_bits<KPT>(wfrom, pos0);
      valid &= ~forced;
    }
    if (valid != valid_bits<KPT>(KPT, 0)) {
#pragma unroll
      for (int j = 0; j < KPT; ++j)
        if (!((valid >> j) & 1u)) key[j] = kNoKey;
    }
  };

  // ---- range of the keys
  uint32_t kmax = 0, kmin = 0xffffffffu;
  for (int r = 0; r < rounds; ++r) {
    load_round(r);
#pragma unroll
    for (int j = 0; j < KPT; ++j) {
      kmax = (uint32_t)max((int)kmax, (int)key[j]);  // (kNoKey is negative)
      kmin = min(kmin, key[j]);
    }
  }
  team_range<TEAM, 1>(sh, rank, kmax, kmin);
  auto to_t = [&]() {
#pragma unroll
    for (int j = 0; j < KPT; ++j) key[j] = key[j] == kNoKey ? kNoKey : kmax - key[j];
  };
  if (rounds == 1) to_t();
  auto reload = [&](int r) {
    if (rounds > 1) {
      load_round(r);
      to_t();
    }
  };

  RankRange r0 = want0 ? RankRange{0u, kmax - kmin, kNoKey, 0u} : RankRange{kNowhere, 0u, 0u, 0u};
  RankRange r1 = want1 ? RankRange{0u, kmax - kmin, kNoKey, 0u} : RankRange{kNowhere, 0u, 0u, 0u};
  bool short0 = false, short1 = false;  // the modality has no more keys than are wanted: all of them are kept
  auto crowded = [](const RankRange& g) { return g.in > kListCap && g.span > 0; };
  uint32_t n_vis = 0;  // visual tokens in the ranking

  for (int pass = 0; pass < 2; ++pass) {
    // ---- buckets
    const int shift0 = range_shift(pass ? r0.span : kmax - kmin, SH::kDig), shift1 = range_shift(pass ? r1.span : kmax - kmin, SH::kDig);
    if (pass == 0) {  // all keys take part, both modalities over the same range (one of which nothing is wanted is not walked)
      for (int r = 0; r < rounds; ++r) {
        reload(r);
#pragma unroll
        for (int j = 0; j < KPT; ++j)
          atomicAdd(sh.cnt + ((vis >> j) & 1u ? 0 : SH::kStride) + min(key[j] >> shift0, (uint32_t)SH::kBuckets), 1u);
      }
    } else {
      for (int x = tid; x < 2 * SH::kStride / 4; x += kRankThreads) reinterpret_cast<uint4*>(sh.cnt)[x] = make_uint4(0, 0, 0, 0);
      __syncthreads();
      for (int r = 0; r < rounds; ++r) {
        reload(r);
#pragma unroll
        for (int j = 0; j < KPT; ++j) {
          const bool v = (vis >> j) & 1u;
          const uint32_t x = key[j] - (v ? r0.lo : r1.lo);
          if (x <= (v ? r0.span : r1.span)) atomicAdd(sh.cnt + (v ? 0 : SH::kStride) + (x >> (v ? shift0 : shift1)), 1u);
        }
      }
    }
    // ---- walk: block r of the team adds up its share of the buckets over all blocks; half of the threads per modality
    const int m = tid / kHalf, i = tid % kHalf;
    const uint32_t b0 = (rank * kHalf + i) * kPer;
    const uint32_t want = m ? want1 : want0;
    if (i == 0) sh.first[m] = ~0ull;  // (stays if the modality has fewer keys than wanted)
    team_sync<TEAM>();
    uint32_t c[kPer], lc = 0;
    bucket_counts<TEAM, 1>(sh, m * SH::kStride + b0, c);
#pragma unroll
    for (int k = 0; k < kPer; ++k) lc += c[k];
    uint32_t ic = warp_scan32(lc);
    if (lane == 31) sh.wscan_c[warp] = ic;
    __syncthreads();
    ic += __reduce_add_sync(kFull, lane >= m * (kRankWarps / 2) && lane < warp ? sh.wscan_c[lane] : 0u);
    if (i >= kHalf - 32) {  // the last warp of the modality has the block's total (in its last lane): to every block
      const uint32_t tc = __shfl_sync(kFull, ic, 31);
      if (lane < TEAM) peer_store<TEAM>(&sh.slice_c[m][rank], lane, tc);
    }
    if (TEAM > 1) {
      team_sync<TEAM>();
      ic += __reduce_add_sync(kFull, lane < (int)rank ? sh.slice_c[m][lane] : 0u);
    }
    ic += m ? r1.above : r0.above;
    if (want && ic - lc < want && ic >= want) {
      uint32_t run = ic - lc, at = 0, at_c = 0, at_in = 0;
#pragma unroll
      for (int k = 0; k < kPer; ++k) {
        if (run < want) {
          at = b0 + k;
          at_c = run;
          at_in = c[k];
        }
        run += c[k];
      }
#pragma unroll
      for (int r = 0; r < TEAM; ++r) {
        peer_store<TEAM>(&sh.first[m], r, ((u64)at_c << 32) | at);
        peer_store<TEAM>(&sh.last[m], r, (u64)at_in);
      }
    }
    team_sync<TEAM>();
    if (pass == 0) n_vis = __reduce_add_sync(kFull, lane < TEAM ? sh.slice_c[0][lane] : 0u);
    {
      auto narrow = [&](RankRange& g, bool& is_short, int q, int s) {
        if (sh.first[q] == ~0ull) {
          is_short = true;
          g = RankRange{kNowhere, 0u, 0u, 0u};
          return;
        }
        const uint32_t cut = (uint32_t)sh.first[q] << s;
        g.span = min(g.span - cut, (1u << s) - 1u);
        g.lo += cut;
        g.above = (uint32_t)(sh.first[q] >> 32);
        g.in = (uint32_t)sh.last[q];
      };
      if (want0 && !short0) narrow(r0, short0, 0, shift0);
      if (want1 && !short1) narrow(r1, short1, 1, shift1);
    }
    if (!crowded(r0) && !crowded(r1)) break;
  }

  // ---- (rare) too many keys in a range: halve it with exact sweeps until they fit the list or are all alike
  while (crowded(r0) || crowded(r1)) {
    const bool on0 = crowded(r0), on1 = crowded(r1);
    const uint32_t mid0 = r0.lo + (r0.span >> 1), mid1 = r1.lo + (r1.span >> 1);
    uint32_t c0 = 0, c1 = 0;
    for (int r = 0; r < rounds; ++r) {
      reload(r);
#pragma unroll
      for (int j = 0; j < KPT; ++j) {
        const bool v = (vis >> j) & 1u;
        if ((v ? on0 : on1) && key[j] >= (v ? r0.lo : r1.lo) && key[j] <= (v ? mid0 : mid1)) {
          if (v) ++c0; else ++c1;
        }
      }
    }
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
    auto halve = [](RankRange& g, uint32_t want, uint32_t c) {
      const uint32_t half = g.span >> 1;
      if (g.above + c >= want) {
        g.span = half;
        g.in = c;
      } else {
        g.above += c;
        g.in -= c;
        g.lo += half + 1;
        g.span -= half + 1;
      }
    };
    if (on0) halve(r0, want0, c0);
    if (on1) halve(r1, want1, c1);
    team_sync<TEAM>();
  }

  // ---- candidates of this block
  for (int r = 0; r < rounds; ++r) {
    reload(r);
    uint32_t in = 0;
#pragma unroll
    for (int j = 0; j < KPT; ++j) {
      const bool v = (vis >> j) & 1u;
      if (key[j] - (v ? r0.lo : r1.lo) <= (v ? r0.span : r1.span)) in |= 1u << j;
    }
    append<TEAM, 1, KPT>(sh, r0.in <= kListCap ? in & vis : 0u, r1.in <= kListCap ? in & ~vis : 0u, key, r0.lo, r1.lo);
  }
  team_sync<TEAM>();
  // ---- every block gathers the team's candidates and finds the thresholds: the smallest t up to which the wanted number of
  // keys lies, and how many keys of exactly that t are still wanted
  const uint32_t got = gather_lists<TEAM, 1>(sh);
  const bool on0 = want0 && !short0 && r0.in <= kListCap, on1 = want1 && !short1 && r1.in <= kListCap;
  finish_lists<TEAM, 1, false>(sh, r0, r1, got, on0, on1, want0, want1, 0ull, 0ull, kmax);
  // (nothing wanted: nothing lies before 0 and no tie is kept; all wanted: everything lies before kNowhere)
  const uint32_t thr0 = !want0 ? 0u : (short0 ? kNowhere : (on0 ? sh.fin_lo[0] : r0.lo));
  const uint32_t thr1 = !want1 ? 0u : (short1 ? kNowhere : (on1 ? sh.fin_lo[1] : r1.lo));
  const uint32_t ties0 = !want0 || short0 ? 0u : want0 - (on0 ? sh.fin_c[0] : r0.above);
  const uint32_t ties1 = !want1 || short1 ? 0u : want1 - (on1 ? sh.fin_c[1] : r1.above);

  // ---- ordered sweep: positions are consecutive within a thread, threads and blocks follow in position order. A key
  // before its modality's threshold is kept, one at the threshold while its rank among these ties (in position order) is
  // below the number still wanted. The counts of (ties v, ties t, kept outright) travel as one 3 x 21-bit word.
  uint32_t eq, gt;
  auto classify = [&]() {
    eq = gt = 0;
#pragma unroll
    for (int j = 0; j < KPT; ++j) {
      const uint32_t thr = (vis >> j) & 1u ? thr0 : thr1;
      if (key[j] == thr) eq |= 1u << j;
      if (key[j] < thr) gt |= 1u << j;
    }
    if (kPool) gt |= forced;
    return (u64)__popc(eq & vis) | ((u64)__popc(eq & ~vis) << 21) | ((u64)__popc(gt) << 42);
  };
  u64 before = 0;  // counts before this block (a block on its own needs no totals before it emits)
  u64 mine = 0;
  if (rounds == 1) {
    mine = classify();
  } else if (TEAM > 1) {
    for (int r = 0; r < rounds; ++r) {
      reload(r);
      mine += classify();
    }
  }
  u64 incl = warp_scan64(mine);
  if (lane == 31) sh.wscan_q[warp] = incl;
  __syncthreads();
  if (TEAM > 1) {
    if (warp == 0) {
      const u64 tot = warp_sum64(lane < kRankWarps ? sh.wscan_q[lane] : 0ull);
      if (lane < TEAM) peer_store<TEAM>(&sh.slice_q[0][rank], lane, tot);
    }
    team_sync<TEAM>();  // (also the last access to a peer's shared memory)
    before = warp_sum64(lane < (int)rank ? sh.slice_q[0][lane] : 0ull);
  }
  int64_t off0;
  if (p.alone) {
    // one sequence: the segments' lengths follow from the budgets and the modalities' token counts, which are at hand
    pdl_go();
    const int n_v = (int)n_vis + lo_v;
    auto length = [&](int x) {
      const int2 bud = __ldg(reinterpret_cast<const int2*>(p.budgets) + x);
      return (p.mpa ? min(max(bud.x, lo_v), n_v) : 0) + min(max(bud.y, lo_t), n - n_v);
    };
    u64 sum = 0;
    for (int x = tid; x < u; x += kRankThreads) sum += (u64)(length(x) + p.headroom);
    sum = warp_sum64(sum);
    __syncthreads();
    if (lane == 0) sh.wsum[0][warp] = sum;
    __syncthreads();
    off0 = (int64_t)warp_sum64(lane < kRankWarps ? sh.wsum[0][lane] : 0ull);
    const int len = length(u);
    const int64_t end = off0 + len + p.headroom;
    if (rank == 0 && tid == 0) {
      p.kept_len[u] = len;
      p.seg_off[u] = off0;
      if (u + 1 == p.units) {
        p.seg_off[p.units] = end;
        if (end > p.capacity) set_status(p.ws, MADAKV_ECAPACITY);
      }
    }
    if (end > p.capacity) return;
  } else {
    if (!kPool) pdl_wait();
    pdl_go();
    off0 = p.seg_off[u];
    if (off0 + p.kept_len[u] + p.headroom > p.capacity) return;  // seg_scan has raised MADAKV_ECAPACITY
  }
  auto emit = [&](int pos0, u64 ahead) {  // ahead: counts before this thread's positions
    const uint32_t e0 = (uint32_t)ahead & 0x1fffffu, e1 = (uint32_t)(ahead >> 21) & 0x1fffffu, g = (uint32_t)(ahead >> 42);
    int32_t* out = p.kept_idx + off0 + g + min(e0, ties0) + min(e1, ties1);
    uint32_t keep = gt;
    uint32_t ev = eq & vis, et = eq & ~vis;
    for (uint32_t k = e0; k < ties0 && ev; ++k) {  // lowest positions first
      keep |= ev & (0u - ev);
      ev &= ev - 1;
    }
    for (uint32_t k = e1; k < ties1 && et; ++k) {
      keep |= et & (0u - et);
      et &= et - 1;
    }
    while (keep) {
      const int j = __ffs(keep) - 1;
      keep &= keep - 1;
      *out++ = pos0 + j;
    }
  };
  if (rounds == 1) {
    emit(pos_first, before + incl - mine + warp_sum64(lane < warp ? sh.wscan_q[lane] : 0ull));
  } else {
    for (int r = 0; r < rounds; ++r) {
      reload(r);
      mine = classify();
      incl = warp_scan64(mine);
      __syncthreads();
      if (lane == 31) sh.wscan_r[warp] = incl;
      __syncthreads();
      const u64 ahead = before + incl - mine + warp_sum64(lane < warp ? sh.wscan_r[lane] : 0ull);
      before += warp_sum64(lane < kRankWarps ? sh.wscan_r[lane] : 0ull);
      emit(pos_first + r * kRound, ahead);
    }
  }
}

template <bool kPool>
void launch_select_unit(const madakv_config& c, const SelParams& p, cudaStream_t st) {
  const RankShape s = rank_shape(p.units, c.max_seq_len);
  switch (s.kpt + s.team) {
    case 8 + 1: launch_team(select_unit_kernel<8, 1, kPool>, p.units, 1, st, p); break;
    case 8 + 2: launch_team(select_unit_kernel<8, 2, kPool>, p.units, 2, st, p); break;
    case 8 + 4: launch_team(select_unit_kernel<8, 4, kPool>, p.units, 4, st, p); break;
    case 8 + 8: launch_team(select_unit_kernel<8, 8, kPool>, p.units, 8, st, p); break;
    case 16 + 1: launch_team(select_unit_kernel<16, 1, kPool>, p.units, 1, st, p); break;
    case 16 + 2: launch_team(select_unit_kernel<16, 2, kPool>, p.units, 2, st, p); break;
    case 16 + 4: launch_team(select_unit_kernel<16, 4, kPool>, p.units, 4, st, p); break;
    default: launch_team(select_unit_kernel<16, 8, kPool>, p.units, 8, st, p); break;
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
  // One sequence, few units: no kernel of its own for the scan of the segments (2 us on the host, 3-5 on the GPU). Units of
  // other sequences would need those sequences' visual-token counts, and a larger call is better off with a scan that runs
  // beside the ranking.
  p.alone = c.batch == 1 && p.units < 148;
  if (!p.alone) launch_pdl(seg_scan_kernel, dim3(1), dim3(1024), 0, st, p);
  if (c.pool_kernel > 1 || c.keep_window) launch_select_unit<true>(c, p, st);
  else launch_select_unit<false>(c, p, st);
  return launch_status();
}

}  // namespace madakv
