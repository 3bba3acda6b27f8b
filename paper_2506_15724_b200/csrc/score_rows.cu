// Stage 1, tensor-core path for wide windows (Eq. 7 with the softmax of Eq. 5): bf16 inputs whose logits do not fit a
// cluster's TMEM, fp32 inputs, and the single-pass form of stage 1 (log-sum-exps supplied by the caller).
//
// A launch takes up to 256 window rows per KV head (fp32: 128); shapes with more go in chunks of query heads (or, for
// windows beyond that, of window rows) one launch after the other, each adding its part to psi.
//
// fp32 inputs are split exactly into three bf16 numbers of 8 significand bits each, and a product q * k is taken as the six
// partial products that are not below 2^-24 of it: hi hi, hi mid, mid hi, mid mid, hi lo, lo hi, all accumulated in fp32.
// An SM's fp32 pipes do 256 FLOP per clock, its tensor cores 8192 / 6. In all but the smallest calls (split_first()) 16 warps of a
// CTA, in the place of the TMA producer and of most of the epilogue, load the fp32 rows and write the terms into the operands'
// shared memory, so that both passes read K as it is (CV). What bounds them is that conversion, 2700-3500 clocks per 64 columns of
// 128 keys and lately the operands' shared-memory traffic, 3072 + 768 clocks per tile of six products; the exponentials of 128 rows
// need 1024, so four epilogue warps do. (us with the terms of all keys written to the workspace by a kernel before, in slices of
// 96 MB -> now, but for the second accumulator of the MMA issuer, which costs the first pass a fifth at head_dim 64: 16 units of 73557 keys at most, 56 rows 1072 -> 329; 1024 of 1263, 64 rows 1064 -> 466; 8 of 82828, 224 rows 964 ->
// 450; 1280 of 2357, head_dim 64, 64 rows 1236 -> 600. Eight converting warps and eight or four for the epilogue: 379 and 359 on
// the first. An issuer chosen by elect.sync, which spares a move to a uniform register per operand, took the MMA issue from 5000 to
// 2900 clocks per tile.)
//
// With that many rows the work per key byte is dominated by the exponentials (g * w of them per key and pass), not
// by HBM: the special-function unit delivers 16 exp2 per clock and SM, which for 256 rows is 2048 clocks per 128-key
// tile against ~1400 clocks for reading the tile from HBM. The kernels are therefore built around keeping that unit
// busy.
//   pass 1  window rows on M (one or two blocks of 128 rows), the 128 keys of a tile on N: an epilogue thread owns
//           ONE window row (a TMEM lane) and a share of the tile's columns and keeps a running (max, sum of exp2) of
//           its row in registers, carried from tile to tile for as long as the CTA stays with the unit; one (max,
//           sum) pair per row, column share and run goes to the workspace
//   merge   per (unit, row): all pairs -> the row's log-sum-exp (a separate small kernel)
//   pass 2  the tile turned back (128 keys on M, the window rows on N): a thread owns one key and a quarter of the
//           window rows, and psi(i) = sum over rows of exp2(s - lse) is an in-thread sum over columns of its TMEM lane.
//           The shift by the row's log-sum-exp is part of the contraction: one more 16-deep step multiplies a
//           constant column of ones on the key side with -lse / scale (as three bf16 terms) on the row side, so the
//           accumulator arrives shifted and the epilogue reads no per-row operand (with the log-sum-exps as
//           shared-memory broadcasts the loads competed with the tensor core's operand reads and cost a fifth of
//           the pass). The four warps that share a key add their partial sums up through shared memory in a
//           fixed order.
// In both passes all 16 epilogue warps work on the same tile while the MMAs of the next tile fill the other half of
// the TMEM; the TMEM load of a warp's next 16 columns is in flight while it works on the present ones.
// K is streamed twice. The passes are separate launches and no CTA ever waits for another CTA. The work is the list
// of all 128-key tiles in (sequence, layer, KV head, tile) order; a CTA takes a contiguous range of it, the same
// number of tiles to within one for every CTA whatever the lengths in the batch. The part of a unit inside a CTA's
// range is a run: queries and log-sum-exps are loaded once per run, and pass 1 leaves one pair per run, so a unit's
// statistics come in as many pieces as CTAs share it (two or three for long sequences). Up to 128 rows the queries (and the
// shift rows) are double-buffered, so that the next unit's are there when its first keys are: with short sequences a CTA
// changes units every few tiles (5 tiles of 128 keys: a change took 7000 clocks, the tiles 4500). The first keys of a unit are
// always asked for before its queries. In a call of a few tiles per CTA the start counts as much as the tiles, so the
// partition is 32-bit arithmetic on lengths in shared memory. Warp roles: warp 0 TMA
// producer, warp 1 MMA issuer and TMEM owner, warps 2-17 epilogue; TMEM lane quarter = warp % 4 throughout. Every wait is bounded: on expiry the kernel records MADAKV_ETIMEOUT, drains and returns.
#include "tc_common.cuh"

namespace madakv {
namespace {

constexpr int kConvertWarps = 16;  // CV: the last 16 warps
constexpr int kMaxSeqScan = 1024; // batches up to this size get the exact (ragged-aware) tile partition
constexpr int kFoldTiles = 16;    // pass 1 moves a row's sum to its second level every this many tiles

// Division of numbers below 2^31 by a number known on the host: a multiplication (Granlund and Montgomery, "Division by invariant
// integers using multiplication", 1994, the multiplier rounded up) instead of some forty instructions, of which every warp of a
// CTA did several before its first tile.
struct FastDiv {
  uint32_t d, mul, shift;
  explicit FastDiv(int by = 1) : d((uint32_t)by), shift(0) {
    while ((1ull << shift) < d) ++shift;
    mul = (uint32_t)((((1ull << shift) - d) << 32) / d + 1);
  }
  __device__ __forceinline__ int div(int x) const { return (int)((__umulhi((uint32_t)x, mul) + (uint32_t)x) >> shift); }
};

struct RowParams {
  const int32_t* seq_len;
  float* psi;        // [units, n_max]
  float2* part;      // ws: [units, smax, cparts, rs] (max, sum) of every row over a column share of one CTA's run
  const float* given_lse;  // pass 2: natural-log sum-exps [B, L, Hq, w] supplied by the caller (lse2 is not used then)
  const float* lse2; // ws: [units, rs] NEGATED log2-domain log-sum-exp, padding rows hold kEmptyMax (pass 2)
  int32_t* status;   // ws header
  int B, units, L, Hq, Hkv, g, w, R, n_max, causal, rs, mblocks, cparts, n16;  // n16: R rounded up to 16
  int lh;            // units per sequence
  FastDiv by_hkv, by_wc, by_grid, by_per;
  const float *qf, *kf;  // fp32 inputs
  madakv_strides sq, sk; // of fp32 inputs, in elements
  int h0, r0, wc;    // the launch's window rows: rows [r0, r0 + wc) of query heads h0 .. of the group, R = heads * wc
  int accumulate;    // psi += instead of =
  int smax;          // runs (CTAs) a unit's tiles can be spread over at most: wide_max_runs()
  int grid;          // CTAs of the two passes (the merge kernel needs the partition)
  int per, slack;    // CTAs per unit (0: fewer CTAs than units), tiles a CTA may have more for it: see partition_of()
  float scale2;
  // 1 / scale2 as the sum of two. In 32 bits it is off by 2.8e-8 for head_dim 128 (64 rows, 20480 keys: 2-norm of the scores' error
  // 3.6e-7 -> 1.8e-7). bf16 with given log-sum-exps does without the second (0), because the first one's error makes up for a part
  // of what the accumulation of q.k cuts off the largest logits (3.3e-7, with the second 6.9e-7).
  float inv, inv_more;
};

template <int D, int PASS, int NS, bool CV>  // NS: bf16 terms per operand (1, or 3 for fp32); CV: fp32 inputs are split here
struct RowSmem {
  // NS = 1: a stage is a whole K tile. NS = 3: a stage is one 64-wide piece of one term of it, 16 KB.
  // pass 2 gives up K stages for the operands of its extra contraction step (see the MMA issuer)
  static constexpr int kStages = NS == 3 ? (PASS == 2 ? 5 : 6 + CV) : (D == 128 ? 4 : 8) - (PASS == 2 ? (D == 128 ? 1 : 2) : 0);
  static constexpr int kKBlocks = D / 64;
  static constexpr int kPieces = NS == 3 ? 3 * kKBlocks : 1;  // stages per tile
  static constexpr int kEpiWarps = CV ? 4 : 16;
  static constexpr int kThreads = 32 * (2 + kEpiWarps + (CV ? kConvertWarps : 0));
  static constexpr int kShares = kEpiWarps / 4;       // column shares of a row block (pass 1), of a tile's rows (pass 2)
  static constexpr int kStageBytes = NS == 3 ? kTileKeys * 128 : kTileKeys * D * 2;
  static constexpr int kQRows = NS == 3 ? 128 : 256;  // up to two blocks of 128 rows
  static constexpr int kQBytes = kQRows * D * 2 * NS;
  static constexpr int kKOff = 0;
  static constexpr int kQOff = kStages * kStageBytes;
  static constexpr int kOnesOff = kQOff + kQBytes;                          // pass 2: [128 keys][64] bf16, 1 in columns 0-2
  static constexpr int kShiftOff = kOnesOff + (PASS == 2 ? 128 * 128 : 0);  // pass 2: [rows][64] bf16, columns 0-2
  static constexpr int kBarOff = kShiftOff + (PASS == 2 ? kQRows * 128 : 0);
  // full[kStages], empty[kStages], qfull[2], qempty[2], tfull[2], tempty[2], drain, xfull[8], xempty[8]
  static constexpr int kNumBars = 2 * kStages + 4 + 4 + 1 + 16;
  static constexpr int kMiscOff = (kBarOff + kNumBars * 8 + 15) / 16 * 16;
  static constexpr int kFirstOff = kMiscOff + 48;          // the CTA's first run and the cursor behind it
  static constexpr int kColOff = kFirstOff + 64;           // window position (row % w) of every row [256]
  static constexpr int kOffOff = kColOff + 256 * 4;        // pass 2: place of every row in the group's log-sum-exps [256]
  static constexpr int kXchOff = kOffOff + 256 * 4;        // pass 2: partial psi of column shares 1-3 [2][3][128]
  static constexpr int kLenOff = kXchOff + 6 * 128 * 4;    // lengths of the sequences
  static constexpr int kTotal = kLenOff + kMaxSeqScan * 4;
  static constexpr int kAlloc = kTotal + 1024;
  static_assert(kQOff % 1024 == 0 && kOnesOff % 1024 == 0 && kShiftOff % 1024 == 0 && kBarOff % 8 == 0, "alignment");
  static_assert(kAlloc <= 227 * 1024, "shared memory");
};

// Instruction descriptor: bf16 x bf16 -> fp32, both operands K-major, M = 128, N = 128.
constexpr uint32_t kIdescRows = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(128 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);

// exp2 of 8 packed pairs, summed
__device__ __forceinline__ uint64_t exp2_sum16(const uint64_t (&x)[8]) {
  uint64_t e[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    float lo, hi;
    unpack2(x[i], lo, hi);
    e[i] = pack2(ex2(lo), ex2(hi));
  }
  return add2(add2(add2(e[0], e[1]), add2(e[2], e[3])), add2(add2(e[4], e[5]), add2(e[6], e[7])));
}

__device__ __forceinline__ float sum4(const uint64_t (&a)[4]) {
  float lo, hi;
  unpack2(add2(add2(a[0], a[1]), add2(a[2], a[3])), lo, hi);
  return lo + hi;
}
__device__ __forceinline__ float block_max16(const uint32_t (&r)[16]) {
  const float a0 = max3f(__uint_as_float(r[0]), __uint_as_float(r[1]), __uint_as_float(r[2]));
  const float a1 = max3f(__uint_as_float(r[3]), __uint_as_float(r[4]), __uint_as_float(r[5]));
  const float a2 = max3f(__uint_as_float(r[6]), __uint_as_float(r[7]), __uint_as_float(r[8]));
  const float a3 = max3f(__uint_as_float(r[9]), __uint_as_float(r[10]), __uint_as_float(r[11]));
  const float a4 = max3f(__uint_as_float(r[12]), __uint_as_float(r[13]), __uint_as_float(r[14]));
  return max3f(max3f(a0, a1, a2), a3, fmaxf(a4, __uint_as_float(r[15])));
}

// A tile's NB blocks of 16 accumulator columns of this thread's TMEM lane, none of them masked, as a software
// pipeline over steps of 8 columns: the exponentials of step s are queued on the special-function unit, then the
// results of step s - 1 are added up and the inputs of step s + 1 prepared, so that a warp on its own keeps the unit
// supplied (with the steps one after the other a lone warp kept it half busy, and at the end of every tile the
// last warps of a scheduler are on their own). The TMEM load of block j + 1 is in flight during block j.
//
// Pass 2: acc += exp2(scale2 * column); the accumulator already holds q.k - lse / scale.
template <int NB>
__device__ __forceinline__ void psi_tile(uint32_t taddr, uint64_t sc2, uint64_t (&acc)[4]) {
  uint32_t r[2][16];
  uint64_t x[2][4], e[2][4];
  tmem_ld16_issue(taddr, r[0]);
  tmem_ld_wait16(r[0]);
  if (NB > 1) tmem_ld16_issue(taddr + 16, r[1]);
#pragma unroll
  for (int i = 0; i < 4; ++i) x[0][i] = mul2(pack2u(r[0][2 * i], r[0][2 * i + 1]), sc2);
#pragma unroll
  for (int s = 0; s < 2 * NB; ++s) {
    const int cur = s & 1, nxt = cur ^ 1;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float lo, hi;
      unpack2(x[cur][i], lo, hi);
      e[cur][i] = pack2(ex2(lo), ex2(hi));
    }
    if (s > 0) {
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[i] = add2(acc[i], e[nxt][i]);
    }
    if (s + 1 < 2 * NB) {
      const int blk = (s + 1) >> 1, half = (s + 1) & 1, b = blk & 1;
      if (half == 0) {
        tmem_ld_wait16(r[b]);
        if (blk + 1 < NB) tmem_ld16_issue(taddr + (blk + 1) * 16, r[b ^ 1]);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) x[nxt][i] = mul2(pack2u(r[b][8 * half + 2 * i], r[b][8 * half + 2 * i + 1]), sc2);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) acc[i] = add2(acc[i], e[(2 * NB - 1) & 1][i]);
}

// Pass 1: the row's running maximum m (log2 domain) is checked once per block; it rarely grows once a few hundred
// keys have been seen, so the rescaling sits behind a warp-uniform branch. acc holds the sum of exp2(scale2 * s - m)
// of the item at hand, z_run that of the run's earlier items.
template <int NB>
__device__ __forceinline__ void stat_tile(uint32_t taddr, float scale2, uint64_t sc2, float& m, uint64_t (&acc)[4],
                                          float& z_run) {
  uint32_t r[2][16];
  uint64_t x[2][4], e[2][4];
  auto grow = [&](float bm) {
    const float mn = fmaxf(m, bm);
    const float f = ex2(m - mn);
    const uint64_t f2 = pack2(f, f);
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i] = mul2(acc[i], f2);
    z_run *= f;
    m = mn;
  };
  tmem_ld16_issue(taddr, r[0]);
  tmem_ld_wait16(r[0]);
  if (NB > 1) tmem_ld16_issue(taddr + 16, r[1]);
  {
    const float bm = block_max16(r[0]) * scale2;
    if (__any_sync(0xffffffffu, bm > m)) grow(bm);
  }
  uint64_t nm2 = pack2(-m, -m);
#pragma unroll
  for (int i = 0; i < 4; ++i) x[0][i] = fma2(pack2u(r[0][2 * i], r[0][2 * i + 1]), sc2, nm2);
#pragma unroll
  for (int s = 0; s < 2 * NB; ++s) {
    const int cur = s & 1, nxt = cur ^ 1;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float lo, hi;
      unpack2(x[cur][i], lo, hi);
      e[cur][i] = pack2(ex2(lo), ex2(hi));
    }
    if (s > 0) {
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[i] = add2(acc[i], e[nxt][i]);
    }
    if (s + 1 < 2 * NB) {
      const int blk = (s + 1) >> 1, half = (s + 1) & 1, b = blk & 1;
      if (half == 0) {
        tmem_ld_wait16(r[b]);
        if (blk + 1 < NB) tmem_ld16_issue(taddr + (blk + 1) * 16, r[b ^ 1]);
        const float bm = block_max16(r[b]) * scale2;
        if (__any_sync(0xffffffffu, bm > m)) {
          // the exponentials just queued were taken against the old maximum: they go in before the rescaling
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            acc[i] = add2(acc[i], e[cur][i]);
            e[cur][i] = 0ull;
          }
          grow(bm);
          nm2 = pack2(-m, -m);
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) x[nxt][i] = fma2(pack2u(r[b][8 * half + 2 * i], r[b][8 * half + 2 * i + 1]), sc2, nm2);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) acc[i] = add2(acc[i], e[(2 * NB - 1) & 1][i]);
}

// The CTA's share of the work: a contiguous range of the 128-key tiles of all units, in (sequence, layer, KV head,
// tile) order, cut at tile granularity (every CTA gets the same number of tiles to within one, whatever the batch's
// length mix). The part of one unit inside a CTA's range is a run: the queries are loaded once per run, and pass 1
// leaves one (max, sum) pair per run, row and column share. Sequence b has L * Hkv * tiles_of(b) tiles.
struct TileCursor {
  int b;        // sequence
  int r;        // index among the tiles of sequence b
  int tb;       // tiles per unit of sequence b
  int per_b;    // tiles of sequence b
  int left;     // tiles of the range still to do
  int done;     // tiles of the range already done
};
struct Run {
  int u, b, n;  // unit, its sequence and that sequence's length
  int l, h;     // layer and KV head
  int t0, cnt;  // first tile of the run within the unit, tiles in the run (what the partition counts)
  int tiles;    // tiles of the run that hold keys (fewer than cnt only in the uniform partition of very large batches)
};

// `lens`: the lengths in shared memory, or null (batches too large for that: the uniform partition)
__device__ __forceinline__ int seq_length(const RowParams& p, const int* lens, int b) {
  return lens ? lens[b] : clamped_len(p.seq_len, b, p.n_max);
}
__device__ __forceinline__ int tiles_of(const RowParams& p, const int* lens, int b) {
  return ((lens ? lens[b] : p.n_max) + kTileKeys - 1) / kTileKeys;
}
__device__ __forceinline__ void cursor_settle(const RowParams& p, TileCursor& c, const int* lens) {
  // move on to the next sequence that has tiles
  while (c.left > 0 && c.r >= c.per_b) {
    c.r -= c.per_b;
    ++c.b;
    if (c.b >= p.B) {
      c.left = 0;
      break;
    }
    c.tb = tiles_of(p, lens, c.b);
    c.per_b = p.lh * c.tb;
  }
}
__device__ __forceinline__ Run cursor_run(const RowParams& p, const TileCursor& c, const int* lens) {
  Run r;
  int ub = 0;  // c.r / c.tb: by the reciprocal, then put right (it is off by one at most where there are fewer than 2^20 units)
  r.t0 = c.r;
  if (c.r >= c.tb) {
    ub = (int)__fdividef((float)c.r, (float)c.tb);
    r.t0 = c.r - ub * c.tb;
    while (r.t0 < 0) --ub, r.t0 += c.tb;
    while (r.t0 >= c.tb) ++ub, r.t0 -= c.tb;
  }
  r.l = p.by_hkv.div(ub);
  r.h = ub - r.l * p.Hkv;
  r.cnt = min(c.tb - r.t0, c.left);
  r.b = c.b;
  r.u = c.b * p.lh + ub;
  r.n = seq_length(p, lens, c.b);
  const int real = (r.n + kTileKeys - 1) / kTileKeys;  // tiles of the unit that hold keys
  r.tiles = max(0, min(r.t0 + r.cnt, real) - r.t0);
  return r;
}
__device__ __forceinline__ void cursor_advance(const RowParams& p, TileCursor& c, const Run& r, const int* lens) {
  c.r += r.cnt;
  c.left -= r.cnt;
  c.done += r.cnt;
  cursor_settle(p, c, lens);
}
// The partition: of `total` tiles CTA c of `ctas` gets [first_tile(c), first_tile(c + 1)), the first ones one more each.
// (The host refuses shapes with 2^30 tiles or more.) Units of equal length that are fewer than CTAs get `per` CTAs of their
// own each, if that makes no CTA's share longer by more than p.slack tiles: a CTA that changes units waits for the new row
// operands, 5000 clocks with one buffer for them, 2-3 tiles' time, and ends that much later than all others (4 units of 256
// tiles, 224 rows: three of 148 CTAs did, and a layer took 17.1 us; with this, and a start under
// the kernel before it (see score_rows_kernel), 14.8).
struct Partition {
  int total, ctas, per, tb;  // per: 0, or the CTAs of a unit, all of tb tiles
};
template <typename Tiles>
__device__ __forceinline__ Partition partition_of(const RowParams& p, bool exact, Tiles tiles) {
  Partition x{0, 0, 0, tiles(0)};
  bool same = exact && x.tb > 0 && p.per > 0;
  if (exact) {
    for (int b = 0; b < p.B; ++b) {
      const int tb = tiles(b);
      x.total += p.lh * tb;
      same = same && tb == x.tb;
    }
  } else {
    x.total = p.units * x.tb;
  }
  // (a batch with fewer tiles than CTAs is spread over as many CTAs as it has tiles: no empty range lies between
  // two CTAs that share a unit)
  x.ctas = min(x.total, p.grid);
  if (same && p.by_per.div(x.tb + p.per - 1) <= p.by_grid.div(x.total + p.grid - 1) + p.slack) x.per = p.per;
  return x;
}
__device__ __forceinline__ int first_tile(const RowParams& p, const Partition& x, int c) {  // (without CTAs of a unit's own)
  if (x.total < p.grid) return min(c, x.total);
  const int q = p.by_grid.div(x.total);
  return q * c + min(c, x.total - q * p.grid);
}
__device__ __forceinline__ int cta_of(int total, int ctas, int x) {
  const int q = total / ctas, more = total % ctas;
  return x < more * (q + 1) ? x / (q + 1) : more + (x - more * (q + 1)) / q;  // (x < total, so q > 0 in the second case)
}

// Four fp32 values as three bf16 terms each, whose sum is the value exactly (8 significand bits per term): lo goes to `store`,
// hi (x, y) and mid (z, w) are returned, packed. The conversion stops at the largest finite number, which is exact for values that
// would round up to infinity; of an infinity all three terms are that number, so that its products have the sign of an
// infinity's (and none is infinite that should not be, for partners below 2^9), not NaN.
template <typename Store>
__device__ __forceinline__ uint4 split4(float4 v, Store store) {
  auto pack = [](float a, float b) {
    uint32_t x;
    asm("cvt.rn.satfinite.bf16x2.f32 %0, %1, %2;" : "=r"(x) : "f"(b), "f"(a));
    return x;
  };
  auto low = [](uint32_t x) { return __uint_as_float(x << 16); };
  auto high = [](uint32_t x) { return __uint_as_float(x & 0xffff0000u); };
  uint4 t;
  t.x = pack(v.x, v.y);
  t.y = pack(v.z, v.w);
  v.x = __fsub_rn(v.x, low(t.x));
  v.y = __fsub_rn(v.y, high(t.x));
  v.z = __fsub_rn(v.z, low(t.y));
  v.w = __fsub_rn(v.w, high(t.y));
  t.z = pack(v.x, v.y);
  t.w = pack(v.z, v.w);
  store(make_uint2(pack(__fsub_rn(v.x, low(t.z)), __fsub_rn(v.y, high(t.z))), pack(__fsub_rn(v.z, low(t.w)), __fsub_rn(v.w, high(t.w)))));
  return t;
}

// A load that stays where it is written (the compiler may move a plain one down to its use, which is a step later).
__device__ __forceinline__ float4 load4(const float* p) {
  float4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}

template <int D, int PASS, int NS, bool CV>
__global__ void __launch_bounds__((RowSmem<D, PASS, NS, CV>::kThreads), 1)  // 96 registers: warps are allocated four at a time (18 -> 20); CV: 80 (22 -> 24)
score_rows_kernel(const __grid_constant__ CUtensorMap tmap_k, const __grid_constant__ CUtensorMap tmap_q, RowParams p) {
  using SL = RowSmem<D, PASS, NS, CV>;
  constexpr int kStages = SL::kStages;
  constexpr int kKBlocks = SL::kKBlocks;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* k_s = smem + SL::kKOff;
  uint8_t* q_s = smem + SL::kQOff;
  uint8_t* ones_s = smem + SL::kOnesOff;
  uint8_t* shift_s = smem + SL::kShiftOff;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + SL::kBarOff);
  uint64_t* full = bars;               // [kStages] TMA -> MMA
  uint64_t* empty = bars + kStages;    // [kStages] MMA -> TMA
  uint64_t* qfull = empty + kStages;   // [2]       TMA (and in pass 2 the shift rows' warp) -> MMA: a unit's row operands
  uint64_t* qempty = qfull + 2;        // [2]       MMA -> TMA
  uint64_t* tfull = qempty + 2;        // [2]       MMA -> epilogue
  uint64_t* tempty = tfull + 2;        // [2]       epilogue -> MMA
  uint64_t* drain = tempty + 2;        // [1]
  uint64_t* xfull = drain + 1;         // [2][4]    pass 2: column shares 1-3 -> share 0, per buffer and lane quarter
  uint64_t* xempty = xfull + 8;        // [2][4]    pass 2: share 0 -> shares 1-3
  uint32_t* tmem_base_s = reinterpret_cast<uint32_t*>(smem + SL::kMiscOff);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + SL::kMiscOff + 4);
  int* range_s = reinterpret_cast<int*>(smem + SL::kMiscOff + 8);  // are there empty sequences, first tile, total, CTAs in use, CTAs per unit or 0
  int* len_s = reinterpret_cast<int*>(smem + SL::kLenOff);
  int* rowpos = reinterpret_cast<int*>(smem + SL::kColOff);
  int* rowoff = reinterpret_cast<int*>(smem + SL::kOffOff);
  float* xch = reinterpret_cast<float*>(smem + SL::kXchOff);
  int* rowhead = reinterpret_cast<int*>(xch);  // fp32, whose tiles are not shared out: query head of every row within the launch's

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  // The lengths are read, the CTA's range is found and its first operands are asked for (into the L2) under the kernel before
  // this one, on whose results none of that rests: the lengths are read again behind the wait, and should one have changed the
  // range is found anew. Apart from that nothing before the wait touches more than this CTA's shared memory and TMEM. In a call
  // of a few tiles per CTA the way to the first MMA counts as much as the tiles, and what it costs is instructions that
  // are run once, by one warp: so all threads together write the first unit's shift rows, only what the MMAs read is
  // cleared, and the roles find the first run in shared memory. (Range, loads and shift rows one after the other behind the
  // wait, 112 KB cleared: first MMA 7000 clocks behind it; now 2700. One layer of 4 units of 256 tiles, 224 rows: 17.1 -> 14.8 us;
  // 8 units of 33 tiles, 448 rows in two chunks 20.9 -> 19.3; an fp32 call of 4 units of 4 tiles 17.1 -> 16.3. Prefetching by one
  // instruction per 128 bytes and thread, and the range by a warp of its own: slower where CTAs change units, 373 against 346 us
  // for 32 layers of 40 units of 20 tiles.)
  const int* lens = p.B <= kMaxSeqScan ? len_s : nullptr;
  auto length_now = [&](int b) { return max(0, min(__ldcg(p.seq_len + b), p.n_max)); };
  auto read_lengths = [&]() {  // (by the last threads first: the first warps have more to set up)
    if (lens)
      for (int b = SL::kThreads - 1 - (int)threadIdx.x; b < p.B; b += SL::kThreads) len_s[b] = length_now(b);
  };
  read_lengths();
  if (warp == 0) {
    for (int x = lane; x < SL::kNumBars; x += 32) {
      const int y = x - 2 * kStages;  // qfull, qempty, tfull, tempty, drain, xfull, xempty from 0 on
      uint32_t count = 1;
      if (x < kStages) count = CV ? kConvertWarps : 1;
      if (y >= 0 && y < 2) count = (CV ? kConvertWarps : 1) + (PASS == 2 ? 1 : 0);
      if (y >= 6 && y < 8) count = 32 * SL::kEpiWarps;  // every epilogue thread
      if (y >= 9 && y < 17) count = SL::kShares > 1 ? 32 * (SL::kShares - 1) : 1;
      if (y >= 17) count = 32;
      mbar_init(&bars[x], count);
    }
    if (lane == 0) *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // Rows R.. of the Q buffers are never written by TMA: keep them zero so their logits are 0 (CV writes all rows; where
  // the operands are fp32 terms or have two buffers all of them are cleared). Pass 2: of the operands of the extra contraction step an MMA reads
  // columns 0-15 of every row, two 16-byte pieces (128-byte rows with the 128-byte swizzle: piece x of row r sits at position
  // x ^ (r % 8)): the key side gets its three ones per row, the shift rows start as zeros.
  {
    const bool some = NS == 1 && p.R > 128;
    const int rows = some ? SL::kQRows - p.R : SL::kQRows;
#pragma unroll 1
    for (int kb = 0; kb < (CV ? 0 : kKBlocks * NS); ++kb) {
      uint4* at = reinterpret_cast<uint4*>(q_s + (kb * SL::kQRows + (some ? p.R : 0)) * 128);
      for (int x = threadIdx.x; x < rows * 8; x += SL::kThreads) at[x] = make_uint4(0, 0, 0, 0);
    }
  }
  if (PASS == 2) {
    for (int x = threadIdx.x; x < 2 * (SL::kQRows + kTileKeys); x += SL::kThreads) {
      const int piece = x & 1, r = x >> 1, rr = r < SL::kQRows ? r : r - SL::kQRows;
      uint8_t* at = (r < SL::kQRows ? shift_s : ones_s) + rr * 128 + ((piece ^ (rr & 7)) * 16);
      *reinterpret_cast<uint4*>(at) = r >= SL::kQRows && !piece ? make_uint4(0x3f803f80u, 0x00003f80u, 0u, 0u) : make_uint4(0, 0, 0, 0);
    }
  }
  if (threadIdx.x < 256) {
    const int x = threadIdx.x, hh = p.by_wc.div(x), pos = p.r0 + x - hh * p.wc;
    rowpos[x] = pos;
    if (CV && x < 128) rowhead[x] = hh;
    rowoff[x] = x < p.R ? hh * p.w + pos : 0;
  }
  if (!CV && threadIdx.x == 32) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmap_k) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmap_q) : "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_base_s)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  struct First {  // what the roles need of the CTA's first run
    Run run;
    TileCursor behind;
  };
  static_assert(sizeof(First) <= 64, "its place in shared memory");
  First* first_s = reinterpret_cast<First*>(smem + SL::kFirstOff);
  auto find_range = [&]() {  // one thread
    const Partition x = partition_of(p, lens != nullptr, [&](int b) { return tiles_of(p, lens, b); });
    int none = 0;
    if (lens)
      for (int b = 0; b < p.B; ++b) none |= lens[b] == 0 ? 1 : 0;
    range_s[0] = none;
    range_s[2] = x.total;
    range_s[3] = x.ctas;
    range_s[4] = x.per;
    if (x.per) {  // a part of one unit
      const int u = p.by_per.div(blockIdx.x), i = (int)blockIdx.x - u * x.per, q = p.by_per.div(x.tb), more = x.tb - q * x.per;
      Run run = {};
      if (u < p.units) {
        run.u = u;
        for (run.b = 0; u >= (run.b + 1) * p.lh;) ++run.b;
        const int ub = u - run.b * p.lh;
        run.n = lens[run.b];
        run.l = p.by_hkv.div(ub);
        run.h = ub - run.l * p.Hkv;
        run.t0 = i * q + min(i, more);
        run.cnt = run.tiles = q + (i < more ? 1 : 0);
      }
      range_s[1] = u * x.tb + run.t0;
      first_s->run = run;
      TileCursor none_left = {};
      none_left.done = run.cnt;
      first_s->behind = none_left;
      return;
    }
    const int lo = first_tile(p, x, blockIdx.x), hi = first_tile(p, x, blockIdx.x + 1);
    int b0 = 0, r0 = lo;
    if (lens) {
      while (b0 < p.B) {
        const int per = p.lh * tiles_of(p, lens, b0);
        if (r0 < per) break;
        r0 -= per;
        ++b0;
      }
    } else {
      const int per = p.lh * tiles_of(p, lens, 0);
      b0 = lo / per;
      r0 = lo - b0 * per;
    }
    range_s[1] = lo;
    TileCursor c;
    c.b = b0;
    c.r = r0;
    c.left = c.b < p.B ? hi - lo : 0;
    c.done = 0;
    c.tb = c.left > 0 ? tiles_of(p, lens, c.b) : 1;
    c.per_b = p.lh * c.tb;
    cursor_settle(p, c, lens);
    Run run = {};
    if (c.left > 0) {
      run = cursor_run(p, c, lens);
      cursor_advance(p, c, run, lens);
    }
    first_s->run = run;
    first_s->behind = c;
  };
  // Where a role starts, and its next run: the first one from shared memory, the others from the cursor.
  auto cursor_begin = [&]() {
    TileCursor c = {};
    c.left = first_s->run.cnt;
    return c;
  };
  auto take_run = [&](TileCursor& c) {
    Run run;
    if (c.done == 0) {
      run = first_s->run;
      c = first_s->behind;
    } else {
      run = cursor_run(p, c, lens);
      cursor_advance(p, c, run, lens);
    }
    return run;
  };
  __syncthreads();
  if (warp == 0) {
    if (lens && lane == 0) find_range();
    __syncwarp();
    if (NS == 1 && lens && first_s->run.tiles > 0) {
      const Run run = first_s->run;
      if (PASS == 2 && p.given_lse) {
        const float* src = p.given_lse + (((int64_t)run.b * p.L + run.l) * p.Hq + run.h * p.g + p.h0) * p.w;
        if (lane * 32 < p.R) asm volatile("prefetch.global.L2 [%0];" ::"l"(src + rowoff[lane * 32]));
      }
      if (lane < 2 * kKBlocks) {  // the queries and the first tiles, half a row at a time
        const bool is_q = lane < kKBlocks;
        const int kb = lane % kKBlocks;
        for (int t = 0; t < (is_q ? 1 : min(run.tiles, kStages)); ++t)
          tma_prefetch_5d(is_q ? &tmap_q : &tmap_k, kb * 64, is_q ? p.r0 : (run.t0 + t) * kTileKeys, is_q ? run.h * p.g + p.h0 : run.h, run.l, run.b);
      }
    }
  }
  pdl_wait();
  pdl_go();
  bool moved = !lens;  // (very large batches: found behind the wait)
  if (lens)
    for (int b = SL::kThreads - 1 - (int)threadIdx.x; b < p.B; b += SL::kThreads) moved = moved || length_now(b) != len_s[b];
  if (__syncthreads_or(moved)) {
    read_lengths();
    __syncthreads();
    if (threadIdx.x == 0) find_range();
    __syncthreads();
  }
  // Row r of the shift operand: -lse_r / scale as the sum of three bf16 numbers (24 bits) in columns 0-2. Multiplied by
  // the key side's ones in the extra contraction step, the accumulator holds q.k - lse / scale and the epilogue needs no
  // per-row operand at all.
  auto load_lse = [&](const Run& run, int r) {
    const float* src = p.given_lse ? p.given_lse + (((int64_t)run.b * p.L + run.l) * p.Hq + run.h * p.g + p.h0) * p.w : p.lse2 + (int64_t)run.u * p.rs;
    return __ldcg(src + (p.given_lse ? rowoff[r] : min(r, p.rs - 1)));
  };
  auto store_shift = [&](int buf, int r, float nl) {
    // a row that sees no key (-inf) and the padding rows get a shift that turns every weight into 0
    if (p.given_lse) nl = nl > -INFINITY ? -nl * kLog2e : kEmptyMax;
    if (r >= p.R) nl = kEmptyMax;
    if (r < p.n16) {
      // (v + more is the quotient to some 40 bits, see RowParams)
      const float v = nl * p.inv, more = p.inv_more != 0.f ? fmaf(nl, p.inv, -v) + nl * p.inv_more : 0.f;
      const float hi = __bfloat162float(__float2bfloat16_rn(v)), rest = (v - hi) + more;
      const float mid = __bfloat162float(__float2bfloat16_rn(rest));
      const float low = __bfloat162float(__float2bfloat16_rn(rest - mid));
      const uint32_t w0 = (__float_as_uint(hi) >> 16) | (__float_as_uint(mid) & 0xffff0000u);
      *reinterpret_cast<uint4*>(shift_s + (buf * 128 + r) * 128 + (r & 7) * 16) = make_uint4(w0, __float_as_uint(low) >> 16, 0u, 0u);
    }
  };
  // The first unit's operands, before the roles begin: one thread asks for them, all write the shift rows.
  const bool begun = first_s->run.tiles > 0;
  const int ahead0 = NS == 1 ? min(kStages, first_s->run.tiles) : 0;
  if (begun) {
    const Run run = first_s->run;
    if (NS == 1 && threadIdx.x == 0) {
      const uint64_t pol_k = l2_policy_evict_first(), pol_q = l2_policy_evict_last();
      for (int t = 0; t < ahead0; ++t) {
        mbar_expect_tx(&full[t], (uint32_t)SL::kStageBytes);
        for (int kb = 0; kb < kKBlocks; ++kb)
          tma_load_5d(k_s + t * SL::kStageBytes + kb * kTileKeys * 128, &tmap_k, &full[t], kb * 64, (run.t0 + t) * kTileKeys, run.h, run.l, run.b, pol_k);
        if (t) continue;
        mbar_expect_tx(&qfull[0], (uint32_t)(p.R * 128 * kKBlocks));
        for (int kb = 0; kb < kKBlocks; ++kb)
          tma_load_5d(q_s + kb * SL::kQRows * 128, &tmap_q, &qfull[0], kb * 64, p.r0, run.h * p.g + p.h0, run.l, run.b, pol_q);
      }
    }
    if (PASS == 2 && (int)threadIdx.x >= 32 && (int)threadIdx.x < 32 + SL::kQRows) store_shift(0, threadIdx.x - 32, load_lse(run, threadIdx.x - 32));
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_base_s;
  const int nq = NS == 1 && p.R <= 128 ? 2 : 1;  // buffers of the row operands: buffer i starts at row 128 * i

  if (warp == 0) {
    // ================================================================ TMA producer: lane 0 waits and issues the copies;
    // in pass 2 all lanes write the units' shift rows (with
    // CV all that this warp does)
    const uint64_t pol_k = NS == 3 ? l2_policy_evict_last() : l2_policy_evict_first();  // (split keys are read again)
    const uint64_t pol_q = l2_policy_evict_last();
    int stage = ahead0 % kStages, k = 0;  // k: units begun
    uint32_t stage_par = ahead0 == kStages ? 1u : 0u;
    bool ok = true;
    if (PASS == 2 && begun && lane == 0) mbar_arrive(&qfull[0]);  // (its shift rows)
    for (TileCursor c = cursor_begin(); ok && c.left > 0;) {
      const Run run = take_run(c);
      const int u = run.u, key_begin = run.t0 * kTileKeys, loads = run.tiles * SL::kPieces;
      if (loads == 0) continue;
      const int h = run.h, l = run.l, b = run.b;
      // split operands are [units][n_max][3 D] and [units * g][w][3 D]
      const int th = NS == 3 ? u : h, tl = NS == 3 ? 0 : l, tb = NS == 3 ? 0 : b;
      const int buf = k % nq;
      const uint32_t q_par = (uint32_t)(k / nq) & 1u;
      const bool under_way = k == 0 && begun;  // the first unit's shift rows are written, and with NS = 1 its first loads issued
      float nl[SL::kQRows / 32];  // (all loads first; one after the other they took 5 us)
      if (PASS == 2 && !under_way) {
#pragma unroll
        for (int i = 0; i < SL::kQRows / 32; ++i) nl[i] = load_lse(run, lane + 32 * i);
      }
      // [from, to) of the unit's K loads, by lane 0
      auto load_keys = [&](int from, int to) {
        for (int x = from; ok && x < to; ++x) {
          const int t = x / SL::kPieces, piece = x % SL::kPieces;
          ok = mbar_wait(&empty[stage], stage_par ^ 1, abort_flag, p.status, kSiteStage);
          if (!ok) break;
          mbar_expect_tx(&full[stage], (uint32_t)SL::kStageBytes);
          if (NS == 3) {  // (the order of the MMA issuer: lo, mid, hi of 64 columns, then of the others)
            tma_load_5d(k_s + stage * SL::kStageBytes, &tmap_k, &full[stage], ((2 - piece % 3) * kKBlocks + piece / 3) * 64,
                        key_begin + t * kTileKeys, th, tl, tb, pol_k);
          } else {
            for (int kb = 0; kb < kKBlocks; ++kb)
              tma_load_5d(k_s + stage * SL::kStageBytes + kb * kTileKeys * 128, &tmap_k, &full[stage], kb * 64,
                          key_begin + t * kTileKeys, th, tl, tb, pol_k);
          }
          if (++stage == kStages) {
            stage = 0;
            stage_par ^= 1;
          }
        }
      };
      // The unit's queries once the stages are full of its keys (those stages were the unit's before, whose tiles need
      // nothing that is still to come; from the next load on the stages wait for this unit's own tiles); the first
      // unit's at once.
      const int ahead = k == 0 ? (NS == 1 && begun ? ahead0 : 1) : min(kStages, loads);
      ++k;
      if (lane == 0 && !(NS == 1 && under_way)) {
        if (!CV) load_keys(0, ahead);
        ok = ok && mbar_wait(&qempty[buf], q_par ^ 1, abort_flag, p.status, kSiteQEmpty);
        if (ok && !CV) {
          mbar_expect_tx(&qfull[buf], (uint32_t)(p.R * 128 * kKBlocks * NS));
          for (int kb = 0; kb < kKBlocks * NS; ++kb)
            tma_load_5d(q_s + (kb * SL::kQRows + buf * 128) * 128, &tmap_q, &qfull[buf], kb * 64, p.r0, th * p.g + p.h0, tl, tb, pol_q);
        }
      }
      if (PASS == 2 && !under_way) {
        ok = __shfl_sync(0xffffffffu, ok, 0);
        if (!ok) break;
#pragma unroll
        for (int i = 0; i < SL::kQRows / 32; ++i) store_shift(buf, lane + 32 * i, nl[i]);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();  // every lane's rows are written (and fenced) before lane 0 signals them
        if (lane == 0) mbar_arrive(&qfull[buf]);
      }
      if (NS == 1 && nq == 1 && lane == 0 && c.left > 0) {  // the next unit's queries, to the L2: their place here is free only when this unit's MMAs are done
        const Run next = cursor_run(p, c, lens);
        for (int kb = 0; kb < kKBlocks; ++kb) tma_prefetch_5d(&tmap_q, kb * 64, p.r0, next.h * p.g + p.h0, next.l, next.b);
      }
      if (!CV && lane == 0) load_keys(ahead, loads);
      ok = __shfl_sync(0xffffffffu, ok, 0);
    }
    if (!CV && !ok && lane == 0) {  // abandoned: give copies in flight time to land before the CTA's shared memory goes away
      const long long t0 = clock64();
      while (clock64() - t0 < 2000000ll) __nanosleep(1000);
    }
  } else if (warp == 1) {
    // ================================================================ MMA issuer
    if (CV ? elect_one() : lane == 0) {
      const uint32_t k_lo0 = smem_desc_lo(smem_u32(k_s)), q_lo00 = smem_desc_lo(smem_u32(q_s));
      const uint32_t ones_lo = smem_desc_lo(smem_u32(ones_s)), shift_lo0 = smem_desc_lo(smem_u32(shift_s));
      const uint32_t idesc2 = instr_desc_bf16(p.n16);
      int stage = 0, n_tile = 0, k = 0;  // k: units begun
      uint32_t stage_par = 0;
      bool ok = true;
      for (TileCursor c = cursor_begin(); ok && c.left > 0;) {
        const Run run = take_run(c);
        const int tiles = run.tiles;
        if (tiles == 0) continue;
        const int qb = k % nq;
        ok = mbar_wait(&qfull[qb], (uint32_t)(k / nq) & 1u, abort_flag, p.status, kSiteQFull);
        if (!ok) break;
        ++k;
        const uint32_t q_lo0 = q_lo00 + (uint32_t)qb * (128 * 128 >> 4), shift_lo = shift_lo0 + (uint32_t)qb * (128 * 128 >> 4);
        for (int t = 0; t < tiles; ++t, ++n_tile) {
          const int buf = n_tile & 1;
          const uint32_t use_par = (uint32_t)(n_tile >> 1) & 1u;
          ok = mbar_wait(&tempty[buf], use_par ^ 1, abort_flag, p.status, kSiteTEmpty);
          if (!ok) break;
          if (NS == 3) {
            // A stage is one term of 64 columns of the keys, in the order lo, mid, hi of the first 64, then of the others. The
            // accumulation truncates, so the small products come first (lo hi, mid hi, mid mid, hi lo, hi mid) and the 8 or 4
            // steps of hi hi last, for which the stages of hi are held; the second half of those goes to an accumulator of its
            // own, which the epilogue adds. With one accumulator large logits lost more than in the fp32 FMA kernels (8000 keys,
            // 32 heads, head_dim 128: log-sum-exps off by 7.7e-7 rms and -4.8e-7 on average, scores with given ones by 4.9e-7
            // in the 2-norm; FMA 5.1e-7, -1.0e-7 and 4.2e-7; now 4.5e-7, -2.9e-7 and 2.1e-7). us with one / two: 32 units of
            // 8000 keys, head_dim 128 100.9 / 101.2; with given log-sum-exps 80.1 / 80.3; head_dim 64: 16 of 8000 46.2 / 49.2,
            // 1024 of 2357 472 / 527, given 75.1 / 73.3.
            const uint32_t d1 = tmem_base + buf * 256, d2 = d1 + 128;
            auto product = [&](uint32_t k_lo, int qt, int kb, bool first, bool hi_hi) {
#pragma unroll
              for (int kk = 0; kk < 4; ++kk) {
                const int step = kb * 4 + kk, half = D / 32;  // of hi hi
                const uint32_t q_op = q_lo0 + (((qt * kKBlocks + kb) * SL::kQRows * 128 + kk * 32) >> 4);
                const uint32_t k_op = k_lo + ((kk * 32) >> 4), add = (first && kk == 0) || (hi_hi && step == half) ? 0u : 1u;
                const uint32_t d = hi_hi && step >= half ? d2 : d1;
                if (PASS == 1) umma_bf16(d, q_op, k_op, kIdescRows, add);
                else umma_bf16(d, k_op, q_op, idesc2, add);
              }
            };
            uint32_t hi_lo[kKBlocks];
            int hi_stage[kKBlocks];
#pragma unroll
            for (int piece = 0; piece < 3 * kKBlocks; ++piece) {
              const int term = 2 - piece % 3, kb = piece / 3;
              ok = ok && mbar_wait(&full[stage], stage_par, abort_flag, p.status, kSiteFull);
              if (ok) {
                tc_fence_after();
                const uint32_t k_lo = k_lo0 + (uint32_t)stage * (SL::kStageBytes >> 4);
                if (term == 2) {
                  product(k_lo, 0, kb, piece == 0, false);
                } else {
                  product(k_lo, term == 1 ? 0 : 2, kb, false, false);
                  product(k_lo, 1, kb, false, false);
                }
                if (term == 0) {
                  hi_lo[kb] = k_lo;
                  hi_stage[kb] = stage;
                } else {
                  umma_commit(&empty[stage]);  // the K stage may be refilled
                }
                if (++stage == kStages) {
                  stage = 0;
                  stage_par ^= 1;
                }
              }
            }
            if (!ok) break;
#pragma unroll
            for (int kb = 0; kb < kKBlocks; ++kb) {
              product(hi_lo[kb], 0, kb, false, true);
              umma_commit(&empty[hi_stage[kb]]);
            }
            if (PASS == 2) umma_bf16(d2, ones_lo, shift_lo, idesc2, 1u);
          } else {
          const uint32_t k_lo = k_lo0 + (uint32_t)stage * (SL::kStageBytes >> 4);
          ok = mbar_wait(&full[stage], stage_par, abort_flag, p.status, kSiteFull);
          if (!ok) break;
          tc_fence_after();
          if (PASS == 1) {  // D[row, key]: a row block of the queries is operand A, the K tile operand B
            for (int mb = 0; mb < p.mblocks; ++mb) {
              const uint32_t d_tmem = tmem_base + buf * 256 + mb * 128;
#pragma unroll
              for (int ks = 0; ks < D / 16; ++ks) {
                const int kb = ks >> 2, kk = ks & 3;
                umma_bf16(d_tmem, q_lo0 + ((kb * 256 * 128 + mb * 128 * 128 + kk * 32) >> 4),
                          k_lo + ((kb * kTileKeys * 128 + kk * 32) >> 4), kIdescRows, ks > 0 ? 1u : 0u);
              }
            }
          } else {  // D[key, row]: the K tile is operand A, all n16 query rows operand B; then the shift step
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks) {
              const int kb = ks >> 2, kk = ks & 3;
              umma_bf16(tmem_base + buf * 256, k_lo + ((kb * kTileKeys * 128 + kk * 32) >> 4),
                        q_lo0 + ((kb * 256 * 128 + kk * 32) >> 4), idesc2, ks > 0 ? 1u : 0u);
            }
            umma_bf16(tmem_base + buf * 256, ones_lo, shift_lo, idesc2, 1u);
          }
          umma_commit(&empty[stage]);  // the K stage may be refilled
          if (++stage == kStages) {
            stage = 0;
            stage_par ^= 1;
          }
          }
          umma_commit(&tfull[buf]);    // the accumulators are ready
        }
        if (ok) umma_commit(&qempty[qb]);  // the row operands may be replaced once the MMAs issued so far are done
      }
      if (!ok) {  // abandoned: TMEM may only be freed once this thread's MMAs have completed
        umma_commit(drain);
        const long long t0 = clock64();
        while (!mbar_try(drain, 0) && clock64() - t0 < 20000000ll) __nanosleep(200);
      }
    }
  } else if (warp < 2 + SL::kEpiWarps) {
    // ================================================================ epilogue (warps 2-17, with CV 2-5)
    // All of its warps work on the same tile while the MMAs of the next tile fill the other accumulator buffer;
    // warp = (TMEM lane quarter, column share); the TMEM load of a warp's next 16 columns is in flight while it works.
    const int ew = warp - 2;
    const int quarter = warp & 3;  // TMEM lanes [32 * quarter, 32 * quarter + 32)
    // pass 1: (row block mb, column share): two row blocks x 2 shares of 64 keys, or one row block x 4 shares of 32 (CV:
    // one of 128)
    // pass 2: column share = a quarter (CV: all) of the n16 / 16 blocks of window rows (as even as possible)
    const int mb = PASS == 1 && p.mblocks == 2 ? (ew >> 2) & 1 : 0;
    const int share = PASS == 1 ? (p.mblocks == 2 ? ew >> 3 : ew >> 2) : ew >> 2;
    int blk0, nblk;  // this warp's 16-column blocks of a tile's accumulator: blk0 .. blk0 + nblk - 1
    if (PASS == 1) {
      nblk = 8 / p.cparts;
      blk0 = nblk * share;
    } else {
      const int total = p.n16 >> 4, base = total / SL::kShares, rem = total % SL::kShares;
      nblk = base + (share < rem ? 1 : 0);
      blk0 = share * base + min(share, rem);
    }
    const uint32_t tlane = tmem_base + ((uint32_t)(quarter * 32) << 16) + (PASS == 1 ? mb * 128 : 0) + blk0 * 16;
    const uint64_t sc2 = pack2(p.scale2, p.scale2);
    int n_tile = 0;
    bool ok = true;
    // pass 1 state: running maximum and sums of the thread's window row, log2 domain; m starts below any masked
    // logit. The sum is kept on two levels (the item at hand, the run's earlier items): one accumulator over a whole
    // long sequence would lose the small terms to rounding.
    const int row = mb * 128 + quarter * 32 + lane;
    float m = 4.f * kEmptyMax, z_run = 0.f;
    uint64_t zacc[4] = {0ull, 0ull, 0ull, 0ull};  // pass 1: the item's sum, as four packed partial sums
    float* xslot = xch + quarter * 32 + lane;  // pass 2: [buffer][share - 1][128 keys]
    if (PASS == 2 && range_s[0] && !p.accumulate) {  // sequences without keys have no tiles
      for (int b = 0; b < p.B; ++b)
        if (len_s[b] == 0)
          for (int64_t x = ((int64_t)blockIdx.x * SL::kEpiWarps + ew) * 32 + lane; x < (int64_t)p.lh * p.n_max;
               x += (int64_t)gridDim.x * SL::kEpiWarps * 32)
            p.psi[(int64_t)b * p.lh * p.n_max + x] = 0.f;
    }

    for (TileCursor c = cursor_begin(); ok && c.left > 0;) {
      const int run_first = range_s[1] + c.done;  // the run's first tile in the global order
      const Run run = take_run(c);
      const int u = run.u, tiles = run.tiles, key_begin = run.t0 * kTileKeys, n = run.n;
      float* psi = p.psi + (int64_t)u * p.n_max;
      m = 4.f * kEmptyMax;  // pass 1: every run starts its own statistics
      z_run = 0.f;
      zacc[0] = zacc[1] = zacc[2] = zacc[3] = 0ull;
      int vis = 0;  // pass 1: keys the row may see: [0, vis)
      if (PASS == 1 && row < p.R) {
        const int pos = n - p.w + rowpos[row];
        if (pos >= 0) vis = p.causal ? pos + 1 : n;
      }
      for (int t = 0; t < tiles; ++t, ++n_tile) {
        const int buf = n_tile & 1;
        ok = __all_sync(0xffffffffu, mbar_wait(&tfull[buf], (uint32_t)(n_tile >> 1) & 1u, abort_flag, p.status, kSiteTile));
        if (!ok) break;
        tc_fence_after();
        const int key0 = key_begin + t * kTileKeys;
        const uint32_t taddr = tlane + buf * 256;
        uint64_t acc[4] = {0ull, 0ull, 0ull, 0ull};  // pass 2: the key's sum over this warp's window rows
        const int key = key0 + quarter * 32 + lane;  // pass 2: the thread's key
        const bool plain = key0 + kTileKeys <= n - p.w;  // every row sees the whole tile: nothing to mask
        uint32_t ra[16], rb[16];
        auto block = [&](uint32_t (&r)[16], int j) {  // block blk0 + j of the accumulator
          if (PASS == 1) {
            const int col0 = key0 + 16 * (blk0 + j);  // first key of the block
            if (col0 + 16 > vis) {
#pragma unroll
              for (int i = 0; i < 16; ++i)
                if (col0 + i >= vis) r[i] = __float_as_uint(kEmptyMax);
            }
            const float bm = block_max16(r) * p.scale2;
            if (__any_sync(0xffffffffu, bm > m)) {
              const float mn = fmaxf(m, bm);
              const float f = ex2(m - mn);
              const uint64_t f2 = pack2(f, f);
#pragma unroll
              for (int i = 0; i < 4; ++i) zacc[i] = mul2(zacc[i], f2);
              z_run *= f;
              m = mn;
            }
            const uint64_t nm2 = pack2(-m, -m);
            uint64_t x[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) x[i] = fma2(pack2u(r[2 * i], r[2 * i + 1]), sc2, nm2);
            zacc[0] = add2(zacc[0], exp2_sum16(x));
          } else {
            if (!plain) {  // the tiles at the window: every logit is checked against what its row may see
#pragma unroll
              for (int i = 0; i < 16; ++i) {
                const int pos = n - p.w + rowpos[16 * (blk0 + j) + i];
                const int v = pos < 0 ? 0 : (p.causal ? pos + 1 : n);
                if (key >= v) r[i] = __float_as_uint(kEmptyMax);
              }
            }
            uint64_t x[8];  // the accumulator already holds q.k - lse / scale
#pragma unroll
            for (int i = 0; i < 8; ++i) x[i] = mul2(pack2u(r[2 * i], r[2 * i + 1]), sc2);
            acc[0] = add2(acc[0], exp2_sum16(x));
          }
        };
        if (NS == 3) {  // the two accumulators' sum, block by block (loads of the next block under the work on this one: the
                        // registers do not suffice, 527 -> 675 us on 1024 units of 2357 keys, head_dim 64)
#pragma unroll 1
          for (int j = 0; j < nblk; ++j) {
            tmem_ld16_issue(taddr + j * 16, ra);
            tmem_ld16_issue(taddr + 128 + j * 16, rb);
            tmem_ld_wait16(ra);
            tmem_ld_tie16(rb);
#pragma unroll
            for (int i = 0; i < 16; ++i) ra[i] = __float_as_uint(__uint_as_float(ra[i]) + __uint_as_float(rb[i]));
            block(ra, j);
          }
        } else if (plain) {  // all but the tiles at the window
          if (PASS == 1) {
            if (SL::kShares == 1) stat_tile<8>(taddr, p.scale2, sc2, m, zacc, z_run);
            else if (nblk == 4) stat_tile<4>(taddr, p.scale2, sc2, m, zacc, z_run);
            else stat_tile<2>(taddr, p.scale2, sc2, m, zacc, z_run);
          } else {
            switch (nblk) {
              case 8: if (SL::kShares == 1) psi_tile<8>(taddr, sc2, acc); break;
              case 7: if (SL::kShares == 1) psi_tile<7>(taddr, sc2, acc); break;
              case 6: if (SL::kShares == 1) psi_tile<6>(taddr, sc2, acc); break;
              case 5: if (SL::kShares == 1) psi_tile<5>(taddr, sc2, acc); break;
              case 4: psi_tile<4>(taddr, sc2, acc); break;
              case 3: psi_tile<3>(taddr, sc2, acc); break;
              case 2: psi_tile<2>(taddr, sc2, acc); break;
              case 1: psi_tile<1>(taddr, sc2, acc); break;
              default: break;
            }
          }
        } else if (nblk > 0) {
          tmem_ld16_issue(taddr, ra);
#pragma unroll 1
          for (int j = 0; j < nblk; j += 2) {
            tmem_ld_wait16(ra);
            if (j + 1 < nblk) tmem_ld16_issue(taddr + (j + 1) * 16, rb);
            block(ra, j);
            if (j + 1 < nblk) {
              tmem_ld_wait16(rb);
              if (j + 2 < nblk) tmem_ld16_issue(taddr + (j + 2) * 16, ra);
              block(rb, j + 1);
            }
          }
        }
        tc_fence_before();
        mbar_arrive(&tempty[buf]);
        if (PASS == 1 && (t % kFoldTiles) == kFoldTiles - 1) {  // second level of the row's sum
          z_run += sum4(zacc);
          zacc[0] = zacc[1] = zacc[2] = zacc[3] = 0ull;
        }
        if (PASS == 2) {
          // the warps that share the key add up in a fixed order: shares 1-3 hand their sums to share 0 (a
          // slot is free once share 0 has taken the tile before last)
          float total = sum4(acc);
          const uint32_t xp = (uint32_t)(n_tile >> 1) & 1u;
          if (SL::kShares == 1) {
            if (key < p.n_max) psi[key] = key < n ? (p.accumulate ? psi[key] + total : total) : 0.f;
          } else if (share) {
            ok = __all_sync(0xffffffffu, mbar_wait(&xempty[buf * 4 + quarter], xp ^ 1, abort_flag, p.status, kSiteFlag));
            if (!ok) break;
            xslot[(buf * (SL::kShares - 1) + share - 1) * 128] = total;
            mbar_arrive(&xfull[buf * 4 + quarter]);
          } else {
            ok = __all_sync(0xffffffffu, mbar_wait(&xfull[buf * 4 + quarter], xp, abort_flag, p.status, kSiteFlag));
            if (!ok) break;
#pragma unroll
            for (int x = 0; x < SL::kShares - 1; ++x) total += xslot[(buf * (SL::kShares - 1) + x) * 128];
            mbar_arrive(&xempty[buf * 4 + quarter]);
            if (key < p.n_max) psi[key] = key < n ? (p.accumulate ? psi[key] + total : total) : 0.f;
          }
        }
      }
      if (PASS == 2 && ok && !p.accumulate && run.t0 + run.cnt >= (n + kTileKeys - 1) / kTileKeys) {
        // the keys no tile covers, by the CTA that has the unit's last tile
        for (int key = (n + kTileKeys - 1) / kTileKeys * kTileKeys + ew * 32 + lane; key < p.n_max; key += SL::kEpiWarps * 32)
          psi[key] = 0.f;
      }
      if (!ok) break;
      if (PASS == 1) {
        z_run += sum4(zacc);
        if (row < p.R) {
          // one pair per run: slot = this CTA's place among the CTAs that the unit's tiles are spread over (the merge
          // kernel walks the same partition). A row that saw no visible key only summed masked entries: it is
          // recorded as empty, and so is a run without keys (the uniform partition of very large batches has those).
          const int k = range_s[4] ? (int)blockIdx.x - p.by_per.div(blockIdx.x) * p.per : run.t0 ? (int)blockIdx.x - cta_of(range_s[2], range_s[3], run_first - run.t0) : 0;
          const bool none = tiles == 0 || m < 0.5f * kEmptyMax * p.scale2;
          if (k >= 0 && k < p.smax)
            p.part[(((int64_t)u * p.smax + k) * p.cparts + share) * p.rs + row] =
                none ? make_float2(kEmptyMax, 0.f) : make_float2(m, z_run);
          else
            set_status(p.status, MADAKV_ESHAPE);  // cannot happen: smax bounds the runs of a unit
        }
      }
    }
  }
  if constexpr (CV) {
    if (warp >= 2 + SL::kEpiWarps) {
      // ============================================================== converters (CV): a step is 64 columns of the 128 keys of
      // a tile; half a warp reads the 256 bytes of a row, and each thread turns 8 x 4 values into three terms each, written as
      // three stages. The next step's values are on their way to registers meanwhile, those of two steps later to the L2.
      const int cw = warp - 2 - SL::kEpiWarps, sub = lane >> 4, c4 = (lane & 15) * 4;  // rows kStep * i + 2 * cw + sub, columns c4 .. c4 + 3
      const int r0 = 2 * cw + sub;
      constexpr int kStep = 2 * kConvertWarps, kRep = kTileKeys / kStep;  // rows per load of all warps, loads per thread and step
      auto place = [&](int r) { return r * 128 + (((lane & 15) >> 1) ^ (r & 7)) * 16 + (lane & 1) * 8; };  // in a piece
      int stage = 0, k = 0;
      uint32_t stage_par = 0;
      bool ok = true;
      for (TileCursor c = cursor_begin(); ok && c.left > 0;) {
        const Run run = take_run(c);
        if (run.tiles == 0) continue;
        const int h = run.h, l = run.l, b = run.b, n = run.n;
        const float* kf = p.kf + b * p.sk.batch + l * p.sk.layer + h * p.sk.head;
        const float* qf = p.qf + b * p.sq.batch + l * p.sq.layer + (int64_t)(h * p.g + p.h0) * p.sq.head;
        const int steps = run.tiles * kKBlocks;
        float4 next[kRep];
        auto load = [&](int step) {
          const int key0 = (run.t0 + step / kKBlocks) * kTileKeys + r0;
          const float* src = kf + (step % kKBlocks) * 64 + c4;
#pragma unroll
          for (int i = 0; i < kRep; ++i)
            next[i] = key0 + kStep * i < n ? load4(src + (int64_t)(key0 + kStep * i) * p.sk.token)
                                        : make_float4(0.f, 0.f, 0.f, 0.f);
        };
        auto prefetch = [&](int step) {  // 2 x 128 bytes of each of the 128 rows, one per thread
          const int x = cw * 32 + lane, key = (run.t0 + step / kKBlocks) * kTileKeys + (x >> 1);
          if (x < 256 && step < steps && key < n)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(kf + (int64_t)key * p.sk.token + (step % kKBlocks) * 64 + (x & 1) * 32));
        };
        load(0);
        // the unit's queries
        float4 qv[kKBlocks][kRep];
#pragma unroll
        for (int kb = 0; kb < kKBlocks; ++kb)
#pragma unroll
          for (int i = 0; i < kRep; ++i) {
            const int r = r0 + kStep * i;
            qv[kb][i] = r < p.R ? load4(qf + rowhead[r] * p.sq.head + rowpos[r] * p.sq.token + kb * 64 + c4) : make_float4(0.f, 0.f, 0.f, 0.f);
          }
        prefetch(1);
        prefetch(2);
        ok = __all_sync(0xffffffffu, mbar_wait(&qempty[0], ((uint32_t)k & 1u) ^ 1u, abort_flag, p.status, kSiteQEmpty));
        if (!ok) break;
        ++k;
#pragma unroll
        for (int kb = 0; kb < kKBlocks; ++kb)
#pragma unroll
          for (int i = 0; i < kRep; ++i) {
            uint8_t* to = q_s + kb * SL::kQRows * 128 + place(r0 + kStep * i);
            constexpr int kTerm = kKBlocks * SL::kQRows * 128;
            const uint4 t = split4(qv[kb][i], [&](uint2 lo) { *reinterpret_cast<uint2*>(to + 2 * kTerm) = lo; });
            *reinterpret_cast<uint2*>(to + kTerm) = make_uint2(t.z, t.w);
            *reinterpret_cast<uint2*>(to) = make_uint2(t.x, t.y);
          }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&qfull[0]);
        // its keys
        auto take_stage = [&]() {
          ok = __all_sync(0xffffffffu, mbar_wait(&empty[stage], stage_par ^ 1u, abort_flag, p.status, kSiteStage));
          return k_s + stage * SL::kStageBytes;
        };
        auto give_stage = [&]() {
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(&full[stage]);
          if (++stage == kStages) {
            stage = 0;
            stage_par ^= 1;
          }
        };
#pragma unroll 1
        for (int step = 0; step < steps; ++step) {
          uint4 t[kRep];  // hi and mid of four values each, packed
          uint8_t* to = take_stage();
          if (!ok) break;
#pragma unroll
          for (int i = 0; i < kRep; ++i)
            t[i] = split4(next[i], [&](uint2 lo) { *reinterpret_cast<uint2*>(to + place(r0 + kStep * i)) = lo; });
          give_stage();
          if (step + 1 < steps) load(step + 1);
          prefetch(step + 3);
          const int s1 = stage, s2 = stage + 1 == kStages ? 0 : stage + 1;
          const uint32_t par2 = s2 ? stage_par : stage_par ^ 1u;
          const bool free = mbar_wait(&empty[s1], stage_par ^ 1u, abort_flag, p.status, kSiteStage) &&
                            mbar_wait(&empty[s2], par2 ^ 1u, abort_flag, p.status, kSiteStage);
          ok = __all_sync(0xffffffffu, free);
          if (!ok) break;
#pragma unroll
          for (int i = 0; i < kRep; ++i) {
            const int at = place(r0 + kStep * i);
            *reinterpret_cast<uint2*>(k_s + s1 * SL::kStageBytes + at) = make_uint2(t[i].z, t[i].w);
            *reinterpret_cast<uint2*>(k_s + s2 * SL::kStageBytes + at) = make_uint2(t[i].x, t[i].y);
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane < 2) mbar_arrive(&full[lane ? s2 : s1]);
          stage = s2 + 1 == kStages ? 0 : s2 + 1;
          stage_par = s2 + 1 == kStages ? par2 ^ 1u : par2;
        }
      }
    }
  }

  // ---- teardown
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
  }
}

// merge: per (unit, row) the (max, sum) pairs of all runs and column shares, in a fixed order -> log2-domain log-sum-exp,
// stored negated (pass 2 adds it inside the contraction); padding rows get a shift that turns every weight into 0. A block
// takes 32 rows of one unit, eight threads per row: a call's only unit can be spread over all CTAs (one thread per row took 53 us
// for 300 pairs).
__global__ void __launch_bounds__(256) score_rows_merge_kernel(RowParams p, float* nlse2, float* lse_out) {
  __shared__ float s_m[8][32], s_z[8][32];
  __shared__ int s_entries;
  const int blocks = p.rs / 32, u = blockIdx.x / blocks, lane = threadIdx.x & 31, part_i = threadIdx.x >> 5;
  const int row = blockIdx.x % blocks * 32 + lane;
  pdl_wait();
  pdl_go();
  if (threadIdx.x == 0) {
    // the CTAs of pass 1 that the unit's tiles were spread over: the same partition as in the kernel
    const int b = u / p.lh;
    const bool exact = p.B <= kMaxSeqScan;
    auto seq_tiles = [&](int b2) { return ((exact ? clamped_len(p.seq_len, b2, p.n_max) : p.n_max) + kTileKeys - 1) / kTileKeys; };
    const Partition x = partition_of(p, exact, seq_tiles);
    const int tb = seq_tiles(b);
    int first = 0;  // the unit's first tile in the global order
    if (exact) {
      for (int b2 = 0; b2 < b; ++b2) first += p.lh * seq_tiles(b2);
    } else {
      first = b * p.lh * tb;
    }
    first += (u - b * p.lh) * tb;
    s_entries = 0;
    if (tb > 0)
      s_entries = p.cparts * min(p.smax, x.per ? min(x.per, tb) : cta_of(x.total, x.ctas, first + tb - 1) - cta_of(x.total, x.ctas, first) + 1);
  }
  __syncthreads();
  const int entries = s_entries;
  const float2* part = p.part + (int64_t)u * p.cparts * p.smax * p.rs + row;
  float M = kEmptyMax, Z = 0.f;
  for (int s0 = part_i; s0 < entries; s0 += 32) {
    float2 v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = s0 + 8 * j < entries ? part[(int64_t)(s0 + 8 * j) * p.rs] : make_float2(kEmptyMax, 0.f);
    const float mn = fmaxf(fmaxf(fmaxf(v[0].x, v[1].x), fmaxf(v[2].x, v[3].x)), M);
    Z *= exp2f(M - mn);
#pragma unroll
    for (int j = 0; j < 4; ++j) Z += v[j].y * exp2f(v[j].x - mn);  // an empty pair has sum 0
    M = mn;
  }
  s_m[part_i][lane] = M;
  s_z[part_i][lane] = Z;
  __syncthreads();
  if (part_i) return;
  const int64_t x = (int64_t)u * p.rs + row;
  if (row >= p.R) {
    nlse2[x] = kEmptyMax;
    return;
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) M = fmaxf(M, s_m[j][lane]);
  Z = 0.f;
#pragma unroll
  for (int j = 0; j < 8; ++j) Z += s_z[j][lane] * exp2f(s_m[j][lane] - M);
  // (the sum's exponent apart and the additions in 64 bits: M + log2f(Z) in 32 is off by up to 2^-20)
  int e = 0;
  const float f = Z > 0.f ? frexpf(Z, &e) : 1.f;
  const double l2 = Z > 0.f ? (double)M + (double)e + (double)log2f(f) : 0.0;
  nlse2[x] = (float)-l2;
  if (lse_out) {
    const int h = u % p.Hkv, bl = u / p.Hkv;
    const int hq = h * p.g + p.h0 + row / p.wc, wr = p.r0 + row % p.wc;
    lse_out[((int64_t)bl * p.Hq + hq) * p.w + wr] = Z > 0.f ? (float)(l2 * 0.6931471805599453) : -INFINITY;
  }
}

template <int D, int PASS, int NS, bool CV>
int launch_pass(const CUtensorMap& mk, const CUtensorMap& mq, const RowParams& p, int grid, cudaStream_t st) {
  using SL = RowSmem<D, PASS, NS, CV>;
  if (cudaFuncSetAttribute(score_rows_kernel<D, PASS, NS, CV>, cudaFuncAttributeMaxDynamicSharedMemorySize, SL::kAlloc) !=
      cudaSuccess)
    return MADAKV_ECUDA;
  launch_pdl(score_rows_kernel<D, PASS, NS, CV>, dim3(grid), dim3(SL::kThreads), (size_t)SL::kAlloc, st, mk, mq, p);
  return MADAKV_OK;
}
template <int PASS>
int launch_pass(const madakv_config& c, bool convert, const CUtensorMap& mk, const CUtensorMap& mq, const RowParams& p, int grid, cudaStream_t st) {
  const bool wide = c.head_dim == 128;
  if (c.dtype != MADAKV_F32)
    return wide ? launch_pass<128, PASS, 1, false>(mk, mq, p, grid, st) : launch_pass<64, PASS, 1, false>(mk, mq, p, grid, st);
  if (convert)
    return wide ? launch_pass<128, PASS, 3, true>(mk, mq, p, grid, st) : launch_pass<64, PASS, 3, true>(mk, mq, p, grid, st);
  return wide ? launch_pass<128, PASS, 3, false>(mk, mq, p, grid, st) : launch_pass<64, PASS, 3, false>(mk, mq, p, grid, st);
}

// ---- fp32 operands -> three bf16 terms each, whose sum is the operand exactly (8 significand bits per term)
struct SplitParams {
  const float* src;
  __nv_bfloat16* dst;  // [rows][3][D]
  const int32_t* seq_len;
  madakv_strides s;    // of src, in elements
  int L, H, D, tokens;  // seq_len: nullptr = all tokens
};
// (blocks: first the keys' heads, k_blocks each, then the queries')
__global__ void __launch_bounds__(256) split_kernel(SplitParams pk, SplitParams pq, int k_heads, int k_blocks, int q_blocks) {
  pdl_wait();
  pdl_go();
  int bx = (int)blockIdx.x;
  const bool is_q = bx >= k_heads * k_blocks;
  if (is_q) bx -= k_heads * k_blocks;
  const SplitParams& p = is_q ? pq : pk;
  const int per = is_q ? q_blocks : k_blocks, y = bx / per;
  const int lg = p.D == 128 ? 5 : 4;  // 16-byte pieces per row: 32 or 16
  const int x = (bx - y * per) * 256 + threadIdx.x, tok = x >> lg, c = (x & ((1 << lg) - 1)) * 4;
  const int h = y % p.H, l = y / p.H % p.L, b = y / (p.H * p.L);
  if (tok >= (p.seq_len ? clamped_len(p.seq_len, b, p.tokens) : p.tokens)) return;  // (keys beyond the sequence are masked)
  const int64_t row = (int64_t)y * p.tokens + tok;
  const float4 v = __ldg(reinterpret_cast<const float4*>(p.src + b * p.s.batch + l * p.s.layer + h * p.s.head + tok * p.s.token + c));
  __nv_bfloat16* dst = p.dst + row * 3 * p.D + c;
  const uint4 t = split4(v, [&](uint2 lo) { *reinterpret_cast<uint2*>(dst + 2 * p.D) = lo; });
  *reinterpret_cast<uint2*>(dst + p.D) = make_uint2(t.z, t.w);
  *reinterpret_cast<uint2*>(dst) = make_uint2(t.x, t.y);
}

// Window rows chunk by chunk. given_lse: single pass with supplied log-sum-exps.
int score_rows(const madakv_config& c, const void* q, madakv_strides sq, const void* k, madakv_strides sk, const int32_t* seq_len,
               const float* given_lse, float* lse, float* psi, void* ws, cudaStream_t st) {
  const WsLayout wl = ws_layout(c);
  const bool f32 = c.dtype == MADAKV_F32;
  const int g = c.n_q_heads / c.n_kv_heads, d = c.head_dim;
  RowParams p;
  p.seq_len = seq_len;
  p.psi = psi;
  p.part = reinterpret_cast<float2*>((char*)ws + wl.score_part_off);
  float* lse2 = reinterpret_cast<float*>((char*)ws + wl.score_lse_off);
  p.lse2 = lse2;
  p.status = reinterpret_cast<int32_t*>(ws);
  p.B = c.batch;
  p.lh = c.n_layers * c.n_kv_heads;
  p.units = c.batch * p.lh;
  p.qf = static_cast<const float*>(q);
  p.kf = static_cast<const float*>(k);
  p.sq = sq;
  p.sk = sk;
  p.L = c.n_layers;
  p.Hq = c.n_q_heads;
  p.Hkv = c.n_kv_heads;
  p.g = g;
  p.w = c.window;
  p.n_max = c.max_seq_len;
  p.causal = c.causal;
  p.smax = wide_max_runs(p.lh, c.max_seq_len);
  p.scale2 = scale_of(c) * kLog2e;
  p.inv = 1.0f / p.scale2;
  p.inv_more = f32 || !given_lse ? (float)(1.0 / (double)p.scale2 - (double)p.inv) : 0.f;
  p.by_hkv = FastDiv(c.n_kv_heads);
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return MADAKV_ECUDA;
  const long long tiles = (long long)p.units * ((c.max_seq_len + kTileKeys - 1) / kTileKeys);
  if (tiles > 0x3fffffff) return MADAKV_EUNSUPPORTED;
  if (sms > kWideMaxGrid) sms = kWideMaxGrid;
  const int grid = (int)(tiles < sms ? tiles : sms);
  p.grid = grid;
  p.per = grid / p.units;
  p.by_grid = FastDiv(grid);
  p.by_per = FastDiv(p.per > 0 ? p.per : 1);
  const bool convert = f32 && (given_lse || !split_first(c));
  CUtensorMap mk = {}, mq = {};  // (convert: not used)
  const madakv_strides split_k{0, 0, (int64_t)c.max_seq_len * 3 * d, 3 * d}, split_q{0, 0, (int64_t)c.window * 3 * d, 3 * d};
  if (f32 && !convert) {
    __nv_bfloat16* ks = reinterpret_cast<__nv_bfloat16*>((char*)ws + wl.score_split_off);
    __nv_bfloat16* qs = ks + (int64_t)p.units * c.max_seq_len * 3 * d;
    if (!make_map(&mk, ks, 3 * d, c.max_seq_len, p.units, 1, 1, split_k, kTileKeys, 1)) return MADAKV_EUNSUPPORTED;
    SplitParams x{(const float*)k, ks, seq_len, sk, c.n_layers, c.n_kv_heads, d, c.max_seq_len};
    SplitParams y{(const float*)q, qs, nullptr, sq, c.n_layers, c.n_q_heads, d, c.window};
    const int kb = (c.max_seq_len * (d / 4) + 255) / 256, qb = (c.window * (d / 4) + 255) / 256;
    launch_pdl(split_kernel, dim3((unsigned)(p.units * (kb + g * qb))), dim3(256), 0, st, x, y, p.units, kb, qb);
    q = qs;
  } else if (!f32 && !make_map(&mk, k, d, c.max_seq_len, c.n_kv_heads, c.n_layers, c.batch, sk, kTileKeys, 1)) {
    return MADAKV_EUNSUPPORTED;
  }
  const int rows_max = f32 ? 128 : 256;
  // chunks of equal size as far as possible (7 heads of 64 rows: 4 + 3)
  const int heads_max = c.window < rows_max ? rows_max / c.window : 1, head_chunks = (g + heads_max - 1) / heads_max;
  const int row_chunks = (c.window + rows_max - 1) / rows_max;
  const int hc = (g + head_chunks - 1) / head_chunks, rc = (c.window + row_chunks - 1) / row_chunks;
  p.accumulate = 0;
  for (p.h0 = 0; p.h0 < g; p.h0 += hc)
    for (p.r0 = 0; p.r0 < c.window; p.r0 += rc) {
      const int heads = g - p.h0 < hc ? g - p.h0 : hc;
      p.wc = c.window - p.r0 < rc ? c.window - p.r0 : rc;
      p.R = heads * p.wc;
      p.by_wc = FastDiv(p.wc);
      p.rs = (p.R + 31) / 32 * 32;  // row stride of the workspace arrays
      p.mblocks = p.R <= 128 ? 1 : 2;
      p.cparts = convert ? 1 : (p.R <= 128 ? 4 : 2);
      p.n16 = (p.R + 15) / 16 * 16;
      // (bf16 rows beyond 128 have one buffer, and a change of units costs two or three tiles' time; fp32 has one, too, but its tiles
      // take several times as long: 60 units of 24 tiles, 32 rows, 84.0 us with CTAs of two tiles more, 77.1 without; 40 of
      // 16 51.3 and 49.4; 20 of 71 78.9 and 77.1)
      p.slack = !f32 && p.R > 128 ? 2 : 0;
      if (!convert && !(f32 ? make_map(&mq, q, 3 * d, c.window, p.units * g, 1, 1, split_q, p.wc, heads)
                            : make_map(&mq, q, d, c.window, c.n_q_heads, c.n_layers, c.batch, sq, p.wc, heads)))
        return MADAKV_EUNSUPPORTED;
      p.given_lse = given_lse;
      int rc2;
      if (!given_lse) {
        if ((rc2 = launch_pass<1>(c, convert, mk, mq, p, grid, st))) return rc2;
        launch_pdl(score_rows_merge_kernel, dim3(p.units * (p.rs / 32)), dim3(256), 0, st, p, lse2, lse);
      }
      if ((rc2 = launch_pass<2>(c, convert, mk, mq, p, grid, st))) return rc2;
      p.accumulate = 1;
    }
  return launch_status();
}

}  // namespace

int launch_score_rows(const madakv_config& c, const void* q, madakv_strides sq, const void* k, madakv_strides sk,
                      const int32_t* seq_len, float* lse, float* psi, void* ws, cudaStream_t st) {
  return score_rows(c, q, sq, k, sk, seq_len, nullptr, lse, psi, ws, st);
}

// Single-pass scoring with the rows' log-sum-exps supplied by the caller: pass 2 alone.
int launch_score_lse_rows(const madakv_config& c, const void* q, madakv_strides sq, const void* k, madakv_strides sk,
                          const int32_t* seq_len, const float* lse, float* psi, void* ws, cudaStream_t st) {
  return score_rows(c, q, sq, k, sk, seq_len, lse, nullptr, psi, ws, st);
}

}  // namespace madakv
