// Stage 5: cache append (Eq. 4) and decode attention over the ragged per-head cache (Eq. 5), one launch per call.
//
//   append   (Eq. 4) has no kernel of its own: the block whose share holds the new row copies it from k_new / v_new
//            behind the segment and attends over it; the block that merges the segment bumps kept_len
//   attend   a segment's rows are shared out over up to `slots` blocks (decode_shape). Scalar kernel: a group of LPR lanes owns
//            a cache row (16 bytes per lane), the g query heads of the KV group share every K/V row read; online
//            softmax in the log2 domain, fp32 accumulation; the block's row groups are merged in shared memory. For bf16
//            caches with 3 <= g <= 16 the same share is computed by decode_mma_kernel on the tensor cores instead.
//   merge    the block that arrives last at the segment's counter combines the blocks' results in block order and rounds
//            to dtype once. (A second kernel for it cost a launch on the host, 2.2 us, and 3-9 us on the GPU per call; a
//            thread-block cluster per segment that merges through distributed shared memory left too few blocks
//            resident: 248 us instead of 148 on 1024 segments of 1638 rows.)
#include <mutex>
#include <type_traits>

#include "common.cuh"

namespace madakv {
namespace {

constexpr int NT = 128;
constexpr int kDecodeSlots = 32;    // blocks per segment at most

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

struct DecodeParams {
  const void* q;
  const void* k_new;
  const void* v_new;
  void* k_c;
  void* v_c;
  const int64_t* seg_off;
  int32_t* kept_len;
  int64_t capacity;
  void* out;
  float* lse_out;
  float* part;        // slots > 1: [B*L*Hq, slots, D] partial outputs, then [B*L*Hq, slots, 2] their (max, sum)
  float2* part_ml;
  unsigned* counter;  // slots > 1: one per segment of the call, zero when it begins and when it ends
  void* ws;
  int L, Hq, Hkv, g, layer, slots, n_sel, min_rows;
  float scale2;
  int hold_copies;        // test of waits that run out: no row is copied
  long long wait_clocks;  // bound of a wait for a copy
};

__device__ __forceinline__ float fast_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ int unit_of(const DecodeParams& p, int y) {
  // y enumerates the (sequence, KV head) pairs of the selected layer, or all units when layer < 0
  if (p.layer < 0) return y;
  const int b = y / p.Hkv, h = y % p.Hkv;
  return (b * p.L + p.layer) * p.Hkv + h;
}

// Rows of unit u's segment that attention may read. A segment that selection refused (it, with its headroom, ends
// beyond the cache: MADAKV_ECAPACITY was reported and neither indices nor rows were written) counts as empty, and so
// does one whose length does not fit its own slot: nothing beyond `capacity` rows is ever touched.
__device__ __forceinline__ bool segment_refused(const DecodeParams& p, int u) {
  const int64_t off = p.seg_off[u], end = p.seg_off[u + 1];
  return off < 0 || end < off || end > p.capacity;
}
__device__ __forceinline__ int segment_rows(const DecodeParams& p, int u) {
  const int len = p.kept_len[u];
  if (segment_refused(p, u) || len < 0 || p.seg_off[u] + (int64_t)len > p.seg_off[u + 1]) return 0;
  return len;
}
// The blocks of a segment of `len` rows: how many take part, and the rows of block x (a multiple of 16 each, so
// that the 16-row chunks of the warps never straddle two blocks). Block 0 always takes part: an empty segment still
// gets a well-defined partial.
__device__ __forceinline__ int segment_blocks(const DecodeParams& p, int len) {
  return max(1, min(p.slots, (len + p.min_rows - 1) / p.min_rows));
}
__device__ __forceinline__ void block_rows(int nb, int len, int x, int& row_begin, int& row_end) {
  const int share = ((len + nb - 1) / nb + 15) / 16 * 16;
  row_begin = min(len, x * share);
  row_end = min(len, row_begin + share);
}

// What a block of unit u works on. When the call appends (Eq. 4), the new row is part of the attention: the one block
// whose share holds it copies it from k_new / v_new into the cache and reads it from there, all others see the old
// rows only. kept_len itself is bumped by the block that merges, after every block of the segment has read the old value.
// A segment without room for the row (or one that selection refused) is left as it is and MADAKV_ECAPACITY is recorded.
struct SegView {
  int len;      // rows attention covers, the appended one included
  int new_row;  // its index in the segment, or -1
};
__device__ __forceinline__ SegView segment_view(const DecodeParams& p, int u, bool reporter) {
  SegView v;
  v.len = segment_rows(p, u);
  v.new_row = -1;
  if (p.k_new) {
    const int len = p.kept_len[u];
    if (segment_refused(p, u) || len < 0 || p.seg_off[u] + (int64_t)len + 1 > p.seg_off[u + 1]) {
      if (reporter) set_status(p.ws, MADAKV_ECAPACITY);
    } else {
      v.new_row = len;
      v.len = len + 1;
    }
  }
  return v;
}
// The owner of the appended row (the block whose rows include it) stores it into the cache.
template <int ROW_BYTES>
__device__ __forceinline__ void store_new_row(const DecodeParams& p, int u, int64_t off, const SegView& v, int row_begin,
                                              int row_end) {
  constexpr int LPR = ROW_BYTES / 16;
  if (v.new_row < row_begin || v.new_row >= row_end || (int)threadIdx.x >= LPR) return;
  const int64_t row = off + v.new_row;
  const uint4 kv = *reinterpret_cast<const uint4*>((const char*)p.k_new + (int64_t)u * ROW_BYTES + threadIdx.x * 16);
  const uint4 vv = *reinterpret_cast<const uint4*>((const char*)p.v_new + (int64_t)u * ROW_BYTES + threadIdx.x * 16);
  *reinterpret_cast<uint4*>((char*)p.k_c + row * ROW_BYTES + threadIdx.x * 16) = kv;
  *reinterpret_cast<uint4*>((char*)p.v_c + row * ROW_BYTES + threadIdx.x * 16) = vv;
}

template <typename T>
struct Vec16;
template <>
struct Vec16<float> {
  static constexpr int N = 4;
  __device__ static void load(const void* p, float* f) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w;
  }
  __device__ static void cvt(const uint4& v, float* f) {
    f[0] = __uint_as_float(v.x); f[1] = __uint_as_float(v.y); f[2] = __uint_as_float(v.z); f[3] = __uint_as_float(v.w);
  }
};
template <>
struct Vec16<__nv_bfloat16> {
  static constexpr int N = 8;
  __device__ static void load(const void* p, float* f) {
    const uint4 v = *reinterpret_cast<const uint4*>(p);
    f[0] = bf16_lo(v.x); f[1] = bf16_hi(v.x); f[2] = bf16_lo(v.y); f[3] = bf16_hi(v.y);
    f[4] = bf16_lo(v.z); f[5] = bf16_hi(v.z); f[6] = bf16_lo(v.w); f[7] = bf16_hi(v.w);
  }
  __device__ static void cvt(const uint4& v, float* f) {
    f[0] = bf16_lo(v.x); f[1] = bf16_hi(v.x); f[2] = bf16_lo(v.y); f[3] = bf16_hi(v.y);
    f[4] = bf16_lo(v.z); f[5] = bf16_hi(v.z); f[6] = bf16_lo(v.w); f[7] = bf16_hi(v.w);
  }
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// The weight of a partial with maximum m against the overall maximum M.
__device__ __forceinline__ float part_weight(float m, float M) { return m == -INFINITY ? 0.f : exp2f(m - M); }

constexpr float kLost = -1.f;  // in the place of a sum of weights: a wait for the rows ran out
// Four results of one query head: `o` unnormalised, l their sum of weights.
template <typename T, int D>
__device__ __forceinline__ void store4(const DecodeParams& p, int64_t row, int c, float4 o, float l) {
  const float none = l < 0.f ? NAN : 0.f;
  const float r0 = l > 0.f ? o.x / l : none, r1 = l > 0.f ? o.y / l : none, r2 = l > 0.f ? o.z / l : none, r3 = l > 0.f ? o.w / l : none;
  if constexpr (sizeof(T) == 4) {
    *reinterpret_cast<float4*>(reinterpret_cast<float*>(p.out) + row * D + c) = make_float4(r0, r1, r2, r3);
  } else {
    const __nv_bfloat162 a = __floats2bfloat162_rn(r0, r1), b = __floats2bfloat162_rn(r2, r3);
    *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(p.out) + row * D + c) =
        make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
  }
}
__device__ __forceinline__ void store_lse(const DecodeParams& p, int64_t row, float M, float l) {
  if (p.lse_out) p.lse_out[row] = l > 0.f ? (M + log2f(l)) * kLn2 : (l < 0.f ? NAN : -INFINITY);
}

// The end of a block: its results lie in shared memory (bo [g][D] unnormalised, bm and bl [g], complete behind a barrier of
// the block); they are combined with those of the segment's other blocks, in block order. fac: kDecodeSlots * g floats of
// shared memory. `nb` blocks of the segment have results; the others arrive at the counter all the same, so that the last
// one knows that all have read the segment's length.
template <typename T, int D, int NTHR>
__device__ __forceinline__ void finish_segment(const DecodeParams& p, const float* bo, const float* bm, const float* bl, float* fac,
                                               int u, int y, int slot, int nb, SegView view) {
  constexpr int C4 = D / 4;
  const int h = u % p.Hkv, blr = u / p.Hkv;
  const int64_t row0 = (int64_t)blr * p.Hq + h * p.g;
  if (p.slots == 1) {
    for (int x = threadIdx.x; x < p.g * C4; x += NTHR) {
      const int i = x / C4, c = x % C4 * 4;
      store4<T, D>(p, row0 + i, c, *reinterpret_cast<const float4*>(bo + i * D + c), bl[i]);
      if (c == 0) store_lse(p, row0 + i, bm[i], bl[i]);
    }
    if (threadIdx.x == 0 && view.new_row >= 0) p.kept_len[u] = view.len;
    return;
  }
  if (slot < nb) {
    for (int x = threadIdx.x; x < p.g * C4; x += NTHR) {
      const int i = x / C4, c = x % C4 * 4;
      __stcg(reinterpret_cast<float4*>(p.part + ((row0 + i) * p.slots + slot) * D + c),
             *reinterpret_cast<const float4*>(bo + i * D + c));
    }
    if ((int)threadIdx.x < p.g) __stcg(p.part_ml + (row0 + threadIdx.x) * p.slots + slot, make_float2(bm[threadIdx.x], bl[threadIdx.x]));
  }
  __shared__ unsigned s_last;
  __syncthreads();
  if (threadIdx.x == 0) s_last = arrive_inc(p.counter + y, (unsigned)p.slots - 1u);  // (wraps to 0: ready for the next call)
  __syncthreads();
  if (s_last != (unsigned)p.slots - 1u) return;
  if (threadIdx.x == 0 && view.new_row >= 0) p.kept_len[u] = view.len;
  // weights of the partials, and every head's maximum and sum; the first partials are on their way meanwhile
  __shared__ float s_l[16];
  constexpr int kFirst = 8, kHeads = 16 * 32 / NTHR;  // heads per warp at most
  float2 ml[kHeads];
#pragma unroll
  for (int j = 0; j < kHeads; ++j) {
    const int i = (int)threadIdx.x / 32 + j * (NTHR / 32), s = threadIdx.x % 32;
    ml[j] = i < p.g && s < nb ? __ldcg(p.part_ml + (row0 + i) * p.slots + s) : make_float2(-INFINITY, 0.f);
  }
  float4 v[kFirst];
  auto load_parts = [&](int x, int s0) {
    const float4* src = reinterpret_cast<const float4*>(p.part + (row0 + x / C4) * p.slots * D + x % C4 * 4);
#pragma unroll
    for (int s = 0; s < kFirst; ++s) v[s] = s0 + s < nb ? __ldcg(src + (s0 + s) * C4) : make_float4(0.f, 0.f, 0.f, 0.f);
  };
  if ((int)threadIdx.x < p.g * C4) load_parts(threadIdx.x, 0);
#pragma unroll
  for (int j = 0; j < kHeads; ++j) {
    const int i = (int)threadIdx.x / 32 + j * (NTHR / 32), s = threadIdx.x % 32;
    if (i >= p.g) break;
    const float m = ml[j].x;
    float M = m;
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, off));
    const float f = part_weight(m, M);
    float l = ml[j].y * f;
    if (s < nb) fac[i * kDecodeSlots + s] = f;
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
    if (__any_sync(0xffffffffu, ml[j].y < 0.f)) l = kLost;
    if (s == 0) {
      s_l[i] = l;
      store_lse(p, row0 + i, M, l);
    }
  }
  __syncthreads();
  for (int x = threadIdx.x; x < p.g * C4; x += NTHR) {
    const int i = x / C4, c = x % C4 * 4;
    float4 O = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s0 = 0; s0 < nb; s0 += kFirst) {
      if (s0 || x != (int)threadIdx.x) load_parts(x, s0);
#pragma unroll
      for (int s = 0; s < kFirst; ++s) {
        const float f = s0 + s < nb ? fac[i * kDecodeSlots + s0 + s] : 0.f;
        O.x += v[s].x * f;
        O.y += v[s].y * f;
        O.z += v[s].z * f;
        O.w += v[s].w * f;
      }
    }
    store4<T, D>(p, row0 + i, c, O, s_l[i]);
  }
}

// ---- scalar kernel (fp32, or bf16 with g <= 2) -------------------------------------------------------------------------
// HBM-bound. The rows of a share lie one behind the other in the cache, so one thread streams them into a ring of
// shared-memory stages with bulk copies (8 KB of K and 8 KB of V each) that count their bytes on the stage's barrier, and
// four warps work on whole stages: 32 KB are on the wire per block whatever the compiler does with the loop (with 16-byte
// loads to registers the kernel took 139 or 241 us on 1024 segments of 1638 rows depending on the code around them; this
// one takes 135, merge included: 0.98 of the measured copy bandwidth. 12 segments of 53038 rows: 118 -> 72 us).
// Stages: two keep six blocks resident per SM, so that a block's start and end are covered by the others (four stages: 163 us
// instead of 135); in a call of at most two blocks per SM six hold most of a share (8 segments of 3020 fp32 rows, us with 2 / 3
// / 4 / 6 stages: g = 1 14.1 / 13.6 / 13.6 / 13.5, g = 4 23.0 / 20.6 / 22.9 / 20.4; 4 of 11329 bf16 rows 15.9 / 15.6 / 15.8 / 15.2).
// (The tensor-core kernel gains nothing by deeper buffers, 10.5 -> 10.9 us for 8 segments of 2952 rows, g = 4: with them the next
// call's blocks find no room beside these.)
constexpr int kStageBytes = 16384;  // K, then V
constexpr long long kCopyWait = 4000000000ll;  // ~2 s: bound of a wait for a copy
constexpr long long kLandWait = 2000000ll;     // ~1 ms: what copies in flight get to land once a wait has run out

__device__ __forceinline__ void bar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count));
}
__device__ __forceinline__ void bar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void bar_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool bar_try(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait. False if it runs out, here or in another thread of the block; that is reported where there is a workspace.
__device__ __forceinline__ bool bar_wait(const DecodeParams& p, uint64_t* bar, uint32_t parity, volatile int* gave_up) {
  if (bar_try(bar, parity)) return true;
  const long long t0 = clock64();
  while (!bar_try(bar, parity)) {
    if (*gave_up) return false;
    if (clock64() - t0 > p.wait_clocks) {
      *gave_up = 1;
      if (p.ws) set_status(p.ws, MADAKV_ETIMEOUT);
    }
  }
  return true;
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(smem_addr(bar))
               : "memory");
}

template <typename T, int D, int G, int kRingStages>
__global__ void __launch_bounds__(NT) decode_kernel(const __grid_constant__ DecodeParams p) {
  constexpr int EPL = Vec16<T>::N;          // elements per lane
  constexpr int LPR = D / EPL;              // lanes per row
  constexpr int GROUPS = NT / LPR;          // rows the block reads per instruction
  constexpr int U = 4;                      // rows per thread and stage
  constexpr int ROW_BYTES = D * (int)sizeof(T);
  constexpr int ROWS = GROUPS * U;          // rows per stage
  static_assert(2 * ROWS * ROW_BYTES == kStageBytes, "stage size");
  static_assert(GROUPS * G * (D + 2) * 4 + G * (D + 2) * 4 <= kRingStages * kStageBytes, "the merge reuses the ring");
  extern __shared__ __align__(128) unsigned char dsmem[];
  __shared__ uint64_t full[kRingStages], empty[kRingStages];
  __shared__ int gave_up;

  if (threadIdx.x == 0) {
    gave_up = 0;
    for (int i = 0; i < kRingStages; ++i) {
      bar_init(&full[i], 1);
      bar_init(&empty[i], NT / 32);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  pdl_wait();
  pdl_go();
  const int y = blockIdx.x / p.slots, slot = blockIdx.x % p.slots;
  const int u = unit_of(p, y);
  const SegView view = segment_view(p, u, slot == 0 && threadIdx.x == 0);
  const int len = view.len, nb = segment_blocks(p, len);
  int row_begin, row_end;
  block_rows(nb, len, slot, row_begin, row_end);  // (empty beyond the nb-th block)
  const int h = u % p.Hkv, bl = u / p.Hkv;
  const int lane = threadIdx.x % LPR, grp = threadIdx.x / LPR;
  __syncthreads();

  float* s_o = reinterpret_cast<float*>(dsmem);  // [GROUPS][G][D], once the ring is done with
  float* s_m = s_o + GROUPS * G * D;             // [GROUPS][G]
  float* s_l = s_m + GROUPS * G;
  float* b_o = s_l + GROUPS * G;                 // the block's result: [G][D], [G], [G]
  float* b_m = b_o + G * D;
  float* b_l = b_m + G;
  static_assert((GROUPS * G * (D + 2)) % 4 == 0, "b_o is read in 16-byte pieces");
  if (slot < nb) {
    const int64_t off = p.seg_off[u];
    store_new_row<ROW_BYTES>(p, u, off, view, row_begin, row_end);
    const int steps = (row_end - row_begin + ROWS - 1) / ROWS;
    // one thread: the rows of a step into their stage. The appended row, always the last one of the segment, is read from
    // where it comes from, not from the cache row this block is writing.
    auto issue = [&](int it) {
      const int r = row_begin + it * ROWS, rows = min(ROWS, row_end - r), st = it % kRingStages;
      const bool fresh = view.new_row >= r && view.new_row < r + rows;
      const uint32_t bytes = (uint32_t)(rows - (fresh ? 1 : 0)) * ROW_BYTES;
      const uint32_t kd = smem_addr(dsmem) + st * kStageBytes, vd = kd + kStageBytes / 2;
      bar_expect(&full[st], (uint32_t)(2 * rows * ROW_BYTES));
      if (p.hold_copies) return;
      if (bytes) {
        bulk_load(kd, (const char*)p.k_c + (off + r) * ROW_BYTES, bytes, &full[st]);
        bulk_load(vd, (const char*)p.v_c + (off + r) * ROW_BYTES, bytes, &full[st]);
      }
      if (fresh) {
        bulk_load(kd + bytes, (const char*)p.k_new + (int64_t)u * ROW_BYTES, ROW_BYTES, &full[st]);
        bulk_load(vd + bytes, (const char*)p.v_new + (int64_t)u * ROW_BYTES, ROW_BYTES, &full[st]);
      }
    };
    if (threadIdx.x == 0)
      for (int it = 0; it < min(kRingStages, steps); ++it) issue(it);

    float qr[G][EPL];
#pragma unroll
    for (int i = 0; i < G; ++i) {
      if (i < p.g) {
        const T* qp = reinterpret_cast<const T*>(p.q) + ((int64_t)bl * p.Hq + h * p.g + i) * D + lane * EPL;
        Vec16<T>::load(qp, qr[i]);
#pragma unroll
        for (int c = 0; c < EPL; ++c) qr[i][c] *= p.scale2;
      } else {
#pragma unroll
        for (int c = 0; c < EPL; ++c) qr[i][c] = 0.f;
      }
    }
    float m[G], l[G], o[G][EPL];
#pragma unroll
    for (int i = 0; i < G; ++i) {
      m[i] = -INFINITY;
      l[i] = 0.f;
#pragma unroll
      for (int c = 0; c < EPL; ++c) o[i][c] = 0.f;
    }
    bool ok = true;  // (else the steps go on, on whatever the stages hold: a way out of the loop cost a fifth at G = 8)
    for (int it = 0; it < steps; ++it) {
      const int st = it % kRingStages;
      const uint32_t use = (uint32_t)(it / kRingStages) & 1u;
      ok &= bar_wait(p, &full[st], use, &gave_up);
      const uint4* ks = reinterpret_cast<const uint4*>(dsmem + st * kStageBytes) + grp * LPR + lane;
      const uint4* vs = ks + kStageBytes / 32;
      const int left = row_end - row_begin - it * ROWS - grp;  // row j of this thread exists while GROUPS * j < left
      // scores of the U rows for all heads (heads beyond g have zero queries), then one softmax step for the U rows
      float sc[G][U];
#pragma unroll
      for (int j = 0; j < U; ++j) {
        float kf[EPL];
        Vec16<T>::cvt(ks[GROUPS * LPR * j], kf);
#pragma unroll
        for (int i = 0; i < G; ++i) {
          float x = 0.f;
#pragma unroll
          for (int c = 0; c < EPL; ++c) x = fmaf(qr[i][c], kf[c], x);
          sc[i][j] = x;
        }
      }
#pragma unroll
      for (int sh = LPR / 2; sh >= 1; sh >>= 1) {
#pragma unroll
        for (int i = 0; i < G; ++i)
#pragma unroll
          for (int j = 0; j < U; ++j) sc[i][j] += __shfl_xor_sync(0xffffffffu, sc[i][j], sh);
      }
#pragma unroll
      for (int i = 0; i < G; ++i) {
        float mn = m[i];
#pragma unroll
        for (int j = 0; j < U; ++j) {
          if (GROUPS * j >= left) sc[i][j] = -INFINITY;
          mn = fmaxf(mn, sc[i][j]);
        }
        const float base = mn == -INFINITY ? 0.f : mn;  // (no row yet: all weights exp2(-inf) = 0)
        const float f = fast_ex2(m[i] - base);
        l[i] *= f;
#pragma unroll
        for (int c = 0; c < EPL; ++c) o[i][c] *= f;
        m[i] = mn;
#pragma unroll
        for (int j = 0; j < U; ++j) {
          sc[i][j] = fast_ex2(sc[i][j] - base);
          l[i] += sc[i][j];
        }
      }
#pragma unroll
      for (int j = 0; j < U; ++j) {
        // (what a stage holds beyond the share's last row is undefined: not to be multiplied, not even by 0)
        const uint4 raw = vs[GROUPS * LPR * j];
        float vf[EPL];
        Vec16<T>::cvt(GROUPS * j < left ? raw : make_uint4(0u, 0u, 0u, 0u), vf);
#pragma unroll
        for (int i = 0; i < G; ++i)
#pragma unroll
          for (int c = 0; c < EPL; ++c) o[i][c] = fmaf(sc[i][j], vf[c], o[i][c]);
      }
      __syncwarp();
      if (threadIdx.x % 32 == 0) bar_arrive(&empty[st]);
      if (threadIdx.x == 0 && it + kRingStages < steps) {  // refill the stage once all warps are done with it
        ok &= bar_wait(p, &empty[st], use, &gave_up);
        if (ok) issue(it + kRingStages);
      }
    }
    const bool lost = __syncthreads_or(!ok);
    if (lost) {  // no copy may land in shared memory that the merge or another block uses
      const long long t0 = clock64();
      while (clock64() - t0 < kLandWait) __nanosleep(1000);
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < G; ++i) {
      if (lane == 0) {
        s_m[grp * G + i] = m[i];
        s_l[grp * G + i] = l[i];
      }
#pragma unroll
      for (int c = 0; c < EPL; c += 4)
        *reinterpret_cast<float4*>(s_o + (grp * G + i) * D + lane * EPL + c) =
            make_float4(o[i][c], o[i][c + 1], o[i][c + 2], o[i][c + 3]);
    }
    __syncthreads();
    for (int x = threadIdx.x; x < p.g * D; x += NT) {
      const int i = x / D, c = x % D;
      float M = -INFINITY;
#pragma unroll
      for (int gq = 0; gq < GROUPS; ++gq) M = fmaxf(M, s_m[gq * G + i]);
      float Lsum = 0.f, O = 0.f;
#pragma unroll
      for (int gq = 0; gq < GROUPS; ++gq) {
        const float f = part_weight(s_m[gq * G + i], M);
        Lsum += s_l[gq * G + i] * f;
        O += s_o[(gq * G + i) * D + c] * f;
      }
      b_o[i * D + c] = O;
      if (c == 0) {
        b_m[i] = M;
        b_l[i] = lost ? kLost : Lsum;
      }
    }
    __syncthreads();
  }
  finish_segment<T, D, NT>(p, b_o, b_m, b_l, s_o, u, y, slot, nb, view);
}

// ---- grouped-query partial on the warp-level tensor-core path (bf16, 3 <= g <= 16) ----------------------------------
// One K/V row serves g query heads: in scalar code that is 2 * g * D fused multiply-adds per 2 * D * 2 bytes read and
// the kernel is bound by the FMA pipe from g = 4 on. Here the g heads sit on the 16 rows of an m16n8k16 tile (rows
// beyond g carry zero queries): a warp takes 16 cache rows at a time, S = Q K^T as 2 key blocks x D/16 MMAs, the
// online softmax on the accumulator fragments, P rounded to bf16 and reused in place as the A operand of O += P V
// (D/8 MMAs). K and V rows go global -> shared with 16-byte asynchronous copies, double-buffered per warp, rows padded
// by 16 bytes so that the 8x8 matrix loads are free of bank conflicts. Warps work independently on interleaved
// 16-row chunks of the split and are merged in shared memory at its end.
constexpr int kMmaWarps = 4;

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool valid) {
  const int bytes = valid ? 16 : 0;  // zero bytes read: the 16 destination bytes are filled with zeros
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

template <int D>
struct MmaTile {
  static constexpr int PITCH = D * 2 + 16;            // bytes from one staged row to the next
  static constexpr int TILE = 16 * PITCH;             // 16 rows of K or of V
  static constexpr int WARP = 4 * TILE;               // two buffers of (K, V)
  static constexpr int OPITCH = D + 8;                // floats from one head's merged row to the next
  static constexpr int BYTES = kMmaWarps * WARP;
  static constexpr int BLOCK_OFF = 16 * OPITCH * 4 + 2 * 16 * 4;  // the block's result in warp 0's area: o [16][D], m [16], l [16]
  static_assert(BLOCK_OFF % 16 == 0 && BLOCK_OFF + 16 * D * 4 + 2 * 16 * 4 <= WARP,
                "the merge staging reuses a warp's K/V buffers");
  static_assert(16 * kDecodeSlots * 4 <= 16 * OPITCH * 4, "the weights of a split call's partials take warp 0's place");
};

template <int D>
__global__ void __launch_bounds__(kMmaWarps * 32, 3) decode_mma_kernel(const __grid_constant__ DecodeParams p) {
  using MT = MmaTile<D>;
  constexpr int ROW_BYTES = D * 2;
  constexpr int LPR = ROW_BYTES / 16;  // 16-byte pieces per row
  constexpr int KC = D / 16;           // contraction chunks of Q K^T
  constexpr int NB = D / 8;            // 8-column blocks of the output
  extern __shared__ __align__(128) unsigned char dsmem[];

  pdl_wait();
  pdl_go();
  const int y = blockIdx.x / p.slots, slot = blockIdx.x % p.slots;
  const int u = unit_of(p, y);
  const SegView view = segment_view(p, u, slot == 0 && threadIdx.x == 0);
  const int len = view.len, nb = segment_blocks(p, len);
  int row_begin, row_end;
  block_rows(nb, len, slot, row_begin, row_end);  // (empty beyond the nb-th block)
  float* bo = reinterpret_cast<float*>(dsmem + MT::BLOCK_OFF);
  if (slot < nb) {
  const int64_t off = p.seg_off[u];
  store_new_row<D * 2>(p, u, off, view, row_begin, row_end);
  const int h = u % p.Hkv, bl = u / p.Hkv;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int hr = lane / 4, t = lane % 4;  // fragment coordinates: row (head) hr and hr + 8, column pair t
  unsigned char* wsm = dsmem + warp * MT::WARP;
  const uint32_t wsm_a = smem_addr(wsm);

  // Q as A fragments, one per contraction chunk: (head hr, d 2t..2t+1), (head hr+8, same), (head hr, d 2t+8..), ...
  uint32_t qa[KC][4];
  {
    const __nv_bfloat16* q0 = reinterpret_cast<const __nv_bfloat16*>(p.q) + ((int64_t)bl * p.Hq + h * p.g) * D;
#pragma unroll
    for (int c = 0; c < KC; ++c) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int head = hr + 8 * (j & 1), dcol = c * 16 + 2 * t + 8 * (j >> 1);
        qa[c][j] = head < p.g ? *reinterpret_cast<const uint32_t*>(q0 + (int64_t)head * D + dcol) : 0u;
      }
    }
  }
  const char* kc = (const char*)p.k_c + off * ROW_BYTES;
  const char* vc = (const char*)p.v_c + off * ROW_BYTES;
  const char* kn = view.new_row >= 0 ? (const char*)p.k_new + (int64_t)u * ROW_BYTES : nullptr;
  const char* vn = view.new_row >= 0 ? (const char*)p.v_new + (int64_t)u * ROW_BYTES : nullptr;
  // per-lane shared-memory offsets of the matrix loads: lanes 8i..8i+7 address the rows of the i-th 8x8 matrix
  const int mi = lane / 8, mr = lane % 8;
  const uint32_t k_lane = ((mi >> 1) * 8 + mr) * MT::PITCH + (mi & 1) * 16;  // keys (mi/2)*8.., d half mi%2
  const uint32_t v_lane = ((mi & 1) * 8 + mr) * MT::PITCH + (mi >> 1) * 16;  // keys (mi%2)*8.., column block mi/2

  {
    float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};
    float o[NB][4];
#pragma unroll
    for (int nb = 0; nb < NB; ++nb) o[nb][0] = o[nb][1] = o[nb][2] = o[nb][3] = 0.f;

    auto load_chunk = [&](int r, int buf) {
      const uint32_t kd = wsm_a + buf * 2 * MT::TILE, vd = kd + MT::TILE;
#pragma unroll
      for (int x = lane; x < 16 * LPR; x += 32) {
        const int rr = x / LPR, cc = x % LPR;
        const bool valid = r + rr < row_end;
        const int64_t src = (int64_t)(valid ? r + rr : r) * ROW_BYTES + cc * 16;  // row r itself is always valid
        // (the appended row comes from k_new / v_new, not from the cache row this block is writing)
        const bool fresh = valid && r + rr == view.new_row;
        cp_async16(kd + rr * MT::PITCH + cc * 16, fresh ? kn + cc * 16 : kc + src, valid);
        cp_async16(vd + rr * MT::PITCH + cc * 16, fresh ? vn + cc * 16 : vc + src, valid);
      }
    };
    if (row_begin + 16 * warp < row_end) load_chunk(row_begin + 16 * warp, 0);
    cp_async_commit();
    for (int it = 0;; ++it) {
      const int r = row_begin + 16 * (warp + kMmaWarps * it);
      if (r >= row_end) break;
      const int buf = it & 1;
      if (r + 16 * kMmaWarps < row_end) load_chunk(r + 16 * kMmaWarps, buf ^ 1);
      cp_async_commit();
      cp_async_wait<1>();
      __syncwarp();
      const uint32_t kb = wsm_a + buf * 2 * MT::TILE, vb = kb + MT::TILE;

      float s[2][4];
#pragma unroll
      for (int b = 0; b < 2; ++b) s[b][0] = s[b][1] = s[b][2] = s[b][3] = 0.f;
#pragma unroll
      for (int c = 0; c < KC; ++c) {
        uint32_t kf[4];
        ldmatrix_x4(kb + k_lane + c * 32, kf);
        mma_bf16_16816(s[0], qa[c], kf[0], kf[1]);
        mma_bf16_16816(s[1], qa[c], kf[2], kf[3]);
      }
      // element j of block b: head hr + 8 * (j / 2), key r + 8 * b + 2 * t + (j & 1)
#pragma unroll
      for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          s[b][j] = (r + 8 * b + 2 * t + (j & 1) < row_end) ? s[b][j] * p.scale2 : -INFINITY;
      float f[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        float mx = fmaxf(fmaxf(s[0][2 * e], s[0][2 * e + 1]), fmaxf(s[1][2 * e], s[1][2 * e + 1]));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        const float mn = fmaxf(m[e], mx);  // finite: key r of the chunk is valid
        f[e] = fast_ex2(m[e] - mn);        // exp2(-inf) = 0 on the first chunk
        m[e] = mn;
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          s[b][2 * e] = fast_ex2(s[b][2 * e] - mn);
          s[b][2 * e + 1] = fast_ex2(s[b][2 * e + 1] - mn);
        }
        l[e] = l[e] * f[e] + ((s[0][2 * e] + s[0][2 * e + 1]) + (s[1][2 * e] + s[1][2 * e + 1]));
      }
      if (__any_sync(0xffffffffu, f[0] != 1.f || f[1] != 1.f)) {
#pragma unroll
        for (int nb = 0; nb < NB; ++nb) {
          o[nb][0] *= f[0]; o[nb][1] *= f[0];
          o[nb][2] *= f[1]; o[nb][3] *= f[1];
        }
      }
      uint32_t pa[4];
      pa[0] = pack_bf16x2(s[0][0], s[0][1]);
      pa[1] = pack_bf16x2(s[0][2], s[0][3]);
      pa[2] = pack_bf16x2(s[1][0], s[1][1]);
      pa[3] = pack_bf16x2(s[1][2], s[1][3]);
#pragma unroll
      for (int nb = 0; nb < NB; nb += 2) {
        uint32_t vf[4];
        ldmatrix_x4_trans(vb + v_lane + nb * 16, vf);
        mma_bf16_16816(o[nb], pa, vf[0], vf[1]);
        mma_bf16_16816(o[nb + 1], pa, vf[2], vf[3]);
      }
      __syncwarp();  // the buffer is refilled two iterations on
    }
    cp_async_wait<0>();
    __syncwarp();
    // the warp's state goes to its own (now idle) staging area: o[16][D + 8], then m[16], l[16]
    float* so = reinterpret_cast<float*>(wsm);
    float* sm = so + 16 * MT::OPITCH;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      l[e] += __shfl_xor_sync(0xffffffffu, l[e], 1);
      l[e] += __shfl_xor_sync(0xffffffffu, l[e], 2);
      if (t == 0) {
        sm[hr + 8 * e] = m[e];
        sm[16 + hr + 8 * e] = l[e];
      }
    }
#pragma unroll
    for (int nb = 0; nb < NB; ++nb) {
      *reinterpret_cast<float2*>(so + hr * MT::OPITCH + nb * 8 + 2 * t) = make_float2(o[nb][0], o[nb][1]);
      *reinterpret_cast<float2*>(so + (hr + 8) * MT::OPITCH + nb * 8 + 2 * t) = make_float2(o[nb][2], o[nb][3]);
    }
    __syncthreads();
    for (int x = threadIdx.x; x < p.g * D; x += kMmaWarps * 32) {
      const int i = x / D, c = x % D;
      float mw[kMmaWarps], M = -INFINITY;
#pragma unroll
      for (int w = 0; w < kMmaWarps; ++w) {
        mw[w] = reinterpret_cast<const float*>(dsmem + w * MT::WARP)[16 * MT::OPITCH + i];
        M = fmaxf(M, mw[w]);
      }
      float Lsum = 0.f, O = 0.f;
#pragma unroll
      for (int w = 0; w < kMmaWarps; ++w) {
        const float* wo = reinterpret_cast<const float*>(dsmem + w * MT::WARP);
        const float fw = part_weight(mw[w], M);
        Lsum += wo[16 * MT::OPITCH + 16 + i] * fw;
        O += wo[i * MT::OPITCH + c] * fw;
      }
      bo[x] = O;
      if (c == 0) {
        bo[16 * D + i] = M;
        bo[16 * D + 16 + i] = Lsum;
      }
    }
  }
  __syncthreads();
  }
  finish_segment<__nv_bfloat16, D, kMmaWarps * 32>(p, bo, bo + 16 * D, bo + 16 * D + 16, reinterpret_cast<float*>(dsmem), u, y,
                                                          slot, nb, view);
}

// Blocks per segment and the rows a block takes at least. The segments' lengths are device data; the rows of the cache per
// segment stand in for them, so that short segments do not launch blocks only to arrive at the counter.
//   fewer than 64 segments (one layer of a model): bound by the latency of the blocks, so shares of at least 128 rows
//     (tensor-core kernel, two iterations of its warps; 256 where that would be more than a block per SM, because every
//     block more makes the merge longer: 4 segments of 771 rows, g = 7, 9.7 us at 128, 10.8 at 256; 8 of 1777 8.6 and
//     9.0; 8 of 2952 11.9 and 10.9; 20 of 2000 15.8 and 15.5), as many blocks as are resident at once, at most 32 (16
//     segments of 8725 rows, g = 4: 46 us with 16 blocks each, 56 with 32, which no longer fit; 12 of 53038, g = 1: 72 with
//     32, 111 with 16). Resident per SM: six of the scalar kernel by their shared memory, but three for fp32 with g > 4 (160
//     registers); three of the tensor-core kernel. (The most that fit against one more per SM: 40 segments of 8000 rows,
//     g = 1 36 and 40; 60 of 3000 21.2 and 23.3; fp32 40 of 5000, g = 4 52 and 58; with g = 8, three against seven, 20 of 5000
//     50 and 64)
//   more: shares of 1024 rows where that gives this many blocks, else 512 (896 segments of 2512 rows, g = 7:
//     190 us at 1024, 197 at 512, 247 at 256; 10240 of 410, g = 1: 311 with one block each, 335 with two; 1024 of 1638,
//     g = 1: 137 at 1024, 135 at 512; 900 of 1500 115 and 111; 640 of 2500 135 and 129; 112 of 3000 44 and 38)
//   more than there are counters: one block each
struct DecodeShape {
  int slots, min_rows;
};
DecodeShape decode_shape(const madakv_config& c, int n_sel, int64_t capacity, bool tensor_core_kernel, int splits) {
  if (n_sel > kCounters) return {1, 1};
  const int64_t units = (int64_t)c.batch * c.n_layers * c.n_kv_heads, longest = c.max_seq_len + c.max_new_tokens;
  const int64_t rows = capacity / units < longest ? capacity / units : longest;
  const int resident = 148 * (tensor_core_kernel || c.n_q_heads / c.n_kv_heads > 4 ? 3 : 6);
  int share, most;
  if (n_sel < 64) {
    share = tensor_core_kernel && n_sel * ((rows + 127) / 128) > 148 ? 256 : 128;
    most = resident / n_sel < kDecodeSlots ? resident / n_sel : kDecodeSlots;
  } else {
    share = n_sel * (rows / 1024 + 1) >= 148 * (tensor_core_kernel ? 6 : 14) ? 1024 : 512;
    most = 8;
  }
  const int64_t want = 3 * rows / (2 * share) + 1;  // (segments may be longer than the mean)
  const int slots = splits < most ? splits : most;
  return {(int)(want < slots ? want : slots), share};
}

template <typename T, int D>
int run(DecodeParams p, const madakv_config& c, int splits, cudaStream_t st) {
  // every host-side refusal comes before the launch (an appending call changes the cache)
  const bool mma = sizeof(T) == 2 && p.g >= 3 && p.g <= 16;
  if (!mma && p.g > 8) return MADAKV_EUNSUPPORTED;
  const DecodeShape s = decode_shape(c, p.n_sel, p.capacity, mma, splits);
  p.slots = s.slots;
  p.min_rows = s.min_rows;
  p.part_ml = reinterpret_cast<float2*>(p.part + (int64_t)c.batch * c.n_layers * c.n_q_heads * s.slots * D);
  // Counters that no caller can reach are cleared by every call: two calls that overlapped may leave them anywhere.
  if (!p.ws && p.slots > 1 && cudaMemsetAsync(p.counter, 0, (size_t)p.n_sel * sizeof(unsigned), st) != cudaSuccess) return MADAKV_ECUDA;
  const dim3 grid((unsigned)p.n_sel * p.slots);  // one dimension: no 65535 limit on the number of segments
  if constexpr (sizeof(T) == 2) {
    if (mma) {
      if (cudaFuncSetAttribute(decode_mma_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, MmaTile<D>::BYTES) !=
          cudaSuccess)
        return MADAKV_ECUDA;
      launch_pdl(decode_mma_kernel<D>, grid, dim3(kMmaWarps * 32), MmaTile<D>::BYTES, st, p);
      return launch_status();
    }
  }
  // Failure-path test (no GPU fault involved): MADAKV_TEST_HOLD_COPIES withholds the copies of cache rows, so every wait for
  // them runs out, after the given number of clock cycles (at least 100 000).
  if (const char* e = getenv("MADAKV_TEST_HOLD_COPIES")) {
    const long long v = atoll(e);
    if (v >= 100000 && v < kCopyWait) {
      p.hold_copies = 1;
      p.wait_clocks = v;
    }
  }
  auto go = [&](auto heads) {
    constexpr int G = decltype(heads)::value;
    if (p.n_sel * p.slots <= 2 * 148) {
      auto kernel = decode_kernel<T, D, G, 6>;
      if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 6 * kStageBytes) != cudaSuccess) return (int)MADAKV_ECUDA;
      launch_pdl(kernel, grid, dim3(NT), 6 * kStageBytes, st, p);
    } else {
      launch_pdl(decode_kernel<T, D, G, 2>, grid, dim3(NT), 2 * kStageBytes, st, p);
    }
    return launch_status();
  };
  if (p.g == 1) return go(std::integral_constant<int, 1>());
  if (p.g == 2) return go(std::integral_constant<int, 2>());
  if constexpr (sizeof(T) == 4) return p.g <= 4 ? go(std::integral_constant<int, 4>()) : go(std::integral_constant<int, 8>());
  return MADAKV_EUNSUPPORTED;
}

}  // namespace

int launch_decode(const madakv_config& c, int layer, const void* q, const void* k_new, const void* v_new, void* k_c,
                  void* v_c, const int64_t* seg_off, int32_t* kept_len, int64_t capacity, void* out, float* lse_out,
                  void* ws, cudaStream_t st) {
  const WsLayout wl = ws_layout(c);
  DecodeParams p;
  p.q = q;
  p.k_new = k_new;
  p.v_new = v_new;
  p.k_c = k_c;
  p.v_c = v_c;
  p.seg_off = seg_off;
  p.kept_len = kept_len;
  p.capacity = capacity;
  p.out = out;
  p.lse_out = lse_out;
  p.part = reinterpret_cast<float*>((char*)ws + wl.decode_off);
  p.counter = reinterpret_cast<unsigned*>((char*)ws + kHeaderBytes);
  p.ws = ws;
  p.L = c.n_layers;
  p.Hq = c.n_q_heads;
  p.Hkv = c.n_kv_heads;
  p.g = c.n_q_heads / c.n_kv_heads;
  p.layer = layer;
  p.n_sel = (layer < 0 ? c.batch * c.n_layers : c.batch) * c.n_kv_heads;
  const int splits = wl.decode_splits;
  p.scale2 = scale_of(c) * kLog2e;
  p.hold_copies = 0;
  p.wait_clocks = kCopyWait;
  if (c.dtype == MADAKV_F32) return c.head_dim == 64 ? run<float, 64>(p, c, splits, st) : run<float, 128>(p, c, splits, st);
  return c.head_dim == 64 ? run<__nv_bfloat16, 64>(p, c, splits, st) : run<__nv_bfloat16, 128>(p, c, splits, st);
}

}  // namespace madakv

// ---------------------------------------------------------------------------------------------------------------
// madakv_decode_attn_static: the same attention kernels with their split partials in a fixed array of the library
// image, for callers that have no way to provide (or allocate) a workspace.
// ---------------------------------------------------------------------------------------------------------------

// Split partials of the no-allocation entry point. One copy per GPU that loads the library, shared by all calls. The segment
// counters of a split call lie behind them; every call clears those it uses (see run()).
struct StaticScratch {
  unsigned char part[MADAKV_STATIC_SCRATCH_BYTES];
  unsigned counter[madakv::kCounters];
};
static __device__ __align__(256) StaticScratch g_static_scratch;

namespace madakv {
namespace {

constexpr int kMaxDevices = 64;
std::mutex g_static_mutex;
void* g_static_ptr[kMaxDevices] = {};  // device address of g_static_scratch on each device, once looked up

// In host code the name g_static_scratch is only a handle; the address kernels can use comes from the runtime,
// per device, with that device current.
int static_scratch(void** out) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return MADAKV_ECUDA;
  std::lock_guard<std::mutex> lock(g_static_mutex);
  if (!g_static_ptr[dev]) {
    void* ptr = nullptr;
    if (cudaGetSymbolAddress((void**)&ptr, g_static_scratch) != cudaSuccess || !ptr) {
      cudaGetLastError();
      return MADAKV_ECUDA;
    }
    g_static_ptr[dev] = ptr;
  }
  *out = g_static_ptr[dev];
  return MADAKV_OK;
}

}  // namespace
}  // namespace madakv

extern "C" int madakv_decode_attn_static(const madakv_config* cfg, int32_t layer, const void* q, const void* k_c,
                                         const void* v_c, const int64_t* seg_off, const int32_t* kept_len,
                                         int64_t capacity, void* out, float* lse_out, void* stream) {
  using namespace madakv;
  int rc = check_config(cfg);
  if (rc) return rc;
  if (!q || !k_c || !v_c || !seg_off || !kept_len || !out) return MADAKV_EINVAL;
  if (layer < -1 || layer >= cfg->n_layers) return MADAKV_ESHAPE;
  if (capacity <= 0) return MADAKV_ECAPACITY;
  if (!aligned16(q) || !aligned16(k_c) || !aligned16(v_c) || !aligned16(out) || ((uintptr_t)seg_off & 7) ||
      ((uintptr_t)kept_len & 3) || ((uintptr_t)lse_out & 3))
    return MADAKV_EALIGN;
  const madakv_config& c = *cfg;
  const int splits = ws_layout(c).decode_splits;
  const size_t need = (size_t)c.batch * c.n_layers * c.n_q_heads * (size_t)splits * (c.head_dim + 2) * sizeof(float);
  if (need > (size_t)MADAKV_STATIC_SCRATCH_BYTES) return MADAKV_ESTATIC;
  void* scratch = nullptr;
  if ((rc = static_scratch(&scratch))) return rc;
  unsigned* counters = reinterpret_cast<unsigned*>((char*)scratch + offsetof(StaticScratch, counter));

  DecodeParams p;
  p.q = q;
  p.k_new = nullptr;  // no append: the caches and kept_len are only read
  p.v_new = nullptr;
  p.k_c = const_cast<void*>(k_c);
  p.v_c = const_cast<void*>(v_c);
  p.seg_off = seg_off;
  p.kept_len = const_cast<int32_t*>(kept_len);
  p.capacity = capacity;
  p.out = out;
  p.lse_out = lse_out;
  p.part = reinterpret_cast<float*>(scratch);
  p.counter = counters;
  p.ws = nullptr;  // no status word: a wait that ran out shows as NaN in the segment's results
  p.L = c.n_layers;
  p.Hq = c.n_q_heads;
  p.Hkv = c.n_kv_heads;
  p.g = c.n_q_heads / c.n_kv_heads;
  p.layer = layer;
  p.n_sel = (layer < 0 ? c.batch * c.n_layers : c.batch) * c.n_kv_heads;
  p.scale2 = scale_of(c) * kLog2e;
  p.hold_copies = 0;
  p.wait_clocks = kCopyWait;
  cudaStream_t st = (cudaStream_t)stream;
  if (c.dtype == MADAKV_F32) return c.head_dim == 64 ? run<float, 64>(p, c, splits, st) : run<float, 128>(p, c, splits, st);
  return c.head_dim == 64 ? run<__nv_bfloat16, 64>(p, c, splits, st) : run<__nv_bfloat16, 128>(p, c, splits, st);
}
