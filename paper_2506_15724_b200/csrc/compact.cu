// Stage 4b: gather the kept K/V rows of every unit into the ragged per-head cache (bit copies).
//
// A row is d * elem_bytes = 128..512 bytes = LPR lanes of 16 bytes; a warp moves 32 / LPR rows of K and of V per
// instruction. Reads are whole 128-byte lines at random rows, writes are contiguous. A thread has U rows of K and of V in
// flight: all positions are read before the first row, all rows before the first store.
#include "common.cuh"

namespace madakv {
namespace {

constexpr int NT = 256;
constexpr int kMaxBlocksX = 64;  // blocks per unit at most in calls with many units

struct CompactParams {
  const char* k;
  const char* v;
  char* k_c;
  char* v_c;
  const int32_t* kept_idx;
  const int64_t* seg_off;
  const int32_t* kept_len;
  int64_t capacity;
  int64_t stride_b, stride_l, stride_h, stride_t;  // bytes
  int L, Hkv, n_max, row_bytes, headroom;
};

template <int LPR, int U>  // 16-byte lanes per row, rows per thread and iteration
__global__ void __launch_bounds__(NT) compact_kernel(CompactParams p) {
  constexpr int RPI = NT / LPR;  // rows the block's threads cover once
  pdl_wait();
  pdl_go();
  const int u = blockIdx.y;
  const int len = p.kept_len[u];
  const int64_t off = p.seg_off[u];  // (read beside the length, not after it)
  if ((int)blockIdx.x * RPI * U >= len) return;
  // a segment that selection refused (MADAKV_ECAPACITY: it would end beyond the cache) has no index list: skip it
  if (off + len + p.headroom > p.capacity) return;
  const int h = u % p.Hkv, l = (u / p.Hkv) % p.L, b = u / (p.Hkv * p.L);
  const int lane = threadIdx.x % LPR, sub = threadIdx.x / LPR;
  const int64_t src_base = b * p.stride_b + l * p.stride_l + h * p.stride_h + lane * 16;
  // a block takes every gridDim.x-th stretch of RPI * U rows
  for (int row0 = blockIdx.x * RPI * U; row0 < len; row0 += gridDim.x * RPI * U) {
    int idx[U];
    uint4 kv[U], vv[U];
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const int r = row0 + j * RPI + sub;
      idx[j] = r < len ? __ldg(p.kept_idx + off + r) : -1;
      if (idx[j] >= p.n_max) idx[j] = -1;
    }
#pragma unroll
    for (int j = 0; j < U; ++j)
      if (idx[j] >= 0) {
        const int64_t src = src_base + (int64_t)idx[j] * p.stride_t;
        kv[j] = __ldg(reinterpret_cast<const uint4*>(p.k + src));
        vv[j] = __ldg(reinterpret_cast<const uint4*>(p.v + src));
      }
#pragma unroll
    for (int j = 0; j < U; ++j)
      if (idx[j] >= 0) {
        const int64_t dst = (off + row0 + j * RPI + sub) * (int64_t)p.row_bytes + lane * 16;
        *reinterpret_cast<uint4*>(p.k_c + dst) = kv[j];
        *reinterpret_cast<uint4*>(p.v_c + dst) = vv[j];
      }
  }
}

// Calls with many units are bound by HBM: four rows of K and V per thread keep enough loads on the wire. A call with few
// units (one layer) is bound by the latency of its blocks: one row per thread and as many blocks as a segment of half as much
// again as the cache's rows per segment can use, so that nearly every row's chain of loads and a store runs once (one layer of
// 4 heads with 128-row blocks that looped eight times: 13.5 us; with the blocks of the longest possible segment, most of
// which only returned: 5.1 us, now 4.1).
template <int LPR>
void launch_rows(const CompactParams& p, int units, cudaStream_t st) {
  constexpr int RPI = NT / LPR;
  if (units >= 64) {
    const int stretches = (p.n_max + RPI * 4 - 1) / (RPI * 4);
    launch_pdl(compact_kernel<LPR, 4>, dim3(stretches < kMaxBlocksX ? stretches : kMaxBlocksX, units), dim3(NT), 0, st, p);
  } else {
    const int64_t mean = p.capacity / units, rows = mean + mean / 2 < p.n_max ? mean + mean / 2 : p.n_max;
    const int stretches = (int)((rows + RPI - 1) / RPI), most = 4096 / units;
    launch_pdl(compact_kernel<LPR, 1>, dim3(stretches < 1 ? 1 : stretches < most ? stretches : most, units), dim3(NT), 0, st, p);
  }
}

}  // namespace

int launch_compact(const madakv_config& c, const void* k, const void* v, madakv_strides s, const int32_t* kept_idx,
                   const int64_t* seg_off, const int32_t* kept_len, void* k_c, void* v_c, int64_t capacity, void* ws,
                   cudaStream_t st) {
  (void)ws;
  const int e = elem_bytes(c);
  CompactParams p;
  p.k = (const char*)k;
  p.v = (const char*)v;
  p.k_c = (char*)k_c;
  p.v_c = (char*)v_c;
  p.kept_idx = kept_idx;
  p.seg_off = seg_off;
  p.kept_len = kept_len;
  p.capacity = capacity;
  p.stride_b = s.batch * e;
  p.stride_l = s.layer * e;
  p.stride_h = s.head * e;
  p.stride_t = s.token * e;
  p.L = c.n_layers;
  p.Hkv = c.n_kv_heads;
  p.n_max = c.max_seq_len;
  p.row_bytes = c.head_dim * e;
  p.headroom = c.max_new_tokens;
  const int units = c.batch * c.n_layers * c.n_kv_heads;
  if (units > 65535) return MADAKV_EUNSUPPORTED;
  switch (p.row_bytes / 16) {
    case 8: launch_rows<8>(p, units, st); break;
    case 16: launch_rows<16>(p, units, st); break;
    case 32: launch_rows<32>(p, units, st); break;
    default: return MADAKV_EUNSUPPORTED;
  }
  return launch_status();
}

}  // namespace madakv
