// Chunked-prefill GQA attention over the retained cache.
//
// For each session of the last append (T <= 32 tokens, e.g. the 17 acoustic
// positions of a one-second unit), each KV head and its G = 4 query heads, the
// T*G query rows attend to every resident key at or before their own position
// (causal inside the chunk).
//
// bfloat16 runs on the tcgen05 tensor cores (kvc_attn_prefill_tc.cu), binary32
// on CUDA cores (kvc_attn_prefill_f32.cu); this file holds the launcher, the
// choice of split and the TMA tensor maps over the pool.
#include <cuda.h>

#include <algorithm>
#include <cmath>

#include "kvc_launch.cuh"

namespace kvc {

namespace {

constexpr int PF_D = 128;  // head dim of the bfloat16 pool views

// ---------------------------------------------------------------------------
// Host side: tensor maps over the pool (two 2-D views, dims 0-63 and 64-127).
// ---------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    cudaDriverEntryPointQueryResult q;
    void* p = nullptr;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

struct PoolMaps {
  const uint8_t* pool = nullptr;
  uint64_t rows = 0;
  CUtensorMap lo, hi;
  bool ok = false;
};

uint64_t pool_rows(const Dev& d) {
  return (uint64_t)d.n_pages * d.layers * 2 * d.kv_heads * PS;
}

bool make_pool_maps(const Dev& d, PoolMaps& m) {
  EncodeTiledFn enc = get_encode();
  if (!enc) return false;
  const uint64_t rows = pool_rows(d);
  cuuint64_t dims[2] = {64, rows};
  cuuint64_t strides[1] = {(cuuint64_t)PF_D * 2};
  cuuint32_t box[2] = {64, PS};
  cuuint32_t estr[2] = {1, 1};
  CUresult r1 = enc(&m.lo, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void*)d.pool, dims, strides, box,
                    estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  CUresult r2 = enc(&m.hi, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void*)(d.pool + 128), dims,
                    strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  m.ok = (r1 == CUDA_SUCCESS && r2 == CUDA_SUCCESS);
  m.pool = d.pool;
  m.rows = rows;
  return m.ok;
}

}  // namespace

bool pool_tensor_maps(const Dev& d, CUtensorMap* lo, CUtensorMap* hi) {
  // Keyed on the pool's address and extent: a later context may get the same address
  // for a pool of another shape.
  static thread_local PoolMaps maps;
  if (!maps.ok || maps.pool != d.pool || maps.rows != pool_rows(d)) {
    if (!make_pool_maps(d, maps)) return false;
  }
  *lo = maps.lo;
  *hi = maps.hi;
  return true;
}

namespace {

// Slices per pair of the pair split, or 0 for stream-K, whichever is expected to take less.
// n_pairs pairs, the longest of `s_max` stages (4 pages), `total` stages in all.  Times in
// us, fitted to 32-layer runs of 1-20 sessions of 8 KV heads at 200-10,600 positions:
//   pair split: launch, query tile and output 5, then 0.6 per stage of a slice (the issue of
//     S = Q K^T, one CTA per SM), 2.5 for the exchange between slices; never below the
//     bytes' time, 0.0048 per stage (32 KiB at 6.8 TB/s);
//   stream-K: 13 (partial states, two or more segments per CTA), 0.68 per stage of a CTA and
//     0.9 per part of a pair (merged one after the other).
// Measured at 4,100 positions (pair split with the k chosen / stream-K): 12.6 / 33.4 at one
// session, 14.4 / 28.5 at 2, 19.6 / 27.7 at 4, 31.1 / 35.6 at 9, 43.9 / 37.1 at 10 (k = 1),
// 45.5 / 49.4 at 16; at 250 positions 7.6 / 14.9 at one session, 8.9 / 18.9 at 16.
int prefill_slices(const Limits& lim, int n_pairs, double s_max, double total) {
  const double per = std::max(1.0, total / lim.pf_stream_k);
  double best = 13.0 + 0.68 * per + 0.9 * std::max(1.0, s_max / per);
  int best_k = 0;
  for (int k = 1; k <= PF_MAX_SLICES; ++k) {
    if (n_pairs > lim.pf_clusters[k]) continue;
    const double t = std::max(0.0048 * total, 5.0 + 0.6 * std::ceil(s_max / k) + (k > 1 ? 2.5 : 0.0));
    if (t < best) {
      best = t;
      best_k = k;
    }
  }
  return best_k;
}

}  // namespace

cudaError_t launch_attn_prefill(const Dev& d, const Limits& lim, int layer, const void* q,
                                void* out, int n_seq, int max_t, int pages_max,
                                int64_t pages_sum, bool early, cudaStream_t s, const void* new_k,
                                const void* new_v) {
  if (d.esz == 2) {
    CUtensorMap lo, hi;
    if (!pool_tensor_maps(d, &lo, &hi)) return cudaErrorInvalidValue;
    const int n_pairs = n_seq * d.kv_heads;
    const int k = prefill_slices(lim, n_pairs, (pages_max + 3) / 4,
                                 (double)d.kv_heads * (pages_sum / 4.0 + n_seq));
    // Each CTA of the stream-K split may write two partial slots.
    const int grid = k > 0 ? n_pairs * k : std::min(lim.pf_stream_k, d.pf_slots / 2);
    return launch_attn_prefill_tc(d, layer, lo, hi, q, out, grid, k, max_t, early, s, new_k, new_v);
  }
  if (new_k != nullptr) return cudaErrorInvalidValue;  // binary32: the API writes the rows first
  return launch_attn_prefill_f32(d, lim, layer, q, out, n_seq, max_t, pages_max, early, s);
}

}  // namespace kvc
