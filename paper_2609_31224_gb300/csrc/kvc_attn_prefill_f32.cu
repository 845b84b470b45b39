// Chunked-prefill GQA attention in binary32, on CUDA cores.
//
// A CTA takes one slice of one (session, KV head) pair's pages for up to 8 RT of the
// pair's T*G query rows, in tiles of 64 keys (4 pages).  The work is bound by the FMA rate
// (68 rows give 34 flop per byte of K/V), so both products are register tiles: with thread
// (ty, tx) of an 8 x 16 grid, S = Q K^T gives it RT rows x 4 keys (tx + 16 c), O += P V its
// RT rows x 4 dims, each shared-memory load of 16 bytes feeding 16 RT / (RT + 4) FMAs or
// more.  K/V tiles are copied asynchronously, one ahead, into rows padded against bank
// conflicts.  The half-warp of a row block holds a row's whole score tile, so the running
// maximum takes four shuffles and P needs no CTA barrier.
// The k slices of a pair are a thread-block cluster: each CTA leaves its partial rows
// (O, max, sum) in shared memory and merges its share of them from all k.
// Measured per launch with 17-token chunks: 4 sessions x 8 heads x 1,040 positions 26.5 us
// (0.29 GFMA; 7.5 us at the FMA peak: the FMA pipe is busy 45 % of the time on the SMs with two
// CTAs, two warps per scheduler, and a third of it over all), one session x 1 head x 520 positions 9.7 us; before,
// with a thread per row and chunks merged through global memory by one CTA, 96.7 and 55 us.
#include <type_traits>

#include "kvc_launch.cuh"

namespace kvc {

namespace {

constexpr int G = 4;
constexpr int D = 64;
constexpr int NK = 64;            // keys per tile
constexpr int THREADS = 128;      // 8 x 16
constexpr int PITCH = D + 4;      // floats per staged row
constexpr int MAX_K = 16;         // cluster size, at most (more than 8 is not portable)
constexpr int ONE_PER_SM = 120 * 1024;  // shared memory that keeps a second CTA off the SM
constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr float LOG2E = 1.4426950408889634f;

template <int RT>
struct Shape {
  static constexpr int ROWS = 8 * RT;
  static constexpr int Q = 0;                              // [ROWS][PITCH]
  static constexpr int P = Q + ROWS * PITCH;               // [ROWS][PITCH]
  static constexpr int KV = P + ROWS * PITCH;              // [2][K, V][NK][PITCH]
  static constexpr int ML = KV + 4 * NK * PITCH;           // [ROWS] (max, sum)
  static constexpr int FLOATS = ML + 2 * ROWS;
  static constexpr int SMEM = FLOATS * 4;
  static_assert(ROWS <= 2 * NK, "partial rows fit the first tile buffer");
  static_assert(SMEM <= ONE_PER_SM && 2 * (SMEM + 1024) <= 228 * 1024, "two CTAs per SM");
};

__device__ inline void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ inline void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ inline void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
// (The aligned barriers want the warp converged: its lanes come from loops of different lengths.)
__device__ inline void cluster_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ inline uint32_t cluster_map(uint32_t saddr, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
__device__ inline float4 ld_cluster_f4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ inline float2 ld_cluster_f2(uint32_t addr) {
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0,%1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr)
               : "memory");
  return v;
}

// Normalised merge of 16 bytes of a row over the k <= K CTAs of the cluster: (max, sum) at
// a_ml, the row's chunk at a_o in each.
template <int K>
__device__ inline float4 merge_chunk(uint32_t a_ml, uint32_t a_o, int k) {
  float2 ml[K];
  float4 v[K];
#pragma unroll
  for (int p = 0; p < K; ++p) {
    ml[p] = ld_cluster_f2(cluster_map(a_ml, min(p, k - 1)));
    v[p] = ld_cluster_f4(cluster_map(a_o, min(p, k - 1)));
  }
  float mx = -INFINITY, L = 0.f;
#pragma unroll
  for (int p = 0; p < K; ++p) mx = fmaxf(mx, ml[p].x);
  float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int p = 0; p < K; ++p) {
    const float w = p < k ? exp2_safe(ml[p].x, mx) : 0.f;
    L = fmaf(ml[p].y, w, L);
    a.x = fmaf(v[p].x, w, a.x);
    a.y = fmaf(v[p].y, w, a.y);
    a.z = fmaf(v[p].z, w, a.z);
    a.w = fmaf(v[p].w, w, a.w);
  }
  const float inv = 1.f / L;
  return make_float4(a.x * inv, a.y * inv, a.z * inv, a.w * inv);
}

// Grid: ((pair, row block), slice), the slices of a cluster innermost.
template <int RT>
__global__ void __launch_bounds__(THREADS, 2) attn_prefill_f32_kernel(
    Dev d, int layer, const float* __restrict__ q, float* __restrict__ out, float qk_scale,
    int n_rb, int k, int early) {
  using S = Shape<RT>;
  extern __shared__ __align__(16) float sm[];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int slice = blockIdx.x % k, rb = blockIdx.x / k % n_rb, pair = blockIdx.x / k / n_rb;
  const int H = d.kv_heads, seq = pair / H, head = pair % H;
  if (!early) pdl_wait();  // the first call after an append waits for it
  if (d.g->n_units == 0) {  // the append failed: the whole grid has nothing to do
    pdl_wait();
    return;
  }
  const SeqInfo si = d.seq[seq];
  pdl_launch_dependents();
  const int row0 = rb * S::ROWS, R = min(S::ROWS, si.t * G - row0);  // R <= 0: no rows here
  // This slice's pages [blk0, blk1), in tiles of up to 4.
  const int blk0 = (int)((int64_t)slice * si.n_blocks / k);
  const int blk1 = R > 0 ? (int)((int64_t)(slice + 1) * si.n_blocks / k) : blk0;
  const int32_t* hrow = d.hist_pt + (size_t)si.sid * d.max_pages_per_session;
  const int32_t* lrow = d.live_pt + (size_t)si.sid * d.max_pages_per_session;
  const float* pool = reinterpret_cast<const float*>(d.pool);
  const uint32_t s_kv = smem_u32(sm + S::KV);

  // The tile of pages b0 ..: thread (ty, tx) copies chunk tx of keys ty, ty + 8, ... of K and V.
  auto load_tile = [&](int b0, int buf) {
    int page[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) page[p] = b0 + p < blk1 ? block_page(si, hrow, lrow, b0 + p) : -1;
#pragma unroll
    for (int j = 0; j < NK / 8; ++j) {
      const int key = ty + 8 * j, pg = page[j >> 1];
      if (pg < 0) break;
      const float* src = pool + pool_offset_elems(d, pg, layer, 0, head, key & 15) + tx * 4;
      const uint32_t dst = s_kv + (((2 * buf) * NK + key) * PITCH + tx * 4) * 4;
      cp_async16(dst, src);
      cp_async16(dst + NK * PITCH * 4, src + (size_t)H * PS * D);
    }
    cp_async_commit();
  };
  if (blk0 < blk1) load_tile(blk0, 0);

  // Query rows, rotated at their tokens' positions and scaled.
  pdl_wait();
  for (int i = tid; i < S::ROWS * 8; i += THREADS) {
    const int r = i >> 3, c = i & 7;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
    if (r < R) {
      const int t = (row0 + r) / G, g = (row0 + r) % G;
      const float* qrow = q + ((size_t)(si.q_row0 + t) * d.q_heads + head * G + g) * D + c * 4;
      const float4 x = *reinterpret_cast<const float4*>(qrow);
      const float4 y = *reinterpret_cast<const float4*>(qrow + D / 2);
      const float4* cs = reinterpret_cast<const float4*>(
          d.rope + (size_t)(si.pos_first + t) * (D / 2) + c * 4);
      const float4 c0 = cs[0], c1 = cs[1];  // (cos, sin) of four dims
      a = make_float4(fmaf(x.x, c0.x, -y.x * c0.y) * qk_scale, fmaf(x.y, c0.z, -y.y * c0.w) * qk_scale,
                      fmaf(x.z, c1.x, -y.z * c1.y) * qk_scale, fmaf(x.w, c1.z, -y.w * c1.w) * qk_scale);
      b = make_float4(fmaf(y.x, c0.x, x.x * c0.y) * qk_scale, fmaf(y.y, c0.z, x.y * c0.w) * qk_scale,
                      fmaf(y.z, c1.x, x.z * c1.y) * qk_scale, fmaf(y.w, c1.z, x.w * c1.w) * qk_scale);
    }
    *reinterpret_cast<float4*>(sm + S::Q + r * PITCH + c * 4) = a;
    *reinterpret_cast<float4*>(sm + S::Q + r * PITCH + D / 2 + c * 4) = b;
  }

  const int q_log0 = si.n_hist + si.n_live - si.t;  // logical index of the chunk's first token
  float m[RT], l[RT];
  float4 o[RT];
#pragma unroll
  for (int i = 0; i < RT; ++i) {
    m[i] = -INFINITY;
    l[i] = 0.f;
    o[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  const float* s_q = sm + S::Q + ty * RT * PITCH;
  float* s_p = sm + S::P + ty * RT * PITCH;
  // One tile of NC pages (pages b0 .., in buffer buf).
  auto tile = [&](auto nc, int b0, int buf) {
    constexpr int NC = decltype(nc)::value;
    const float* kt = sm + S::KV + 2 * buf * NK * PITCH;
    const float* vt = kt + NK * PITCH;
    // Scores: even and odd dims accumulate in the two halves of a packed pair.
    float2 acc[RT][NC];
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
      for (int c = 0; c < NC; ++c) acc[i][c] = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int j = 0; j < D; j += 4) {
      float4 kv[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c)
        kv[c] = *reinterpret_cast<const float4*>(kt + (tx + 16 * c) * PITCH + j);
      // Rows innermost, so that an accumulator's updates lie RT NC instructions apart.
      float4 x[RT];
#pragma unroll
      for (int i = 0; i < RT; ++i) x[i] = *reinterpret_cast<const float4*>(s_q + i * PITCH + j);
#pragma unroll
      for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int i = 0; i < RT; ++i)
          acc[i][c] = __ffma2_rn(make_float2(x[i].x, x[i].y), make_float2(kv[c].x, kv[c].y), acc[i][c]);
#pragma unroll
      for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int i = 0; i < RT; ++i)
          acc[i][c] = __ffma2_rn(make_float2(x[i].z, x[i].w), make_float2(kv[c].z, kv[c].w), acc[i][c]);
    }
    // Key tx of page c: resident slot, and its logical index for the causal limit.
    float al[RT];
    int base[NC];
    bool valid[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const BlockRange br = block_range(si, b0 + c);
      valid[c] = tx >= br.lo && tx < br.hi;
      base[c] = br.base + tx;
    }
#pragma unroll
    for (int i = 0; i < RT; ++i) {
      const int q_log = q_log0 + (row0 + ty * RT + i) / G;
      float s[NC], mx = -INFINITY;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        s[c] = valid[c] && base[c] <= q_log ? acc[i][c].x + acc[i][c].y : -INFINITY;
        mx = fmaxf(mx, s[c]);
      }
#pragma unroll
      for (int off = 8; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(FULL, mx, off));
      const float mn = fmaxf(m[i], mx);
      al[i] = exp2_safe(m[i], mn);
      m[i] = mn;
      float rs = 0.f;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const float p = exp2_safe(s[c], mn);
        rs += p;
        s_p[i * PITCH + tx + 16 * c] = p;
      }
      l[i] = l[i] * al[i] + rs;  // (this thread's keys; summed over the half-warp at the end)
    }
    __syncwarp();
    // The tile's P V by itself first: one long chain over all keys would round more.
    float2 ot[RT][2];
#pragma unroll
    for (int i = 0; i < RT; ++i) ot[i][0] = ot[i][1] = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int j = 0; j < 16 * NC; j += 4) {
      float4 v[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) v[c] = *reinterpret_cast<const float4*>(vt + (j + c) * PITCH + tx * 4);
      float4 p[RT];
#pragma unroll
      for (int i = 0; i < RT; ++i) p[i] = *reinterpret_cast<const float4*>(s_p + i * PITCH + j);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
#pragma unroll
        for (int i = 0; i < RT; ++i) {
          const float x = c == 0 ? p[i].x : c == 1 ? p[i].y : c == 2 ? p[i].z : p[i].w;
          const float2 pp = make_float2(x, x);
          ot[i][0] = __ffma2_rn(pp, make_float2(v[c].x, v[c].y), ot[i][0]);
          ot[i][1] = __ffma2_rn(pp, make_float2(v[c].z, v[c].w), ot[i][1]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < RT; ++i) {
      o[i].x = fmaf(o[i].x, al[i], ot[i][0].x);
      o[i].y = fmaf(o[i].y, al[i], ot[i][0].y);
      o[i].z = fmaf(o[i].z, al[i], ot[i][1].x);
      o[i].w = fmaf(o[i].w, al[i], ot[i][1].y);
    }
  };
  for (int b0 = blk0, buf = 0; b0 < blk1; b0 += 4, buf ^= 1) {
    if (b0 + 4 < blk1) {
      load_tile(b0 + 4, buf ^ 1);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    switch (min(4, blk1 - b0)) {
      case 1: tile(std::integral_constant<int, 1>(), b0, buf); break;
      case 2: tile(std::integral_constant<int, 2>(), b0, buf); break;
      case 3: tile(std::integral_constant<int, 3>(), b0, buf); break;
      default: tile(std::integral_constant<int, 4>(), b0, buf); break;
    }
    __syncthreads();  // the tile's buffer and P are free
  }
#pragma unroll
  for (int i = 0; i < RT; ++i)
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) l[i] += __shfl_xor_sync(FULL, l[i], off);

  auto out_row = [&](int r) {  // row r of this block: its token's row of query head head G + g
    return out + ((size_t)(si.q_row0 + (row0 + r) / G) * d.q_heads + head * G + (row0 + r) % G) * D;
  };
  if (k == 1) {
#pragma unroll
    for (int i = 0; i < RT; ++i) {
      const int r = ty * RT + i;
      if (r < R) {
        const float inv = 1.f / l[i];
        *reinterpret_cast<float4*>(out_row(r) + tx * 4) =
            make_float4(o[i].x * inv, o[i].y * inv, o[i].z * inv, o[i].w * inv);
      }
    }
    return;
  }
  // Partial rows in the first tile buffer's place (every copy into it is complete).
#pragma unroll
  for (int i = 0; i < RT; ++i) {
    const int r = ty * RT + i;
    *reinterpret_cast<float4*>(sm + S::KV + r * PITCH + tx * 4) = o[i];
    if (tx == 0) *reinterpret_cast<float2*>(sm + S::ML + 2 * r) = make_float2(m[i], l[i]);
  }
  cluster_sync();
  const int rows = max(R, 0), r0 = slice * rows / k, r1 = (slice + 1) * rows / k;
  for (int i = tid; i < (r1 - r0) * 16; i += THREADS) {
    const int r = r0 + (i >> 4), c = i & 15;
    const uint32_t a_ml = smem_u32(sm + S::ML + 2 * r), a_o = s_kv + (r * PITCH + c * 4) * 4;
    const float4 a = k <= 2   ? merge_chunk<2>(a_ml, a_o, k)
                     : k <= 4 ? merge_chunk<4>(a_ml, a_o, k)
                     : k <= 8 ? merge_chunk<8>(a_ml, a_o, k)
                              : merge_chunk<16>(a_ml, a_o, k);
    *reinterpret_cast<float4*>(out_row(r) + c * 4) = a;
  }
  cluster_sync();  // no CTA leaves while a peer reads its shared memory
}

template <int RT>
cudaError_t launch(const Dev& d, int layer, const void* q, void* out, int n_pairs, int n_rb, int k,
                   bool spread, bool early, cudaStream_t s) {
  const float scale = LOG2E / sqrtf((float)d.head_dim);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_pairs * n_rb * k);
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = spread ? ONE_PER_SM : Shape<RT>::SMEM;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (k > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = k;
    attr[n].val.clusterDim.y = 1;
    attr[n].val.clusterDim.z = 1;
    ++n;
  }
  attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[n].val.programmaticStreamSerializationAllowed = 1;
  ++n;
  cfg.attrs = attr;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, &attn_prefill_f32_kernel<RT>, d, layer,
                            static_cast<const float*>(q), static_cast<float*>(out), scale, n_rb, k,
                            (int)early);
}

// Attributes of the kernel, and the largest cluster of it that the device takes, without and
// with the shared memory that spreads its CTAs over the SMs.
template <int RT>
cudaError_t limits(int (&largest)[2]) {
  const void* fn = reinterpret_cast<const void*>(&attn_prefill_f32_kernel<RT>);
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, ONE_PER_SM);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  for (int spread = 0; spread < 2; ++spread) {
    largest[spread] = 1;
    for (int k = MAX_K; k > 1 && largest[spread] == 1; --k) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(k);
      cfg.blockDim = dim3(THREADS);
      cfg.dynamicSmemBytes = spread ? ONE_PER_SM : Shape<RT>::SMEM;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = k;
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      int n = 0;
      e = cudaOccupancyMaxActiveClusters(&n, &attn_prefill_f32_kernel<RT>, &cfg);
      if (e == cudaSuccess && n > 0) largest[spread] = k;
      if (e != cudaSuccess) cudaGetLastError();  // (a size that the device does not take: no error)
    }
  }
  return cudaSuccess;
}

}  // namespace

cudaError_t prefill_f32_limits(Limits* lim) {
  const cudaError_t e = limits<4>(lim->f32_cluster[0]);
  return e != cudaSuccess ? e : limits<9>(lim->f32_cluster[1]);
}

cudaError_t launch_attn_prefill_f32(const Dev& d, const Limits& lim, int layer, const void* q,
                                    void* out, int n_seq, int max_t, int pages_max, bool early,
                                    cudaStream_t s) {
  const int sms = lim.sms;
  // Rows per CTA: 32 (chunks of up to 8 tokens) or 72 (a 17-token unit's 68).
  const int R = max_t * G, n_pairs = n_seq * d.kv_heads;
  const bool small = R <= 32;
  const int n_rb = small ? 1 : (R + 71) / 72;
  // Slices, of two pages each at least: as many as still run at once, 27/32 of the slots of
  // two CTAs per SM (clusters leave gaps; measured at 32 pairs of 65 pages k = 8 27.3 us
  // against 40.8 at 10, at 48 pairs k = 5 38.1 against 49.8 at 6).  Large clusters pay only
  // for few pairs (8 pairs: 15.8 us at 16 against 25.4 at 8; 16 pairs: 23.7 at 12, 29.5 at 16).
  // Calls that need several waves: 3, whose tail is shorter than 1's (192 pairs: 111 against
  // 149 us).
  const int blocks = n_pairs * n_rb;
  const int fit = sms * 27 / 16 / blocks;
  int k = min(blocks <= 8 ? MAX_K : blocks <= 21 ? 12 : 8, fit);
  if (k < 2) k = blocks <= 3 * sms ? 3 : 1;
  const int* largest = lim.f32_cluster[small ? 0 : 1];  // (that the device takes at all)
  k = max(1, min(min(k, largest[0]), pages_max / 2));
  // A small grid's clusters are spread over the SMs (4 pairs: 13.0 against 14.6 us).
  const bool spread = 2 * blocks * k <= sms && k <= largest[1];
  return small ? launch<4>(d, layer, q, out, n_pairs, n_rb, k, spread, early, s)
               : launch<9>(d, layer, q, out, n_pairs, n_rb, k, spread, early, s);
}

}  // namespace kvc
