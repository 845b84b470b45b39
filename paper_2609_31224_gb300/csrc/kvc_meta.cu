// Cache bookkeeping kernels: initialisation, append (positions, units, page
// allocation, RoPE'd K and V writes), online eviction (Sec. 3.3) with
// compaction, and session release.
//
// Allocation rule: pages are taken lowest free id first, in the call's
// session order then token order (append) or session order (evict: all
// sessions' compacted-region pages are allocated before any live page is
// freed).  This makes page tables a deterministic function of the calls.
#include "kvc_launch.cuh"
#include "kvc_rope.cuh"

namespace kvc {

namespace {

constexpr int META_THREADS = 1024;
// Chunks of more tokens are planned by the whole CTA, shorter ones by a warp each (a warp
// takes about 0.4 us per 32 tokens, the CTA about 1.5 us per 1,024).
constexpr int LONG_CHUNK = 256;
constexpr unsigned FULL = 0xFFFFFFFFu;

__device__ inline unsigned lanemask_lt() {
  unsigned m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}
__device__ inline unsigned lanemask_le() {
  unsigned m;
  asm("mov.u32 %0, %%lanemask_le;" : "=r"(m));
  return m;
}

// Block-wide exclusive scan of one int per thread (blockDim.x == 1024).
__device__ int block_exclusive_scan(int v, int* total, int* s_warp) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(FULL, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_warp[warp] = x;
  __syncthreads();
  if (warp == 0) {
    int w = s_warp[lane];
    int xs = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int y = __shfl_up_sync(FULL, xs, o);
      if (lane >= o) xs += y;
    }
    s_warp[lane] = xs - w;  // exclusive warp offsets
    if (lane == 31) s_warp[32] = xs;
  }
  __syncthreads();
  int r = s_warp[warp] + x - v;
  *total = s_warp[32];
  __syncthreads();
  return r;
}

__device__ int block_max(int v, int* s_warp) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(FULL, v, o));
  if (lane == 0) s_warp[warp] = v;
  __syncthreads();
  if (warp == 0) {
    int w = s_warp[lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) w = max(w, __shfl_xor_sync(FULL, w, o));
    if (lane == 0) s_warp[32] = w;
  }
  __syncthreads();
  int r = s_warp[32];
  __syncthreads();
  return r;
}

// Take the k lowest free page ids, mark them used and write them, ascending,
// to d.alloc_list[0..k).  Returns false (and marks nothing) if fewer than k
// pages are free.  Block-uniform result.  The search starts at the first bitmap word
// that can hold a free page: an allocation leaves none below its last one, freeing lowers
// the mark (free_page).
__device__ bool block_alloc_lowest(const Dev& d, int k, int* s_warp) {
  __shared__ int s_found;
  if (k == 0) return true;
  if (threadIdx.x == 0) s_found = 0;
  __syncthreads();
  for (int w0 = d.g->free_word; w0 < d.bitmap_words; w0 += META_THREADS) {
    const int w = w0 + threadIdx.x;
    uint32_t freebits = 0;
    if (w < d.bitmap_words) {
      freebits = ~d.bitmap[w];
      const int64_t first = (int64_t)w * 32;
      if (first + 32 > d.n_pages) {
        const int valid = (int)(d.n_pages - first);
        freebits &= (valid >= 32) ? 0xFFFFFFFFu : ((1u << valid) - 1u);
      }
    }
    int total;
    const int found = s_found;
    const int base = found + block_exclusive_scan(__popc(freebits), &total, s_warp);
    if (w < d.bitmap_words && base < k && freebits) {
      uint32_t take = 0;
      int idx = base;
      uint32_t fb = freebits;
      while (fb && idx < k) {
        const int bit = __ffs(fb) - 1;
        fb &= fb - 1;
        d.alloc_list[idx++] = w * 32 + bit;
        take |= 1u << bit;
      }
      d.bitmap[w] |= take;
    }
    __syncthreads();
    if (threadIdx.x == 0) s_found = min(k, found + total);
    __syncthreads();
    if (s_found >= k) {
      if (threadIdx.x == 0) d.g->free_word = d.alloc_list[k - 1] >> 5;
      return true;
    }
  }
  // Not enough pages: roll back what was marked.
  const int got = s_found;
  for (int i = threadIdx.x; i < got; i += META_THREADS) {
    const int p = d.alloc_list[i];
    atomicAnd(&d.bitmap[p >> 5], ~(1u << (p & 31)));
  }
  __syncthreads();
  return false;
}

__device__ inline void free_page(const Dev& d, int p) {
  atomicAnd(&d.bitmap[p >> 5], ~(1u << (p & 31)));
  atomicMin(&d.g->free_word, p >> 5);
}

__device__ inline bool evictable_type(int t) { return t == KVC_ACOUSTIC || t == KVC_ASR_DELIM; }

// ---------------------------------------------------------------------------
// Initialisation.
// ---------------------------------------------------------------------------
__global__ void init_state_kernel(Dev d) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < d.n_sessions) {
    SessState s = {};
    s.unit_cur = -1;
    d.sess[i] = s;
  }
  if (i < d.bitmap_words) {
    const int64_t first = (int64_t)i * 32;
    uint32_t w = 0;
    if (first + 32 > d.n_pages) {
      const int valid = (int)(d.n_pages - first);
      w = (valid >= 32) ? 0u : ~((1u << valid) - 1u);
    }
    d.bitmap[i] = w;
  }
}

// cos/sin of p * base^(-2i/D), evaluated in binary64 and stored in binary32.
__global__ void init_rope_kernel(Dev d, double base) {
  const int half = d.head_dim / 2;
  const int64_t n = (int64_t)d.max_positions * half;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int p = (int)(idx / half), i = (int)(idx % half);
    const double theta = pow(base, -2.0 * (double)i / (double)d.head_dim);
    double sn, cs;
    sincos((double)p * theta, &sn, &cs);
    d.rope[idx] = make_float2((float)cs, (float)sn);
  }
}

// ---------------------------------------------------------------------------
// Append, part 1 (one CTA): page demand, allocation, positions and units
// (warp ballot over UNIT_BEGIN flags), slot tags, state update and the
// work split of the attention calls that follow.
// ---------------------------------------------------------------------------
// A failed append leaves the state as it was and gives the K/V writer and the
// attention kernels nothing to do.
__device__ void abandon_append(const Dev& d) {
  d.g->total_tokens = 0;
  d.g->n_units = 0;
}

template <int N>
__global__ void __launch_bounds__(META_THREADS) append_plan_kernel(Dev d, AppendArgsT<N> a,
                                                                   const uint8_t* types) {
  __shared__ int s_warp[33];
  __shared__ int s_bad;
  __shared__ int s_total_dec, s_long;
  const int i = threadIdx.x;
  const int n_seq = a.n_seq;
  pdl_wait();
  pdl_launch_dependents();
  if (i == 0) s_bad = 0;
  __syncthreads();

  // 1. Page demand per session (thread i <-> session i of the call).
  int sid = 0, t_len = 0, need = 0;
  SessState st = {};
  if (i < n_seq) {
    sid = a.sessions[i];
    st = d.sess[sid];
    t_len = a.cu[i + 1] - a.cu[i];
    const int tail = st.live_head + st.n_live;
    need = (tail + t_len + PS - 1) / PS - st.n_live_pages;
    if (st.n_live_pages + need > d.max_pages_per_session) atomicOr(&s_bad, KVC_DERR_PAGE_TABLE);
    if (st.pos_next + t_len > d.max_positions) atomicOr(&s_bad, KVC_DERR_POSITION);
  }
  __syncthreads();
  if (s_bad) {
    if (i == 0) {
      set_error(d, s_bad);
      abandon_append(d);
    }
    return;
  }
  int total_need;
  const int off = block_exclusive_scan(need, &total_need, s_warp);
  if (total_need > d.max_alloc || !block_alloc_lowest(d, total_need, s_warp)) {
    if (i == 0) {
      set_error(d, KVC_DERR_POOL);
      abandon_append(d);
    }
    return;
  }
  // 2. New live pages, in call order then token order.
  const int lane = i & 31, warp = i >> 5;
  if (i < n_seq) {
    int32_t* row = d.live_pt + (size_t)sid * d.max_pages_per_session;
    for (int j = 0; j < min(need, LONG_CHUNK / PS + 1); ++j)
      row[st.n_live_pages + j] = d.alloc_list[off + j];
  }
  // Long chunks (a history fed back): the whole CTA takes one session at a time.
  const bool longs = __syncthreads_or(i < n_seq && t_len > LONG_CHUNK);
  for (int q = 0; longs && q < n_seq; ++q) {
    const int tq = a.cu[q + 1] - a.cu[q];
    if (tq <= LONG_CHUNK) continue;
    const int qs = a.sessions[q], g0 = a.cu[q];
    const SessState s0 = d.sess[qs];
    const int tail = s0.live_head + s0.n_live;
    int32_t* row = d.live_pt + (size_t)qs * d.max_pages_per_session;
    if (i == q) s_long = off;
    __syncthreads();
    const int q_need = (tail + tq + PS - 1) / PS - s0.n_live_pages;
    for (int j = i; j < q_need; j += META_THREADS) row[s0.n_live_pages + j] = d.alloc_list[s_long + j];
    __syncthreads();
    int unit_run = s0.unit_cur;
    for (int t0 = 0; t0 < tq; t0 += META_THREADS) {
      const int t = t0 + i;
      const int ty = t < tq ? (int)types[g0 + t] : 0;
      const int slot = tail + t;
      const int gs = t < tq ? row[slot / PS] * PS + (slot % PS) : 0;
      int n_units;
      const int begins = (ty & KVC_UNIT_BEGIN) ? 1 : 0;
      const int unit = unit_run + block_exclusive_scan(begins, &n_units, s_warp) + begins;
      if (t < tq) {
        d.meta_pos[gs] = s0.pos_next + t;
        d.meta_unit[gs] = unit;
        d.meta_type[gs] = (uint8_t)(ty & TYPE_MASK);
        d.tok_slot[g0 + t] = gs;
        d.tok_pos[g0 + t] = s0.pos_next + t;
      }
      unit_run += n_units;
    }
    if (i == 0) {
      SessState s1 = s0;
      s1.pos_next = s0.pos_next + tq;
      s1.unit_cur = unit_run;
      s1.n_live = s0.n_live + tq;
      s1.last_chunk = tq;
      d.sess[qs] = s1;  // n_live_pages updated below by the owning thread
    }
  }

  // 3. Positions, units and slot tags of the others: one warp per session.
  for (int q = warp; q < n_seq; q += META_THREADS / 32) {
    const int qs = a.sessions[q];
    const SessState s0 = d.sess[qs];
    const int tq = a.cu[q + 1] - a.cu[q];
    if (tq > LONG_CHUNK) continue;
    const int g0 = a.cu[q];
    const int tail = s0.live_head + s0.n_live;
    const int32_t* row = d.live_pt + (size_t)qs * d.max_pages_per_session;
    int unit_run = s0.unit_cur;
    for (int t0 = 0; t0 < tq; t0 += 32) {
      const int t = t0 + lane;
      const bool valid = t < tq;
      const int ty = valid ? (int)types[g0 + t] : 0;
      const unsigned flags = __ballot_sync(FULL, valid && (ty & KVC_UNIT_BEGIN));
      const int unit = unit_run + __popc(flags & lanemask_le());
      if (valid) {
        const int slot = tail + t;
        const int gs = row[slot / PS] * PS + (slot % PS);
        d.meta_pos[gs] = s0.pos_next + t;
        d.meta_unit[gs] = unit;
        d.meta_type[gs] = (uint8_t)(ty & TYPE_MASK);
        d.tok_slot[g0 + t] = gs;
        d.tok_pos[g0 + t] = s0.pos_next + t;
      }
      unit_run += __popc(flags);
    }
    __syncwarp();
    if (lane == 0) {
      SessState s1 = s0;
      s1.pos_next = s0.pos_next + tq;
      s1.unit_cur = unit_run;
      s1.n_live = s0.n_live + tq;
      s1.last_chunk = tq;
      d.sess[qs] = s1;  // n_live_pages updated below by the owning thread
    }
  }
  __syncthreads();
  int nb = 0;
  if (i < n_seq) {
    SessState s1 = d.sess[sid];
    s1.n_live_pages = st.n_live_pages + need;
    s1.peak_resident = max(s1.peak_resident, s1.n_hist + s1.n_live);
    d.sess[sid] = s1;
    nb = s1.n_hist_pages + s1.n_live_pages;
    SeqInfo si = {};
    si.sid = sid;
    si.t = t_len;
    si.q_row0 = a.cu[i];
    si.pos_first = st.pos_next;
    si.n_hist = s1.n_hist;
    si.n_hist_pages = s1.n_hist_pages;
    si.live_head = s1.live_head;
    si.n_live = s1.n_live;
    si.n_blocks = nb;
    d.seq[i] = si;
  }
  __syncthreads();
  // 4. Work of the attention calls: the stream-K splits cut the call's (session, kv head,
  // page) units evenly over their CTAs; they need each session's first unit, the total
  // and the largest session.
  {
    int total_units;
    const int ubase = block_exclusive_scan(i < n_seq ? nb * d.kv_heads : 0, &total_units, s_warp);
    const int nb_max = block_max(i < n_seq ? nb : 0, s_warp);
    if (i < n_seq) d.seq[i].unit_base = ubase;
    if (i == 0) {
      s_total_dec = total_units;
      d.g->nb_max = nb_max;
    }
    __syncthreads();
  }
  if (i == 0) {
    d.g->n_seq = n_seq;
    d.g->total_tokens = a.total;
    d.g->n_units = s_total_dec;
    d.g->pages_used += total_need;
  }
}

// Append, part 2: K rotated at its position (rotate-half, binary32 math on
// the binary32 table), V copied, both into the page slots of part 1.  Input layout
// [L][total][Hkv][D]; blockIdx.y is the input layer, cache layer layer0 + blockIdx.y.
// Bound by HBM: a thread takes 16-byte chunk c of the first half of a row of K and V with
// its rotate-half partner, so that its four loads are in flight together, a warp reads
// four whole rows of each (512 B runs) and writes them as whole lines.  The loads depend
// on nothing that part 1 writes and are issued before it ends.  7,900 tokens of 32 layers
// of 8 bfloat16 heads (2.07 GB moved): 299 us, 6.93 TB/s; 588 us with 2-byte K accesses and a
// block per (token, layer).
constexpr int KV_THREADS = 256;
template <typename T>
__global__ void __launch_bounds__(KV_THREADS) append_kv_kernel(Dev d, int total, int layer0,
                                                               const T* k, const T* v) {
  using CK = Chunk16<T>;
  constexpr int VEC = CK::N, KC = 8, HALF = KC * VEC, D = 2 * HALF;
  const int H = d.kv_heads;
  const int idx = blockIdx.x * KV_THREADS + threadIdx.x;
  const int c = idx % KC, row = idx / KC, g = row / H, h = row % H;
  const bool in = g < total;
  pdl_launch_dependents();
  uint4 ka, kb, va, vb;
  if (in) {
    const size_t off = (((size_t)blockIdx.y * total + g) * H + h) * D + c * VEC;
    ka = __ldcs(reinterpret_cast<const uint4*>(k + off));
    kb = __ldcs(reinterpret_cast<const uint4*>(k + off + HALF));
    va = __ldcs(reinterpret_cast<const uint4*>(v + off));
    vb = __ldcs(reinterpret_cast<const uint4*>(v + off + HALF));
  }
  pdl_wait();
  if (!in || g >= d.g->total_tokens) return;  // (the plan kernel failed: error recorded)
  const int gs = d.tok_slot[g], pos = d.tok_pos[g];
  const float4* t4 = reinterpret_cast<const float4*>(d.rope + (size_t)pos * HALF + c * VEC);
  float xa[VEC], xb[VEC], ya[VEC], yb[VEC];
  CK::unpack(ka, xa);
  CK::unpack(kb, xb);
#pragma unroll
  for (int e = 0; e < VEC; e += 2) {
    const float4 cs = t4[e / 2];
    rope_pair(xa[e], xb[e], make_float2(cs.x, cs.y), ya[e], yb[e]);
    rope_pair(xa[e + 1], xb[e + 1], make_float2(cs.z, cs.w), ya[e + 1], yb[e + 1]);
  }
  T* dst = reinterpret_cast<T*>(d.pool) +
           pool_offset_elems(d, gs / PS, layer0 + blockIdx.y, 0, h, gs % PS) + c * VEC;
  T* dv = dst + (size_t)H * PS * D;
  *reinterpret_cast<uint4*>(dst) = CK::pack(ya);
  *reinterpret_cast<uint4*>(dst + HALF) = CK::pack(yb);
  *reinterpret_cast<uint4*>(dv) = va;
  *reinterpret_cast<uint4*>(dv + HALF) = vb;
}

// ---------------------------------------------------------------------------
// Append of exactly one token per session (the decode rounds): the same state and tags as
// the general plan kernel.  append_few_kernel takes calls of up to 32 sessions, lane i of
// its first warp planning session i of the call (page demand, lowest-free allocation in
// call order, position, unit, slot tags, state, the attention calls' work split) with no
// CTA barrier; a one-session call's other threads write its K and V rows of every layer as
// soon as the slot is known, their inputs loaded meanwhile.  append_many_kernel takes the
// larger calls, thread i planning session i.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(META_THREADS) append_few_kernel(Dev d, SeqArgsT<FEW> a,
                                                                  const uint8_t* types, const T* k,
                                                                  const T* v) {
  using CK = Chunk16<T>;
  constexpr int VEC = CK::N, KC = 8, HALF = KC * VEC, D = 2 * HALF;
  constexpr int U = 2;  // K/V items (as in append_kv_kernel) in flight per thread
  __shared__ int s_pages[32];
  __shared__ int s_gs, s_pos;
  const int i = threadIdx.x, lane = i & 31;
  const int n_seq = a.n_seq, H = d.kv_heads;
  pdl_wait();
  pdl_launch_dependents();
  // One session: item idx is chunk idx % 8 of row (layer, head) idx / 8.
  const int n_items = k != nullptr ? d.layers * H * KC : 0;
  uint4 ka[U], kb[U], va[U], vb[U];
  auto load = [&](int base) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int idx = base + u * META_THREADS;
      if (idx < n_items) {
        const size_t off = (size_t)(idx / KC) * D + (idx % KC) * VEC;
        ka[u] = __ldcs(reinterpret_cast<const uint4*>(k + off));
        kb[u] = __ldcs(reinterpret_cast<const uint4*>(k + off + HALF));
        va[u] = __ldcs(reinterpret_cast<const uint4*>(v + off));
        vb[u] = __ldcs(reinterpret_cast<const uint4*>(v + off + HALF));
      }
    }
  };
  load(i);
  if (i < 32) {
    const int mpps = d.max_pages_per_session;
    const bool in = lane < n_seq;
    int sid = 0, need = 0, ty = 0, page = 0, bad = 0;
    SessState st = {};
    if (in) {
      sid = a.sessions[lane];
      ty = (int)types[lane];
      st = d.sess[sid];
      const int tail = st.live_head + st.n_live;
      need = (tail + PS) / PS - st.n_live_pages;
      if (need < 0 || need > 1 || st.n_live_pages + need > mpps) bad |= KVC_DERR_PAGE_TABLE;
      if (st.pos_next + 1 > d.max_positions) bad |= KVC_DERR_POSITION;
      if (need == 0) page = d.live_pt[(size_t)sid * mpps + tail / PS];
    }
    bad = __reduce_or_sync(FULL, bad);
    const unsigned needs = __ballot_sync(FULL, need > 0);
    const int total_need = __popc(needs);
    if (!bad && total_need > 0) {
      // The total_need lowest free pages, 32 bitmap words at a time.
      int found = 0;
      for (int w0 = d.g->free_word; w0 < d.bitmap_words && found < total_need; w0 += 32) {
        const int w = w0 + lane;
        uint32_t freebits = w < d.bitmap_words ? ~d.bitmap[w] : 0u;
        const int64_t first = (int64_t)w * 32;
        if (freebits && first + 32 > d.n_pages) {
          const int valid = (int)(d.n_pages - first);
          freebits &= valid <= 0 ? 0u : (1u << valid) - 1u;
        }
        int base = __popc(freebits);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(FULL, base, o);
          if (lane >= o) base += y;
        }
        const int sum = __shfl_sync(FULL, base, 31);
        int idx = found + base - __popc(freebits);
        for (uint32_t fb = freebits; fb && idx < total_need; fb &= fb - 1)
          s_pages[idx++] = w * 32 + __ffs(fb) - 1;
        found += sum;
      }
      __syncwarp();
      if (found < total_need || total_need > d.max_alloc) {
        bad = KVC_DERR_POOL;
      } else if (lane < total_need) {
        const int p = s_pages[lane];
        atomicOr(&d.bitmap[p >> 5], 1u << (p & 31));
        if (lane == total_need - 1) d.g->free_word = p >> 5;
      }
    }
    if (bad) {
      if (lane == 0) {
        set_error(d, bad);
        abandon_append(d);
        s_gs = -1;
      }
    } else {
      int nb = 0;
      SeqInfo si = {};
      if (in) {
        const int tail = st.live_head + st.n_live;
        if (need) {
          page = s_pages[__popc(needs & lanemask_lt())];
          d.live_pt[(size_t)sid * mpps + st.n_live_pages] = page;
        }
        const int gs = page * PS + tail % PS;
        const int unit = st.unit_cur + ((ty & KVC_UNIT_BEGIN) ? 1 : 0);
        if (lane == 0) {
          s_gs = gs;
          s_pos = st.pos_next;
        }
        d.meta_pos[gs] = st.pos_next;
        d.meta_unit[gs] = unit;
        d.meta_type[gs] = (uint8_t)(ty & TYPE_MASK);
        d.tok_slot[lane] = gs;
        d.tok_pos[lane] = st.pos_next;
        SessState s1 = st;
        s1.pos_next = st.pos_next + 1;
        s1.unit_cur = unit;
        s1.n_live = st.n_live + 1;
        s1.last_chunk = 1;
        s1.n_live_pages = st.n_live_pages + need;
        s1.peak_resident = max(st.peak_resident, s1.n_hist + s1.n_live);
        d.sess[sid] = s1;
        nb = s1.n_hist_pages + s1.n_live_pages;
        si.sid = sid;
        si.t = 1;
        si.q_row0 = lane;
        si.pos_first = st.pos_next;
        si.n_hist = s1.n_hist;
        si.n_hist_pages = s1.n_hist_pages;
        si.live_head = s1.live_head;
        si.n_live = s1.n_live;
        si.n_blocks = nb;
      }
      int units = nb * H;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, units, o);
        if (lane >= o) units += y;
      }
      if (in) {
        si.unit_base = units - nb * H;
        d.seq[lane] = si;
      }
      const int total_units = __shfl_sync(FULL, units, 31);
      const int nb_max = __reduce_max_sync(FULL, nb);
      if (lane == 0) {
        d.g->n_seq = n_seq;
        d.g->total_tokens = n_seq;
        d.g->n_units = total_units;
        d.g->nb_max = nb_max;
        d.g->pages_used += total_need;
      }
    }
  }
  if (n_items == 0) return;
  __syncthreads();
  const int gs = s_gs;
  if (gs < 0) return;
  T* pool = reinterpret_cast<T*>(d.pool);
  for (int base = i; base < n_items;) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int idx = base + u * META_THREADS;
      if (idx >= n_items) break;
      const int c = idx % KC, h = idx / KC % H, l = idx / KC / H;
      const float4* t4 = reinterpret_cast<const float4*>(d.rope + (size_t)s_pos * HALF + c * VEC);
      float xa[VEC], xb[VEC], ya[VEC], yb[VEC];
      CK::unpack(ka[u], xa);
      CK::unpack(kb[u], xb);
#pragma unroll
      for (int e = 0; e < VEC; e += 2) {
        const float4 cs = t4[e / 2];
        rope_pair(xa[e], xb[e], make_float2(cs.x, cs.y), ya[e], yb[e]);
        rope_pair(xa[e + 1], xb[e + 1], make_float2(cs.z, cs.w), ya[e + 1], yb[e + 1]);
      }
      T* dst = pool + pool_offset_elems(d, gs / PS, l, 0, h, gs % PS) + c * VEC;
      T* dv = dst + (size_t)H * PS * D;
      *reinterpret_cast<uint4*>(dst) = CK::pack(ya);
      *reinterpret_cast<uint4*>(dst + HALF) = CK::pack(yb);
      *reinterpret_cast<uint4*>(dv) = va[u];
      *reinterpret_cast<uint4*>(dv + HALF) = vb[u];
    }
    base += U * META_THREADS;
    if (base < n_items) load(base);
  }
}

__global__ void __launch_bounds__(META_THREADS) append_many_kernel(Dev d, AppendArgs a,
                                                                   const uint8_t* types) {
  __shared__ int s_warp[33];
  __shared__ int s_bad;
  const int i = threadIdx.x;
  const int n_seq = a.n_seq;
  const int mpps = d.max_pages_per_session;
  pdl_wait();
  pdl_launch_dependents();
  if (i == 0) s_bad = 0;
  __syncthreads();

  int sid = 0, need = 0, ty = 0, page = 0;
  SessState st = {};
  if (i < n_seq) {
    sid = a.sessions[i];
    st = d.sess[sid];
    ty = (int)types[i];
    const int tail = st.live_head + st.n_live;
    need = (tail + PS) / PS - st.n_live_pages;
    if (need < 0 || need > 1 || st.n_live_pages + need > mpps)
      atomicOr(&s_bad, KVC_DERR_PAGE_TABLE);
    if (st.pos_next + 1 > d.max_positions) atomicOr(&s_bad, KVC_DERR_POSITION);
    if (need == 0) page = d.live_pt[(size_t)sid * mpps + tail / PS];
  }
  __syncthreads();
  if (s_bad) {
    if (i == 0) {
      set_error(d, s_bad);
      abandon_append(d);
    }
    return;
  }
  int total_need;
  const int off = block_exclusive_scan(need, &total_need, s_warp);
  if (total_need > 0 && (total_need > d.max_alloc || !block_alloc_lowest(d, total_need, s_warp))) {
    if (i == 0) {
      set_error(d, KVC_DERR_POOL);
      abandon_append(d);
    }
    return;
  }
  int nb = 0;
  SeqInfo si = {};
  if (i < n_seq) {
    const int tail = st.live_head + st.n_live;
    if (need) {
      page = d.alloc_list[off];
      d.live_pt[(size_t)sid * mpps + st.n_live_pages] = page;
    }
    const int gs = page * PS + tail % PS;
    const int unit = st.unit_cur + ((ty & KVC_UNIT_BEGIN) ? 1 : 0);
    d.meta_pos[gs] = st.pos_next;
    d.meta_unit[gs] = unit;
    d.meta_type[gs] = (uint8_t)(ty & TYPE_MASK);
    d.tok_slot[i] = gs;
    d.tok_pos[i] = st.pos_next;
    SessState s1 = st;
    s1.pos_next = st.pos_next + 1;
    s1.unit_cur = unit;
    s1.n_live = st.n_live + 1;
    s1.last_chunk = 1;
    s1.n_live_pages = st.n_live_pages + need;
    s1.peak_resident = max(st.peak_resident, s1.n_hist + s1.n_live);
    d.sess[sid] = s1;
    nb = s1.n_hist_pages + s1.n_live_pages;
    si.sid = sid;
    si.t = 1;
    si.q_row0 = i;
    si.pos_first = st.pos_next;
    si.n_hist = s1.n_hist;
    si.n_hist_pages = s1.n_hist_pages;
    si.live_head = s1.live_head;
    si.n_live = s1.n_live;
    si.n_blocks = nb;
  }
  // Split-K work of the attention calls (as in append_plan_kernel).
  int total_units;
  const int ubase = block_exclusive_scan(i < n_seq ? nb * d.kv_heads : 0, &total_units, s_warp);
  const int nb_max = block_max(i < n_seq ? nb : 0, s_warp);
  if (i < n_seq) {
    si.unit_base = ubase;
    d.seq[i] = si;
  }
  __syncthreads();
  if (i == 0) {
    d.g->n_seq = n_seq;
    d.g->total_tokens = n_seq;
    d.g->n_units = total_units;
    d.g->nb_max = nb_max;
    d.g->pages_used += total_need;
  }
}

// ---------------------------------------------------------------------------
// Evict, part 1 (one CTA): the rule of Sec. 3.3 for each session (one warp
// each), compacted-region page allocation, survivor move list, slot tags,
// freeing of consumed live pages, state update.
// ---------------------------------------------------------------------------
struct LiveSlot {
  int unit, type, gs, pos;
};

__device__ inline LiveSlot live_slot(const Dev& d, const SessState& st, const int32_t* row,
                                     int j) {
  const int slot = st.live_head + j;
  const int gs = row[slot / PS] * PS + (slot % PS);
  LiveSlot r;
  r.gs = gs;
  r.unit = d.meta_unit[gs];
  r.type = d.meta_type[gs];
  r.pos = d.meta_pos[gs];
  return r;
}

// Whether a slot inside the consumed live prefix is dropped: its type under the
// rule of Sec. 3.3 and its position-granular variant; its position under the
// sink + recent variant.
__device__ inline bool slot_evicted(const Dev& d, const LiveSlot& ls) {
  if (d.policy == KVC_POLICY_SINK_RECENT) return ls.pos >= d.sink;
  return ls.unit >= 0 && evictable_type(ls.type);
}

// Length of the live prefix a position-granular evict consumes: up to and
// including the need-th evictable slot of a unit <= lim (fewer if fewer exist;
// those units are a prefix of the live region).  One warp.
__device__ int position_variant_end(const Dev& d, const SessState& st, const int32_t* row,
                                    int lim, int need, int lane) {
  int cnt = 0, end = 0;
  for (int w0 = 0; w0 < st.n_live; w0 += 32) {
    const int j = w0 + lane;
    const bool valid = j < st.n_live;
    LiveSlot ls = {INT_MAX, 0, 0, 0};
    if (valid) ls = live_slot(d, st, row, j);
    const unsigned stop = __ballot_sync(FULL, !valid || ls.unit > lim);
    const int first_stop = stop ? __ffs(stop) - 1 : 32;
    const unsigned ev = __ballot_sync(FULL, lane < first_stop && ls.unit >= 0 &&
                                                evictable_type(ls.type));
    const int n_ev = __popc(ev);
    if (cnt + n_ev >= need) {
      unsigned m = ev;  // drop the (need - cnt - 1) lowest set bits: the next is the need-th
      for (int k = need - cnt - 1; k > 0; --k) m &= m - 1;
      return w0 + (__ffs(m) - 1) + 1;
    }
    if (ev) end = w0 + (31 - __clz(ev)) + 1;
    cnt += n_ev;
    if (stop) break;
  }
  return end;
}

// Length of the live prefix a sink + recent evict consumes: every live slot
// whose position is below pos_next - recent (positions ascend along the region).
__device__ int sink_recent_end(const Dev& d, const SessState& st, const int32_t* row,
                               int lane) {
  const int hi = st.pos_next - d.recent;
  int end = 0;
  for (int w0 = 0; w0 < st.n_live; w0 += 32) {
    const int j = w0 + lane;
    const bool in = j < st.n_live && live_slot(d, st, row, j).pos < hi;
    const unsigned b = __ballot_sync(FULL, in);
    end += __popc(b);
    if (b != FULL) break;
  }
  return end;
}

template <int N>
__global__ void __launch_bounds__(META_THREADS) evict_plan_kernel(Dev d, SeqArgsT<N> a,
                                                                  int64_t* resident_out,
                                                                  int64_t* used_out) {
  __shared__ int s_warp[33];
  __shared__ int s_end[MAX_SEQ], s_surv[MAX_SEQ], s_nev[MAX_SEQ];
  __shared__ int s_hneed[MAX_SEQ], s_hoff[MAX_SEQ], s_moff[MAX_SEQ];
  __shared__ int s_bad;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n_seq = a.n_seq;
  pdl_wait();
  pdl_launch_dependents();
  if (tid == 0) s_bad = 0;

  // Phase 1: plan.  For live slot j with unit u >= 0 the unit-level test is
  //   u <= unit_cur - W  and  R0 - (evictable positions before u's first slot) > B,
  // which holds for a prefix of the units; u* is the newest unit with an
  // evictable position that passes it, and `end` is the live prefix of units <= u*.
  for (int q = warp; q < n_seq; q += META_THREADS / 32) {
    const int sid = a.sessions[q];
    const SessState st = d.sess[sid];
    const int32_t* row = d.live_pt + (size_t)sid * d.max_pages_per_session;
    const int r0 = st.n_hist + st.n_live;
    const int lim = st.unit_cur - d.window;
    int ustar = -2;
    if (d.policy == KVC_POLICY_UNIT && d.budget >= 0 && (int64_t)r0 > d.budget &&
        st.n_live > 0) {
      int e_before = 0;        // evictable slots before this window
      int prev_unit = INT_MIN; // unit of the slot just before this window
      int e_at_prev_start = 0; // evictable count before prev_unit's first slot
      for (int w0 = 0; w0 < st.n_live; w0 += 32) {
        const int j = w0 + lane;
        const bool valid = j < st.n_live;
        LiveSlot ls = {INT_MAX, 0, 0, 0};
        if (valid) ls = live_slot(d, st, row, j);
        const bool ev = valid && ls.unit >= 0 && evictable_type(ls.type);
        const unsigned bal_ev = __ballot_sync(FULL, ev);
        const int e_excl = e_before + __popc(bal_ev & lanemask_lt());
        int up = __shfl_up_sync(FULL, ls.unit, 1);
        if (lane == 0) up = prev_unit;
        const unsigned starts = __ballot_sync(FULL, valid && ls.unit != up);
        const unsigned mine = starts & lanemask_le();
        const int src = mine ? 31 - __clz(mine) : 0;
        const int e_src = __shfl_sync(FULL, e_excl, src);
        const int e_ustart = mine ? e_src : e_at_prev_start;
        const bool cond = (ls.unit < 0) ||
                          (ls.unit <= lim && (int64_t)(r0 - e_ustart) > d.budget);
        const unsigned stops = __ballot_sync(FULL, valid && !cond);
        const int first_stop = stops ? __ffs(stops) - 1 : 32;
        int cand = (lane < first_stop && ev) ? ls.unit : -2;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) cand = max(cand, __shfl_xor_sync(FULL, cand, o));
        ustar = max(ustar, cand);
        if (stops) break;
        const int last = min(31, st.n_live - 1 - w0);
        prev_unit = __shfl_sync(FULL, ls.unit, last);
        e_at_prev_start = __shfl_sync(FULL, e_ustart, last);
        e_before += __popc(bal_ev);
      }
    }
    // The consumed live prefix: units <= u* under the rule; for the variants its
    // length is decided first.
    int end = 0, surv = 0, nev = 0;
    int vend = -1;
    if (d.policy == KVC_POLICY_POSITION) {
      vend = (d.budget >= 0 && (int64_t)r0 > d.budget)
                 ? position_variant_end(d, st, row, lim, (int)(r0 - d.budget), lane)
                 : 0;
    } else if (d.policy == KVC_POLICY_SINK_RECENT) {
      vend = sink_recent_end(d, st, row, lane);
    }
    if (ustar >= 0 || vend > 0) {
      for (int w0 = 0; w0 < st.n_live; w0 += 32) {
        const int j = w0 + lane;
        const bool valid = j < st.n_live;
        LiveSlot ls = {INT_MAX, 0, 0, 0};
        if (valid) ls = live_slot(d, st, row, j);
        const bool in = valid && (vend >= 0 ? j < vend : ls.unit <= ustar);
        const bool ev = in && slot_evicted(d, ls);
        const unsigned bin = __ballot_sync(FULL, in);
        end += __popc(bin);
        nev += __popc(__ballot_sync(FULL, ev));
        surv += __popc(__ballot_sync(FULL, in && !ev));
        if (bin != FULL) break;
      }
    }
    if (lane == 0) {
      s_end[q] = end;
      s_surv[q] = surv;
      s_nev[q] = nev;
    }
  }
  __syncthreads();

  // Phase 2: compacted-region page demand, move offsets, allocation.
  int hneed = 0, surv = 0;
  if (tid < n_seq) {
    const SessState st = d.sess[a.sessions[tid]];
    surv = s_surv[tid];
    hneed = (st.n_hist + surv + PS - 1) / PS - st.n_hist_pages;
    if (st.n_hist_pages + hneed > d.max_pages_per_session) atomicOr(&s_bad, KVC_DERR_PAGE_TABLE);
  }
  int total_h, total_moves;
  const int hoff = block_exclusive_scan(hneed, &total_h, s_warp);
  const int moff = block_exclusive_scan(surv, &total_moves, s_warp);
  if (tid < n_seq) {
    s_hneed[tid] = hneed;
    s_hoff[tid] = hoff;
    s_moff[tid] = moff;
  }
  if (tid == 0 && total_moves > d.max_moves) s_bad |= KVC_DERR_MOVES;
  if (tid == 0 && total_h > d.max_alloc) s_bad |= KVC_DERR_POOL;
  __syncthreads();
  if (s_bad) {
    if (tid == 0) {
      set_error(d, s_bad);
      d.g->n_moves = 0;
      *used_out = d.g->pages_used;
    }
    return;
  }
  if (!block_alloc_lowest(d, total_h, s_warp)) {
    if (tid == 0) {
      set_error(d, KVC_DERR_POOL);
      d.g->n_moves = 0;
      *used_out = d.g->pages_used;
    }
    return;
  }

  // Phase 3: one warp per session.
  __shared__ int s_freed;
  if (tid == 0) s_freed = 0;
  __syncthreads();
  for (int q = warp; q < n_seq; q += META_THREADS / 32) {
    const int sid = a.sessions[q];
    const SessState st = d.sess[sid];
    int32_t* hrow = d.hist_pt + (size_t)sid * d.max_pages_per_session;
    int32_t* lrow = d.live_pt + (size_t)sid * d.max_pages_per_session;
    const int end = s_end[q];
    for (int j = lane; j < s_hneed[q]; j += 32)
      hrow[st.n_hist_pages + j] = d.alloc_list[s_hoff[q] + j];
    __syncwarp();
    int done = 0;  // survivors placed so far
    for (int w0 = 0; w0 < end; w0 += 32) {
      const int j = w0 + lane;
      const bool in = j < end;
      LiveSlot ls = {0, 0, 0, 0};
      if (in) ls = live_slot(d, st, lrow, j);
      const bool sv = in && !slot_evicted(d, ls);
      const unsigned bal = __ballot_sync(FULL, sv);
      if (sv) {
        const int k = done + __popc(bal & lanemask_lt());
        const int di = st.n_hist + k;
        const int dgs = hrow[di / PS] * PS + (di % PS);
        d.moves[s_moff[q] + k] = make_int2(ls.gs, dgs);
        d.meta_pos[dgs] = d.meta_pos[ls.gs];
        d.meta_unit[dgs] = ls.unit;
        d.meta_type[dgs] = (uint8_t)ls.type;
      }
      done += __popc(bal);
    }
    __syncwarp();
    const int consumed = st.live_head + end;
    const int nfree = consumed / PS;
    for (int j = lane; j < nfree; j += 32) {
      free_page(d, lrow[j]);
    }
    __syncwarp();
    const int remain = st.n_live_pages - nfree;
    if (nfree > 0) {
      constexpr int U = 8;  // loads in flight per lane
      for (int j0 = 0; j0 < remain; j0 += 32 * U) {
        int v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int j = j0 + 32 * u + lane;
          v[u] = j < remain ? lrow[j + nfree] : 0;
        }
        __syncwarp();
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int j = j0 + 32 * u + lane;
          if (j < remain) lrow[j] = v[u];
        }
        __syncwarp();
      }
    }
    if (lane == 0) {
      SessState s1 = st;
      s1.n_hist = st.n_hist + s_surv[q];
      s1.n_hist_pages = st.n_hist_pages + s_hneed[q];
      s1.live_head = consumed - nfree * PS;
      s1.n_live = st.n_live - end;
      s1.n_live_pages = remain;
      s1.n_evicted = st.n_evicted + s_nev[q];
      d.sess[sid] = s1;
      if (resident_out) resident_out[q] = (int64_t)(s1.n_hist + s1.n_live);
      atomicAdd(&s_freed, nfree);
    }
  }
  __syncthreads();
  if (tid == 0) {
    d.g->n_moves = total_moves;
    *used_out = d.g->pages_used += total_h - s_freed;
  }
}

// Evict, part 2: move survivors' K/V for every layer, kv slot and head.
// Work unit: 16 bytes; grid-stride over moves x L x 2 x Hkv x (D*esz/16).
__global__ void __launch_bounds__(256) evict_copy_kernel(Dev d) {
  pdl_wait();
  pdl_launch_dependents();
  const int n_moves = d.g->n_moves;
  const int vec_per_row = d.head_dim * d.esz / 16;
  const int rows_per_move = d.layers * 2 * d.kv_heads;
  const int64_t total = (int64_t)n_moves * rows_per_move * vec_per_row;
  for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < total;
       u += (int64_t)gridDim.x * blockDim.x) {
    const int v = (int)(u % vec_per_row);
    const int64_t r = u / vec_per_row;
    const int rr = (int)(r % rows_per_move);
    const int m = (int)(r / rows_per_move);
    const int h = rr % d.kv_heads;
    const int kv = (rr / d.kv_heads) % 2;
    const int l = rr / (2 * d.kv_heads);
    const int2 mv = d.moves[m];
    const size_t so = pool_offset_elems(d, mv.x / PS, l, kv, h, mv.x % PS) * d.esz;
    const size_t dof = pool_offset_elems(d, mv.y / PS, l, kv, h, mv.y % PS) * d.esz;
    const uint4 x = *reinterpret_cast<const uint4*>(d.pool + so + (size_t)v * 16);
    *reinterpret_cast<uint4*>(d.pool + dof + (size_t)v * 16) = x;
  }
}

// ---------------------------------------------------------------------------
// Transcript export (Sec. 4.2): one session's retained TRANSCRIPT positions in
// retained (= position) order.  Part 1 (one CTA): compaction of the retained
// slots by type (block scan); the global slots go to the move list, used as
// scratch, and the positions to pos_out.  Part 2: K and V rows of every layer.
//
// Part 1 is bound by its rounds of dependent loads (page list, type, position)
// and scans: a thread takes GATHER slots in a row, so that a round covers
// GATHER * META_THREADS slots with its loads in flight together.
// An export of 4,100 slots of one bfloat16 layer: 14.1 -> 6.6 us, of 13,700 slots 26.7 -> 12.7,
// against a slot per thread and round and each kernel waiting for the end of the one before.
// ---------------------------------------------------------------------------
constexpr int GATHER = 8;

__global__ void __launch_bounds__(META_THREADS) transcript_gather_kernel(Dev d, int sid, int cap,
                                                                         int32_t* pos_out,
                                                                         int32_t* count) {
  pdl_wait();
  pdl_launch_dependents();
  __shared__ int s_warp[33];
  const SessState st = d.sess[sid];
  const int n = st.n_hist + st.n_live;
  const int32_t* hrow = d.hist_pt + (size_t)sid * d.max_pages_per_session;
  const int32_t* lrow = d.live_pt + (size_t)sid * d.max_pages_per_session;
  int done = 0;
  for (int b0 = 0; b0 < n; b0 += GATHER * META_THREADS) {
    int gs[GATHER];
#pragma unroll
    for (int e = 0; e < GATHER; ++e) {
      const int i = b0 + GATHER * (int)threadIdx.x + e;
      const int j = st.live_head + i - st.n_hist;
      gs[e] = i >= n          ? -1
              : i < st.n_hist ? hrow[i / PS] * PS + i % PS
                              : lrow[j / PS] * PS + j % PS;
    }
    unsigned tr = 0;
#pragma unroll
    for (int e = 0; e < GATHER; ++e)
      tr |= (unsigned)(gs[e] >= 0 && d.meta_type[gs[e]] == KVC_TRANSCRIPT) << e;
    int total;
    int idx = done + block_exclusive_scan(__popc(tr), &total, s_warp);
#pragma unroll
    for (int e = 0; e < GATHER; ++e) {
      if (!(tr >> e & 1)) continue;
      if (idx < cap) {
        pos_out[idx] = d.meta_pos[gs[e]];
        d.moves[idx] = make_int2(gs[e], 0);
      }
      ++idx;
    }
    done += total;
  }
  if (threadIdx.x == 0) {
    *count = done;
    d.g->n_moves = min(done, cap);
  }
}

// Rows [L][cap][Hkv][D] of K and V.  A warp takes the K or V rows of all heads of one
// position of one layer, four 16-byte loads of a lane in flight before their stores.
// 615 positions of 32 bfloat16 layers (161 MB read and written, 24 us at 6.8 TB/s): 48.5 ->
// 32.1 us with part 1, against one load in flight per thread.
__global__ void __launch_bounds__(256) transcript_copy_kernel(Dev d, int cap, uint8_t* k_out,
                                                              uint8_t* v_out) {
  pdl_wait();
  pdl_launch_dependents();
  constexpr int BATCH = 4;
  const int n = d.g->n_moves, lane = threadIdx.x & 31;
  const int vec_per_row = d.head_dim * d.esz / 16, n_vec = d.kv_heads * vec_per_row;
  const int64_t total = (int64_t)n * d.layers * 2;
  const int64_t n_warps = (int64_t)gridDim.x * (blockDim.x / 32);
  for (int64_t u = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / 32; u < total; u += n_warps) {
    const int lk = (int)(u / n), i = (int)(u - (int64_t)lk * n), l = lk / 2, kv = lk % 2;
    const int gs = d.moves[i].x;
    const uint8_t* src = d.pool + pool_offset_elems(d, gs / PS, l, kv, 0, gs % PS) * d.esz;
    uint8_t* dst = (kv ? v_out : k_out) + ((size_t)l * cap + i) * n_vec * 16;
    for (int v0 = lane; v0 < n_vec; v0 += 32 * BATCH) {
      uint4 x[BATCH];
#pragma unroll
      for (int e = 0; e < BATCH; ++e) {
        const int v = v0 + 32 * e, h = v / vec_per_row;
        // (A head's rows are PS rows apart in a page.)
        if (v < n_vec)
          x[e] = *reinterpret_cast<const uint4*>(
              src + ((size_t)h * PS * vec_per_row + (v - h * vec_per_row)) * 16);
      }
#pragma unroll
      for (int e = 0; e < BATCH; ++e) {
        const int v = v0 + 32 * e;
        if (v < n_vec) *reinterpret_cast<uint4*>(dst + (size_t)v * 16) = x[e];
      }
    }
  }
}

// Release (one CTA): free every page of the listed sessions and reset them.
__global__ void __launch_bounds__(META_THREADS) release_kernel(Dev d, SeqArgs a,
                                                               int64_t* used_out) {
  __shared__ int s_freed;
  if (threadIdx.x == 0) s_freed = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int q = warp; q < a.n_seq; q += META_THREADS / 32) {
    const int sid = a.sessions[q];
    const SessState st = d.sess[sid];
    const int32_t* hrow = d.hist_pt + (size_t)sid * d.max_pages_per_session;
    const int32_t* lrow = d.live_pt + (size_t)sid * d.max_pages_per_session;
    for (int j = lane; j < st.n_hist_pages; j += 32) free_page(d, hrow[j]);
    for (int j = lane; j < st.n_live_pages; j += 32) free_page(d, lrow[j]);
    __syncwarp();
    if (lane == 0) {
      SessState s = {};
      s.unit_cur = -1;
      d.sess[sid] = s;
      atomicAdd(&s_freed, st.n_hist_pages + st.n_live_pages);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) *used_out = d.g->pages_used -= s_freed;
}

}  // namespace

cudaError_t launch_init(const Dev& d, double rope_base, cudaStream_t s) {
  const int n = max(d.n_sessions, d.bitmap_words);
  init_state_kernel<<<(n + 255) / 256, 256, 0, s>>>(d);
  init_rope_kernel<<<1024, 256, 0, s>>>(d, rope_base);
  return cudaGetLastError();
}

// Every kernel below may start while the one before it in the stream finishes (it waits for
// that one before it reads anything but the caller's inputs), so that a chain of short
// kernels does not pay a full launch each.
cudaError_t launch_append(const Dev& d, const AppendArgs& a, const uint8_t* types, const void* k,
                          const void* v, bool single, cudaStream_t s) {
  cudaError_t e;
  if (single && a.n_seq <= FEW) {
    // One CTA writes the K/V rows only for a one-session call (a few hundred KiB at
    // most); larger calls spread the rows over append_kv_kernel's grid.
    const bool fuse_kv = a.n_seq == 1 && k != nullptr;
    const dim3 block(fuse_kv ? META_THREADS : 32);
    SeqArgsT<FEW> few;
    few.n_seq = a.n_seq;
    for (int i = 0; i < a.n_seq; ++i) few.sessions[i] = a.sessions[i];
    if (d.esz == 2)
      e = launch_ex(&append_few_kernel<__nv_bfloat16>, dim3(1), block, 0, s, true, d, few, types,
                    static_cast<const __nv_bfloat16*>(fuse_kv ? k : nullptr),
                    static_cast<const __nv_bfloat16*>(fuse_kv ? v : nullptr));
    else
      e = launch_ex(&append_few_kernel<float>, dim3(1), block, 0, s, true, d, few, types,
                    static_cast<const float*>(fuse_kv ? k : nullptr),
                    static_cast<const float*>(fuse_kv ? v : nullptr));
    if (fuse_kv) return e;
  } else if (single) {
    e = launch_ex(&append_many_kernel, dim3(1), dim3(META_THREADS), 0, s, true, d, a, types);
  } else if (a.n_seq <= FEW) {
    AppendArgsT<FEW> few;
    few.n_seq = a.n_seq;
    few.total = a.total;
    for (int i = 0; i < a.n_seq; ++i) few.sessions[i] = a.sessions[i];
    for (int i = 0; i <= a.n_seq; ++i) few.cu[i] = a.cu[i];
    e = launch_ex(&append_plan_kernel<FEW>, dim3(1), dim3(META_THREADS), 0, s, true, d, few, types);
  } else {
    e = launch_ex(&append_plan_kernel<MAX_SEQ>, dim3(1), dim3(META_THREADS), 0, s, true, d, a, types);
  }
  if (e != cudaSuccess || k == nullptr) return e;  // plan only: layers follow one by one
  return launch_append_layers(d, a.total, 0, d.layers, k, v, true, s);
}

cudaError_t launch_append_layers(const Dev& d, int total, int layer0, int n_layers, const void* k,
                                 const void* v, bool after_plan, cudaStream_t s) {
  const dim3 grid(((int64_t)total * d.kv_heads * 8 + KV_THREADS - 1) / KV_THREADS, n_layers);
  // Right behind its plan kernel the launch may start early: k and v were complete before
  // the plan kernel could start.
  if (d.esz == 2)
    return launch_ex(&append_kv_kernel<__nv_bfloat16>, grid, dim3(KV_THREADS), 0, s, after_plan, d,
                     total, layer0, static_cast<const __nv_bfloat16*>(k),
                     static_cast<const __nv_bfloat16*>(v));
  return launch_ex(&append_kv_kernel<float>, grid, dim3(KV_THREADS), 0, s, after_plan, d, total,
                   layer0, static_cast<const float*>(k), static_cast<const float*>(v));
}

// used_out: the pages in use afterwards are written there (pinned host memory).
cudaError_t launch_evict(const Dev& d, const SeqArgs& a, int64_t* resident_out, int64_t* used_out,
                         int sms, cudaStream_t s) {
  cudaError_t e;
  if (a.n_seq <= FEW) {
    SeqArgsT<FEW> few;
    few.n_seq = a.n_seq;
    for (int i = 0; i < a.n_seq; ++i) few.sessions[i] = a.sessions[i];
    e = launch_ex(&evict_plan_kernel<FEW>, dim3(1), dim3(META_THREADS), 0, s, true, d, few,
                  resident_out, used_out);
  } else {
    e = launch_ex(&evict_plan_kernel<MAX_SEQ>, dim3(1), dim3(META_THREADS), 0, s, true, d, a,
                  resident_out, used_out);
  }
  if (e != cudaSuccess) return e;
  return launch_ex(&evict_copy_kernel, dim3(sms * 4), dim3(256), 0, s, true, d);
}

cudaError_t launch_transcript(const Dev& d, int session, int cap, int32_t* pos_out, void* k_out,
                              void* v_out, int32_t* count, cudaStream_t s) {
  cudaError_t e = launch_ex(&transcript_gather_kernel, dim3(1), dim3(META_THREADS), 0, s, true, d,
                            session, cap, pos_out, count);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return launch_ex(&transcript_copy_kernel, dim3(sms * 4), dim3(256), 0, s, true, d, cap,
                   static_cast<uint8_t*>(k_out), static_cast<uint8_t*>(v_out));
}

cudaError_t launch_release(const Dev& d, const SeqArgs& a, int64_t* used_out, cudaStream_t s) {
  release_kernel<<<1, META_THREADS, 0, s>>>(d, a, used_out);
  return cudaGetLastError();
}

}  // namespace kvc
