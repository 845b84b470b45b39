// Chunked-prefill GQA attention on the 5th-generation tensor cores (tcgen05 +
// TMEM), bfloat16 K/V/q, fp32 softmax and accumulation.
//
// A segment is a run of pages of one (session, KV head) pair; the pair's T*G query rows
// (T <= 32 tokens, G = 4 heads) form the M = 128 rows of an MMA tile, the rows past T*G
// being zero padding.  Two ways to cut a call into segments:
//   - pair split (CLUSTER): each pair's pages are cut into k slices, one CTA each.  The k
//     CTAs of a pair are a thread-block cluster: every CTA sends its partial rows (O, max,
//     sum) to the CTAs that own them through distributed shared memory, and each merges
//     and writes its share of the rows;
//   - stream-K: the call's (session, KV head, page) units are cut into equal contiguous
//     ranges, one per CTA; a pair split over several CTAs is merged by the last of them to
//     finish (log-sum-exp over partial states in global memory).
// Warp roles in one CTA (384 threads, one CTA per SM):
//   warps 0, 1 producers: 2-D TMA loads (128-byte swizzle) of the K (warp 0) and V (warp 1)
//              tiles of 4 pages (64 keys) per stage, one box per lane, into a ring whose K
//              and V halves are released separately;
//   warps 2, 3 MMA issuers: one elected thread each, warp 2 S = Q K^T (N = 64, Q from
//              TMEM, K from shared memory), warp 3 O += P V (N = 128, P from TMEM, V from
//              shared memory); completion is signalled with tcgen05.commit on mbarriers;
//   warps 4-7, 8-11 two softmax groups that take the stages in turn: a thread owns one
//              TMEM lane (= one query row); it reads its row of S, masks (resident slots,
//              causal inside the chunk), keeps a running max/sum and writes P as bfloat16.
//              Each group has its own S and P tiles, its own output accumulator and its own
//              running state, so that the groups never wait for one another inside a
//              segment; the two states are merged when it ends.  O is rescaled in TMEM when
//              a row's maximum grows by more than 2^8.
// All waits are bounded; a timeout records KVC_DERR_WAIT and the CTA stops.
//
// What bounds it: from about 18 sessions of 8 KV heads on HBM (64 sessions of 4,100
// positions: 167 us per launch, 6.55 TB/s of K/V, q and output bytes; one softmax group with
// a stage's boxes issued by one lane and a thread per row for q, partial states and outputs
// took 193); below that, a stage of a lone CTA takes 0.6 us, the issue of S = Q K^T (10
// instructions of about 70 cycles; one softmax group: 0.8 us), and a launch about 7 us beside
// its stages (1 session: 48.1 -> 12.5 us, most of it the merge of 16 parts by one CTA;
// 9 sessions: 48.6 -> 30.1 us; merging the parts that exist instead of 8, own rows in
// place, took the last 2-3 %).  Under load every access that misses L2 waits behind the K/V
// bytes in flight (about 4 us with a full ring on every SM).  So the queries and rotary rows
// of the next segment are copied while the current one runs, K and V carry an evict-first
// hint that keeps them, the rotary table and the partial states in L2, and in the stream-K
// split nothing waits for the arrival of a range's first partial segment.
#include <cuda.h>

#include "kvc_prefill_tc.cuh"

namespace kvc {

namespace {

// Tensor memory (512 columns x 128 lanes of 32 bits; lane = query row), group g:
//   S_g [64 g, +64)        fp32 scores of a stage
//   O_g [128 + 128 g, +128) fp32 output accumulator
//   P_g [384 + 32 g, +32)  bfloat16 probabilities (2 per column), MMA A operand
//   Q   [448, 512)         bfloat16 rotated, scaled query rows, MMA A operand
constexpr int TMEM_COLS = 512;
constexpr int S_COL = 0, O_COL = 128, P_COL = 384, Q_COL = 448;
constexpr int THREADS = 12 * 32;
constexpr int SM_THREADS = 8 * 32;           // softmax threads
constexpr int PF_MIN_UNITS = 16;             // pages per CTA of the stream-K split, at least
constexpr int PF_MAX_PARTS = 1 << 16;        // no limit on CTAs per pair (merged row by row)
constexpr int MAX_RING = 6;                  // K/V stages of the ring, at most

// Shared memory map (offsets from a 1024-aligned base): barriers and (max, sum) pairs
// first, then the K/V ring, then (CLUSTER) the partial rows sent to this CTA.
enum {
  B_K_FULL = 0,                          // [MAX_RING] K half of a stage loaded
  B_K_EMPTY = B_K_FULL + MAX_RING,       // [MAX_RING] ... and read by S = Q K^T
  B_V_FULL = B_K_EMPTY + MAX_RING,       // [MAX_RING] V half loaded
  B_V_EMPTY = B_V_FULL + MAX_RING,       // [MAX_RING] ... and read by O += P V
  // Per group, one phase per stage of the group (its j-th stage is stage 2 j + g of the
  // CTA).  Every waiter has seen the phase before the one it waits for, so parity waits are
  // exact.
  B_S_FULL = B_V_EMPTY + MAX_RING,       // [2] scores complete
  B_S_EMPTY = B_S_FULL + 2,              // [2] scores read by the group's warps
  B_P_FULL = B_S_EMPTY + 2,              // [2] probabilities written
  B_PV = B_P_FULL + 2,                   // [2] O += P V complete
  B_Q = B_PV + 2,                        // one phase per segment (query tile ready)
  // Fused layer write: one phase per segment holding chunk slots, completed when the
  // softmax warps have written those rows into the pool.
  B_ROWS = B_Q + 1,
  B_FINAL = B_ROWS + 1,                  // every MMA of the CTA complete (both issuers)
  B_RECV = B_FINAL + 1,                  // CLUSTER: every part of this CTA's rows received
  // Stream-K: the first segment's partial state is in global memory (warp 1 arrives for the
  // pair then); warp 1 has looked whether the last segment's other parts are all there.
  B_PUB = B_RECV + 1,
  B_PEEK = B_PUB + 1,
  N_BARS = B_PEEK + 1
};
constexpr int OFF_ML = 0;                              // [2][M] (max, sum) of the groups
constexpr int OFF_BAR = OFF_ML + 2 * M * 8;
constexpr int OFF_TMEM_ADDR = OFF_BAR + N_BARS * 8;
constexpr int OFF_SEQ = OFF_TMEM_ADDR + 16;            // [SEQ_CACHE] sessions of the range
constexpr int SEQ_CACHE = 8;
constexpr int OFF_KV = 3 * 1024;
static_assert(OFF_SEQ % 16 == 0 && OFF_SEQ + SEQ_CACHE * sizeof(SeqInfo) <= OFF_KV &&
                  OFF_KV % 1024 == 0, "header fits");
// A partial row sent to its owner: D binary32 values, then (max, sum) in the padding that
// keeps the rows apart in the banks.
constexpr int ROW_PITCH = (D + 4) * 4;
// Staged rows, padded likewise: query and rotary rows on their way to tensor memory, output
// rows on their way out.  With a thread per row a warp's global accesses would touch 32 lines
// each.
constexpr int ST_PITCH = D * 2 + 16, ROPE_PITCH = D * 4 + 16;
constexpr int SMEM_MAX = 227 * 1024 - 256;   // (the rest: static shared memory)

// After the ring of `ring` stages: the query rows of max_t tokens, their rotary rows, then
// the output rows or (CLUSTER, k > 1) the `recv` received rows.
__host__ __device__ constexpr int off_q(int ring) { return OFF_KV + ring * STAGE; }
__host__ __device__ constexpr int off_rope(int ring, int max_t) {
  return off_q(ring) + max_t * G * ST_PITCH;
}
__host__ __device__ constexpr int off_out(int ring, int max_t) {
  return off_rope(ring, max_t) + max_t * ROPE_PITCH;
}
constexpr int tc_smem(int ring, int max_t, int recv) {
  return 1024 + off_out(ring, max_t) + (recv > 0 ? recv * ROW_PITCH : max_t * G * ST_PITCH);
}
static_assert(M * ROW_PITCH <= 3 * STAGE, "a CTA's partial rows fit a ring of three stages");

__device__ inline void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ inline void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Address of this CTA's shared address `saddr` in CTA `rank` of the cluster.
__device__ inline uint32_t cluster_map(uint32_t saddr, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
// Bulk copy of `bytes` (a multiple of 16) to shared address `dst` of a CTA of the cluster,
// completing on `bar` (an address in that CTA too).
__device__ inline void bulk_s2cluster(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(dst),
      "r"(src), "r"(bytes), "r"(bar)
      : "memory");
}

__device__ inline void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ inline void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// A segment: units [u, end) of the pair (session seq of the call, KV head) whose units are
// [pair_start, pair_end); nb pages per pair of the session.
struct PSeg {
  int seq, head, nb, pair_start, pair_end, u, end;
  __device__ int blk() const { return u - pair_start; }
  __device__ int n_blk() const { return end - u; }
  __device__ int n_st() const { return (end - u + 3) / 4; }
  __device__ bool whole() const { return u == pair_start && end == pair_end; }
};

// Session of the call that holds unit u (one warp; one round trip for 32 sessions each).
__device__ inline int session_of_unit(const Dev& d, int u, int lane) {
  const int n_seq = d.g->n_seq;
  int n = 0;
  for (int i = lane; i < n_seq + lane; i += 32)
    n += __popc(__ballot_sync(FULL, i < n_seq && d.seq[i].unit_base <= u));
  return n - 1;
}

// The segment that starts at unit u of a range ending at u_end, in session seq.
__device__ inline PSeg segment_at(const SeqInfo& si, int seq, int u, int u_end) {
  PSeg s;
  s.seq = seq;
  s.nb = si.n_blocks;
  s.head = (u - si.unit_base) / s.nb;
  s.pair_start = si.unit_base + s.head * s.nb;
  s.pair_end = s.pair_start + s.nb;
  s.u = u;
  s.end = min(u_end, s.pair_end);
  return s;
}

// The only segment of a CTA of the pair split: stages (groups of 4 pages) of slice
// blockIdx.x % k of pair blockIdx.x / k; empty if the pair has fewer stages than slices.
__device__ inline PSeg slice_segment(const Dev& d, int k) {
  const int pair = blockIdx.x / k, slice = blockIdx.x % k;
  PSeg s;
  s.seq = pair / d.kv_heads;
  s.head = pair % d.kv_heads;
  const int nb = d.seq[s.seq].n_blocks, n_all = (nb + 3) / 4;
  s.nb = nb;
  s.pair_start = d.seq[s.seq].unit_base + s.head * nb;
  s.pair_end = s.pair_start + nb;
  s.u = s.pair_start + min(nb, 4 * (int)((int64_t)slice * n_all / k));
  s.end = s.pair_start + min(nb, 4 * (int)((int64_t)(slice + 1) * n_all / k));
  return s;
}

// Rows of partial slot `slot`: [D / 4 chunks][M rows] of 16 bytes, so that the threads of a
// warp, a row each, access them side by side.
__device__ inline float4* part_rows(const Dev& d, int slot) {
  return reinterpret_cast<float4*>(d.pf_part_o + (size_t)slot * (M * D));
}

__device__ inline int us_first_part(const UnitSplit& us, const PSeg& s) {
  return us.U > 0 ? us.owner(s.pair_start) : 0;
}

// Log-sum-exp merge of the nch parts of segment s's pair (CTAs cf .. cf + nch - 1) by the
// softmax threads, columns [64 grp, +64) of row r each; columns [64 grp + 32 c, +32) go to
// store(c, .).  Part own_ch (this CTA's, of maximum Mr and sum Lr) comes from own(c, scale,
// .); own_ch < 0: every part from its slot.  The first other part's columns are loaded
// together with its (max, sum), so a pair of two parts costs one round trip.
template <typename OwnFn, typename StoreFn>
__device__ inline void merge_parts(const Dev& d, const UnitSplit& us, const PSeg& s, int cf,
                                   int nch, int own_ch, bool write, int r, int grp, float Mr,
                                   float Lr, OwnFn own, StoreFn store) {
  const int first_slot = us.slot_of(cf, cf, s.pair_start);
  auto slot_of = [&](int ch) { return ch ? 2 * (cf + ch) : first_slot; };
  auto part4 = [&](int ch, int i) {  // 16-byte chunk i of the half row
    return write ? __ldcg(part_rows(d, slot_of(ch)) + (16 * grp + i) * M + r)
                 : make_float4(0.f, 0.f, 0.f, 0.f);
  };
  auto part_ml = [&](int ch) {
    return write && ch != own_ch ? __ldcg(&d.pf_part_ml[(size_t)slot_of(ch) * M + r])
                                 : make_float2(-INFINITY, 0.f);
  };
  const int f0 = own_ch == 0 ? 1 : 0;  // first other part
  float4 v[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = part4(f0, i);
  const float2 mlf = part_ml(f0);
  const float m_own = write ? Mr : -INFINITY;
  float Mx = fmaxf(m_own, mlf.x);
  for (int ch = f0 + 1; ch < nch; ++ch) Mx = fmaxf(Mx, part_ml(ch).x);
  const float s_own = exp2_safe(m_own, Mx), s_f = exp2_safe(mlf.x, Mx);
  float Ls = Lr * s_own + mlf.y * s_f;
  for (int ch = f0 + 1; ch < nch; ++ch) {
    const float2 ml = part_ml(ch);
    Ls += ml.y * exp2_safe(ml.x, Mx);
  }
  const float inv = 1.f / Ls;
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    float o[32];
    own(c, s_own * inv, o);
    auto add = [&](int i, const float4& w, float sc) {
      o[4 * i] = fmaf(w.x, sc, o[4 * i]);
      o[4 * i + 1] = fmaf(w.y, sc, o[4 * i + 1]);
      o[4 * i + 2] = fmaf(w.z, sc, o[4 * i + 2]);
      o[4 * i + 3] = fmaf(w.w, sc, o[4 * i + 3]);
    };
#pragma unroll
    for (int i = 0; i < 8; ++i) add(i, v[8 * c + i], s_f * inv);
    for (int ch = f0 + 1; ch < nch; ++ch) {  // pairs over three or more CTAs
      if (ch == own_ch) continue;
      const float sc = exp2_safe(part_ml(ch).x, Mx) * inv;
#pragma unroll
      for (int i = 0; i < 8; ++i) add(i, part4(ch, 8 * c + i), sc);
    }
    store(c, o);
  }
}

// Merge of this CTA's n_rows rows from the k <= K parts of the cluster, a 4-element chunk per
// thread and pass: part p's rows in slot p of the received ones (`per` rows apart), this
// CTA's own (p = slice) where it left them.
template <int K, typename RowFn>
__device__ inline void merge_rows(const uint8_t* recv, const uint8_t* own, int slice, int k,
                                  int per, int n_rows, int tid, RowFn out_row) {
  for (int i = tid; i < n_rows * (D / 4); i += THREADS) {
    const int rl = i / (D / 4), c = i % (D / 4);
    float2 ml[K];
    float4 o[K];
#pragma unroll
    for (int p = 0; p < K; ++p) {
      const int pp = min(p, k - 1);
      const uint8_t* pr = (pp == slice ? own : recv + pp * per * ROW_PITCH) + rl * ROW_PITCH;
      ml[p] = p < k ? *reinterpret_cast<const float2*>(pr + D * 4) : make_float2(-INFINITY, 0.f);
      o[p] = *reinterpret_cast<const float4*>(pr + c * 16);
    }
    float mx = -INFINITY;
#pragma unroll
    for (int p = 0; p < K; ++p) mx = fmaxf(mx, ml[p].x);
    float L = 0.f;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int p = 0; p < K; ++p) {
      if (ml[p].x == -INFINITY) continue;  // a part without a key of this row
      const float w = exp2f(ml[p].x - mx);
      L += ml[p].y * w;
      a.x = fmaf(o[p].x, w, a.x);
      a.y = fmaf(o[p].y, w, a.y);
      a.z = fmaf(o[p].z, w, a.z);
      a.w = fmaf(o[p].w, w, a.w);
    }
    const float inv = 1.f / L;
    *reinterpret_cast<uint2*>(out_row(rl) + c * 4) =
        make_uint2(pack_bf16(a.x * inv, a.y * inv), pack_bf16(a.z * inv, a.w * inv));
  }
}

// FUSED (the per-layer order): the chunk's K (rotated at each token's position) and
// V of this layer are not in the pool yet; new_k / new_v hold them ([total][Hkv][D],
// the append's token order).  The softmax warps write the rows of a segment's chunk
// slots into the pool when the segment starts (the CTA owning a (session, head, page)
// unit is the only reader of that unit in the launch), and the producers copy a stage
// holding such slots only after that.
template <bool FUSED, bool CLUSTER>
__global__ void __launch_bounds__(THREADS, 1) attn_prefill_tc_kernel(
    Dev d, int layer, const __grid_constant__ CUtensorMap map_lo,
    const __grid_constant__ CUtensorMap map_hi, const __nv_bfloat16* __restrict__ q,
    __nv_bfloat16* __restrict__ out, float qk_scale, int ring, int max_t, int k_slices, int early,
    const __nv_bfloat16* __restrict__ new_k, const __nv_bfloat16* __restrict__ new_v) {
  extern __shared__ uint8_t smem_raw[];
  // (The same offset in every CTA, so that cluster_map() of an address finds the peer's.)
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + OFF_BAR);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + OFF_TMEM_ADDR);
  __shared__ int s_abort_flag, s_last, s_peek, s_first_last;
  volatile int& s_abort = s_abort_flag;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int H = d.kv_heads, L = d.layers;
  // The first call after an append waits for it (and lets nothing else start before that).
  if (!early) pdl_wait();
  if (CLUSTER && d.g->n_units == 0) {  // the append failed: nothing to do for any CTA
    pdl_wait();
    return;
  }
  if (tid == 0) {
    for (int s = 0; s < ring; ++s) {
      mbar_init(&bars[B_K_FULL + s], 1);
      mbar_init(&bars[B_K_EMPTY + s], 1);
      mbar_init(&bars[B_V_FULL + s], 1);
      mbar_init(&bars[B_V_EMPTY + s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&bars[B_S_FULL + s], 1);
      mbar_init(&bars[B_S_EMPTY + s], 4);
      mbar_init(&bars[B_P_FULL + s], 4);
      mbar_init(&bars[B_PV + s], 1);
    }
    mbar_init(&bars[B_Q], 8);
    mbar_init(&bars[B_ROWS], 8);
    mbar_init(&bars[B_FINAL], 2);
    mbar_init(&bars[B_RECV], 1);
    mbar_init(&bars[B_PUB], 1);
    mbar_init(&bars[B_PEEK], 1);
    fence_mbar_init();
    s_abort = 0;
    s_first_last = 0;
  }
  // This CTA's range of units.
  UnitSplit us = {};
  PSeg seg = {};
  int u_begin, u_end;
  const int cta = blockIdx.x;
  SeqInfo* s_seq = reinterpret_cast<SeqInfo*>(smem + OFF_SEQ);
  if constexpr (CLUSTER) {
    seg = slice_segment(d, k_slices);
    u_begin = seg.u;
    u_end = seg.end;
  } else {
    us = unit_split(d, gridDim.x, PF_MIN_UNITS, PF_MAX_PARTS);
    const bool active = cta < us.n_cta;
    u_begin = active ? us.start_of(cta) : 0;
    u_end = active ? us.start_of(cta + 1) : 0;
    if (u_begin < u_end) seg.seq = session_of_unit(d, u_begin, lane);
  }
  // The sessions that the range can touch first, for every role (info()).
  const int seq0 = seg.seq;
  if (tid < SEQ_CACHE * 16 && seq0 + tid / 16 < d.g->n_seq)
    reinterpret_cast<int*>(s_seq)[tid] = reinterpret_cast<const int*>(d.seq + seq0)[tid];
  auto info = [&](int seq) -> const SeqInfo& {
    return seq - seq0 < SEQ_CACHE ? s_seq[seq - seq0] : d.seq[seq];
  };
  if (CLUSTER && k_slices > 1) {
    // Rows [rank R / k, (rank + 1) R / k) of the pair are CTA rank's to merge and write: it
    // receives the other k - 1 parts of each.  Arrival: this CTA has started and its barrier expects them.
    if (tid == 0) {
      const int R = d.seq[seg.seq].t * G, k = k_slices, slice = cta % k;
      mbar_arrive_expect_tx(&bars[B_RECV], (k - 1) * ((slice + 1) * R / k - slice * R / k) * ROW_PITCH);
    }
    __syncwarp();
    cluster_arrive();
  }
  // The V rows that a partly filled stage leaves unwritten in the ring's first pass have to
  // be finite (their weights are 0, and 0 times a NaN would not be 0); later passes find
  // pool values there.
  {
    const int n_v = CLUSTER ? min(ring, (u_end - u_begin + 3) / 4) : ring;
    for (int s = CLUSTER ? max(0, n_v - 1) : 0; s < n_v; ++s) {
      uint4* v = reinterpret_cast<uint4*>(smem + OFF_KV + s * STAGE + 2 * KV_PANEL);
      for (int i = tid; i < 2 * KV_PANEL / 16; i += THREADS) v[i] = make_uint4(0, 0, 0, 0);
    }
    fence_proxy_async_smem();
  }
  __syncwarp();  // (lanes took the branches above apart; the allocation wants them together)
  if (warp == 2) tmem_alloc(tmem_slot, TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // Before pdl_wait() only the append's data is read (work list, page tables, K/V
  // pages); the softmax warps wait before reading q or writing any result.
  pdl_launch_dependents();
  const uint32_t sKV = smem_u32(smem + OFF_KV);
  if (!CLUSTER && u_begin < u_end) seg = segment_at(info(seq0), seq0, u_begin, u_end);
  // The segment that starts where `s` ends, given s.end < u_end: s then ends at its pair's
  // end, and the next segment is the next pair from its first unit, the session's next KV
  // head or the next session's first one.
  auto step = [&](PSeg& s) {
    if (++s.head == H) {
      s.head = 0;
      s.nb = info(++s.seq).n_blocks;
    }
    s.pair_start = s.u = s.end;
    s.pair_end = s.pair_start + s.nb;
    s.end = min(u_end, s.pair_end);
  };
  // Stream-K: a pair's CTAs arrive at its counter.  The first segment's partial state (of a
  // pair that ends inside the range) is published when its segment ends but nothing waits
  // for the arrival; the last one's is not even published when every other part is there.
  const bool defer = !CLUSTER && u_begin < u_end && seg.u != seg.pair_start && seg.end < u_end;

  if (warp < 2) {
    // ---------------- producers ----------------
    // A K half is free again once S = Q K^T of its stage is complete, a V half once O += P V
    // is, so the K loads run ahead of the V loads by up to the ring depth.  Page ids come 32
    // at a time (lane i holds the id of the window's page i); lane 2 pg + h issues half h
    // (columns 0-63, 64-127) of page pg of a stage: one lane issuing all of a stage's boxes
    // is bound by the issue itself (about 50 ns a box).
    const bool is_v = warp == 1;
    uint64_t* full = bars + (is_v ? B_V_FULL : B_K_FULL);
    uint64_t* empty = bars + (is_v ? B_V_EMPTY : B_K_EMPTY);
    const int pg = (lane >> 1) & 3;
    const CUtensorMap* map = (lane & 1) ? &map_hi : &map_lo;
    uint8_t* dst = smem + OFF_KV + (is_v ? 2 * KV_PANEL : 0) + (lane & 1) * KV_PANEL + pg * 2048;
    const uint64_t policy = evict_first_policy();
    bool arrive_first = is_v && defer;  // (lane 0) the first pair's arrival is still to come
    const int first_cf = us_first_part(us, seg), first_pair = seg.seq * H + seg.head;
    const int first_nch = cta - first_cf + 1;
    uint32_t n = 0;          // stages produced
    int st = 0;              // ring slot and pass of the next stage
    uint32_t pass = 0;
    bool stop = false;
    uint32_t rows_seen = 0;  // segments holding chunk slots, before this one
    (void)rows_seen;
    for (int u = u_begin; u < u_end && !stop;) {
      if (u != u_begin) step(seg);
      u = seg.end;
      const int head = seg.head;
      const SeqInfo& si = info(seg.seq);
      const int32_t* hrow = d.hist_pt + (size_t)si.sid * d.max_pages_per_session;
      const int32_t* lrow = d.live_pt + (size_t)si.sid * d.max_pages_per_session;
      const int blk0 = seg.blk(), nblk = seg.n_blk(), n_st = seg.n_st();
      auto page_at = [&](int b) { return b < nblk ? block_page(si, hrow, lrow, blk0 + b) : 0; };
      int pid = page_at(lane), pid_next = page_at(32 + lane);
      if (is_v) {
        // The segment's query rows (T tokens x G heads, 1 KiB per token) and rotary
        // rows (512 B per token) into L2 ahead of the softmax warps, which read them
        // when the segment starts.  A prefetch changes nothing that a later load
        // observes, so it may run before the previous kernel has finished.
        const char* qb = reinterpret_cast<const char*>(
            q + ((size_t)si.q_row0 * d.q_heads + (size_t)head * G) * D);
        const char* rb = reinterpret_cast<const char*>(d.rope + (size_t)si.pos_first * (D / 2));
        const size_t qstride = (size_t)d.q_heads * D * sizeof(__nv_bfloat16);
        for (int x = lane; x < si.t * 12; x += 32) {
          const int tt = x / 12, line = x % 12;
          prefetch_l2(line < 8 ? qb + tt * qstride + line * 128 : rb + (size_t)tt * 512 + (line - 8) * 128);
        }
      }
      for (int k = 0; k < n_st; ++k, ++n) {
        if (k > 0 && (k & 7) == 0) {
          pid = pid_next;
          pid_next = page_at(4 * k + 32 + lane);
        }
        const int page = __shfl_sync(FULL, pid, 4 * (k & 7) + pg);
        if (arrive_first && lane == 0 && mbar_test(&bars[B_PUB], 0)) {
          s_first_last = arrive_acq_rel(&d.pf_count[first_pair], first_nch);
          arrive_first = false;
        }
        __syncwarp();
        const int npg = min(4, nblk - 4 * k);
        bool ok = mbar_wait(d, &empty[st], (pass & 1) ^ 1);
        if constexpr (FUSED) {
          // A stage holding chunk slots is copied only once the softmax warps have
          // written the segment's rows (they do so when the segment starts).
          int t0, t1;
          chunk_tokens_in(si, blk0 + 4 * k, blk0 + 4 * k + npg, t0, t1);
          if (t0 < t1) ok = ok && mbar_wait(d, &bars[B_ROWS], rows_seen & 1);
        }
        if (!__all_sync(FULL, ok)) {
          if (lane == 0) s_abort = 1;
          stop = true;
          break;
        }
        if (lane == 0) mbar_arrive_expect_tx(&full[st], npg * 2 * 2048);
        __syncwarp();
        if (lane < 8 && pg < npg) {
          // Pool rows of this page's K (kv = 0) or V (kv = 1) tile of `head`.
          const int row = (((page * L + layer) * 2 + (is_v ? 1 : 0)) * H + head) * PS;
          tma_load_2d_hint(dst + st * STAGE, map, 0, row, &full[st], policy);
        }
        if (++st == ring) {
          st = 0;
          ++pass;
        }
      }
      if constexpr (FUSED) {
        int t0, t1;
        chunk_tokens_in(si, blk0, blk0 + nblk, t0, t1);
        if (t0 < t1) ++rows_seen;
      }
      stop = stop || __any_sync(FULL, s_abort != 0);
    }
    if (stop) {
      // No copy may still be in flight when the CTA ends.
      for (uint32_t i = n > (uint32_t)ring ? n - ring : 0; i < n; ++i)
        mbar_wait(d, &full[i % ring], (i / ring) & 1);
    }
    if (!CLUSTER && is_v && u_begin < u_end) {
      pdl_wait();  // the counters may still be the previous launch's until then
      if (arrive_first && lane == 0 && mbar_wait(d, &bars[B_PUB], 0))
        s_first_last = arrive_acq_rel(&d.pf_count[first_pair], first_nch);
      __syncwarp();
      if (!seg.whole() && !stop) {
        const int cf = us.owner(seg.pair_start), nch = us.owner(seg.pair_end - 1) - cf + 1;
        int there = 0;
        if (lane == 0) {
          asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(there)
                       : "l"(&d.pf_count[seg.seq * H + seg.head]) : "memory");
          s_peek = there == nch - 1;
        }
        there = __shfl_sync(FULL, there, 0);
        if (there == nch - 1) {
          // The first other part's rows into L2 (written long ago, perhaps).
          const int ch = cta == cf ? 1 : 0;
          const char* p = reinterpret_cast<const char*>(
              d.pf_part_o + (size_t)(ch ? 2 * (cf + 1) : us.slot_of(cf, cf, seg.pair_start)) * (M * D));
          const int lines = (info(seg.seq).t * G * 16 + 127) / 128;  // per 16-byte chunk column
          for (int i = lane; i < lines * (D / 4); i += 32)
            prefetch_l2(p + (size_t)(i / lines) * (M * 16) + (i % lines) * 128);
        }
      } else if (lane == 0) {
        s_peek = 0;
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars[B_PEEK]);
    }
  } else if (warp < 4) {
    // ---------------- MMA issuers ----------------
    // One elected thread each: their products use different accumulators, and each
    // thread's tcgen05.commit tracks only its own MMAs, so the two streams interleave in
    // the tensor pipe and neither waits behind the other's issue cost (about 60 cycles per
    // instruction, 8 + 2 for a stage's S).
    if (lane == 0) {
      uint32_t n = 0;  // stage
      int st = 0;
      uint32_t pass = 0;
      bool ok = true;
      if (warp == 2) {
        constexpr uint32_t ID_S = instr_desc(NK, M, false);
        uint32_t segs = 0;
        for (int u = u_begin; u < u_end && ok && !s_abort; ++segs) {
          if (u != u_begin) step(seg);
          u = seg.end;
          const int n_st = seg.n_st();
          ok = mbar_wait(d, &bars[B_Q], segs & 1);
          for (int k = 0; k < n_st && ok; ++k, ++n) {
            const int g = n & 1;
            ok = mbar_wait2(d, &bars[B_K_FULL + st], pass & 1, &bars[B_S_EMPTY + g],
                            ((n >> 1) & 1) ^ 1);
            if (!ok) break;
            tc_fence_after();
            const uint64_t kdesc = smem_desc(sKV + st * STAGE, 0, 1024);
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk) {
              // 16 dims per step: 8 TMEM columns of Q; 32 bytes of a swizzled K row.
              tc_mma_ts(tmem + S_COL + g * NK, tmem + Q_COL + kk * 8,
                        desc_at(kdesc, (kk >> 2) * KV_PANEL + (kk & 3) * 32), ID_S, kk > 0 ? 1u : 0u);
            }
            tc_commit(&bars[B_S_FULL + g]);
            tc_commit(&bars[B_K_EMPTY + st]);
            if (++st == ring) {
              st = 0;
              ++pass;
            }
          }
        }
      } else {
        constexpr uint32_t ID_PV = instr_desc(D, M, true);
        for (int u = u_begin; u < u_end && ok && !s_abort;) {
          if (u != u_begin) step(seg);
          u = seg.end;
          const int n_st = seg.n_st();
          for (int k = 0; k < n_st && ok; ++k, ++n) {
            const int g = n & 1;
            ok = mbar_wait2(d, &bars[B_V_FULL + st], pass & 1, &bars[B_P_FULL + g], (n >> 1) & 1);
            if (!ok) break;
            tc_fence_after();
            const uint64_t vdesc = smem_desc(sKV + st * STAGE + 2 * KV_PANEL, KV_PANEL, 1024);
#pragma unroll
            for (int kk = 0; kk < NK / 16; ++kk) {
              // 16 keys per step: 8 TMEM columns of P; 16 rows of the V panels.  A group's
              // first product of a segment overwrites its O (both groups read the previous
              // contents before they wrote any P of this segment).
              tc_mma_ts(tmem + O_COL + g * D, tmem + P_COL + g * (NK / 2) + kk * 8,
                        desc_at(vdesc, kk * 16 * 128), ID_PV, (k > 1 || kk > 0) ? 1u : 0u);
            }
            tc_commit(&bars[B_PV + g]);
            tc_commit(&bars[B_V_EMPTY + st]);
            if (++st == ring) {
              st = 0;
              ++pass;
            }
          }
        }
      }
      if (!ok) s_abort = 1;
      // No MMA may still be running when the tensor memory is released.
      tc_commit(&bars[B_FINAL]);
      mbar_wait(d, &bars[B_FINAL], 0);
    }
    __syncwarp();
  } else {
    // ---------------- softmax / epilogue ----------------
    // A failed (timed-out) wait makes the warp "dead": it then skips waits and
    // work but still walks the same segments and named barriers, so the other
    // softmax warps never wait for it.
    const int grp = (warp >> 2) - 1;           // group 0 (warps 4-7) or 1 (warps 8-11)
    const int quarter = warp & 3;              // TMEM lanes 32*quarter .. +31
    const int r = quarter * 32 + lane;         // this thread's query row
    const int ts = tid - (THREADS - SM_THREADS);
    const uint32_t trow = tmem + ((uint32_t)(quarter * 32) << 16);
    float2* s_ml = reinterpret_cast<float2*>(smem + OFF_ML);
    uint32_t n = 0;                            // stages of the earlier segments
    bool dead = false;
    auto wait = [&](uint64_t* bar, uint32_t parity) {
      if (dead) return;
      dead = !__all_sync(FULL, mbar_wait(d, bar, parity));
      if (dead && lane == 0) s_abort = 1;
    };
    // (bar.sync and the tensor-memory accesses want the warp converged.)
    auto sync_groups = [] {
      __syncwarp();
      asm volatile("bar.sync 1, %0;" ::"n"(SM_THREADS) : "memory");
    };
    uint8_t* st_q = smem + off_q(ring);
    uint8_t* st_rope = smem + off_rope(ring, max_t);
    uint8_t* st_out = smem + off_out(ring, max_t);
    // Asynchronous copies of a segment's rotary and query rows into their staging rows.
    auto copy_rope = [&](const PSeg& sg) {
      const SeqInfo& si = info(sg.seq);
      const uint4* src = reinterpret_cast<const uint4*>(d.rope + (size_t)si.pos_first * (D / 2));
      const uint32_t dst = smem_u32(st_rope);
      for (int i = ts; i < si.t * 32; i += SM_THREADS)
        cp_async16(dst + (i >> 5) * ROPE_PITCH + (i & 31) * 16, src + i);
    };
    auto copy_q = [&](const PSeg& sg) {
      const SeqInfo& si = info(sg.seq);
      const uint4* src = reinterpret_cast<const uint4*>(
          q + ((size_t)si.q_row0 * d.q_heads + sg.head * G) * D);
      const uint32_t dst = smem_u32(st_q);
      const size_t tok = (size_t)d.q_heads * D / 8;
      for (int i = ts; i < si.t * 64; i += SM_THREADS)  // a token's G rows are contiguous
        cp_async16(dst + (i >> 4) * ST_PITCH + (i & 15) * 16, src + (i >> 6) * tok + (i & 63));
    };
    // The staged query rows, rotated at their tokens' positions, scaled and rounded, into
    // tensor memory: this thread's row, its group's 4 of the 8 pairs of 16-byte chunks (c,
    // c + 8) that rotate together.  Padding rows: zero, and their P too.  Then, in the
    // per-layer order, the segment's new rows into the pool.
    auto start_segment = [&](const PSeg& sg) {
      const SeqInfo& si = info(sg.seq);
      uint32_t qw[32];
      if (r < si.t * G) {
        const uint4* qrow = reinterpret_cast<const uint4*>(st_q + r * ST_PITCH) + 4 * grp;
        const float4* cs = reinterpret_cast<const float4*>(st_rope + (r / G) * ROPE_PITCH) + 16 * grp;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const uint4 wa = qrow[c], wb = qrow[c + 8];
          const uint32_t ua[4] = {wa.x, wa.y, wa.z, wa.w}, ub[4] = {wb.x, wb.y, wb.z, wb.w};
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            const float4 t4 = cs[c * 4 + h];  // (cos, sin) of dims 8c + 2h, 8c + 2h + 1
            const float a0 = bf16lo(ua[h]), a1 = bf16hi(ua[h]);
            const float b0 = bf16lo(ub[h]), b1 = bf16hi(ub[h]);
            qw[4 * c + h] = pack_bf16(fmaf(a0, t4.x, -b0 * t4.y) * qk_scale,
                                      fmaf(a1, t4.z, -b1 * t4.w) * qk_scale);
            qw[16 + 4 * c + h] = pack_bf16(fmaf(b0, t4.x, a0 * t4.y) * qk_scale,
                                           fmaf(b1, t4.z, a1 * t4.w) * qk_scale);
          }
        }
      } else {
#pragma unroll
        for (int i = 0; i < 32; ++i) qw[i] = 0u;
      }
      __syncwarp();
      tmem_st16(trow + Q_COL + 16 * grp, qw);
      tmem_st16(trow + Q_COL + 32 + 16 * grp, qw + 16);
      if (quarter * 32 >= si.t * G) tmem_st32(trow + P_COL + grp * (NK / 2), qw);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars[B_Q]);
      if constexpr (FUSED) {
        int t0, t1;
        chunk_tokens_in(si, sg.blk(), sg.blk() + sg.n_blk(), t0, t1);
        if (t0 < t1) {
          if (!dead)
            write_chunk_rows(d, layer, si, sg.head, new_k, new_v, t0, t1, ts, SM_THREADS);
          __syncwarp();
          if (lane == 0) mbar_arrive(&bars[B_ROWS]);
        }
      }
    };
    if (u_begin < u_end) copy_rope(seg);  // (the table is not written by any launch)
    pdl_wait();
    if (u_begin < u_end) {
      copy_q(seg);
      cp_async_wait_all();
      sync_groups();
      start_segment(seg);
    }
    for (int u = u_begin; u < u_end;) {
      const bool first = u == u_begin;
      u = seg.end;
      const PSeg cur = seg;
      const SeqInfo& si = info(cur.seq);
      const int head = cur.head;
      const int blk0 = cur.blk(), nblk = cur.n_blk(), n_st = cur.n_st();
      const int R = si.t * G;
      if (u < u_end) {
        // The next segment's rows are copied while this one runs (every thread is done with
        // the staged ones: the last segment's end synchronised them).
        step(seg);
        if (first) sync_groups();
        copy_rope(seg);
        copy_q(seg);
      }
      const bool live = r < R, idle = quarter * 32 >= R;
      const int qlog = si.n_hist + si.n_live - si.t + r / G;
      // Blocks that may need a mask: the partly filled last history page, the
      // first live page when it starts mid-page, and every block from the one
      // holding the chunk's first query on (causal).  A stage of four pages that
      // avoids them all is interior.
      const int nhp = si.n_hist_pages;
      const int b_hist_part = (si.n_hist % PS) ? nhp - 1 : -PS;
      const int b_live_part = si.live_head ? nhp : -PS;
      const int sl_first = si.live_head + si.n_live - si.t;  // live slot of the first query
      const int b_causal = nhp + sl_first / PS + ((sl_first % PS) == PS - 1 ? 1 : 0);
      float m_used = -INFINITY, l = 0.f;
      const int k_first = (grp ^ n) & 1;  // this group's stages: k_first, + 2, ...
      for (int k = k_first; k < n_st; k += 2) {
        const uint32_t j = (n + k) >> 1;
        wait(&bars[B_S_FULL + grp], j & 1);
        if (dead) break;
        tc_fence_after();
        if (idle) {  // padding rows alone: their P is zero already
          if (lane == 0) mbar_arrive(&bars[B_S_EMPTY + grp]);
          if (j > 0) wait(&bars[B_PV + grp], (j - 1) & 1);
          if (lane == 0 && !dead) mbar_arrive(&bars[B_P_FULL + grp]);
          continue;
        }
        float s[NK];
        tmem_ld64(trow + S_COL + grp * NK, s);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars[B_S_EMPTY + grp]);
        // Mask the keys that are not resident slots or lie after the row's query.
        // Interior stages (four full pages, every key before the chunk's first
        // query) need no mask.  Padding rows (r >= T*G) are left unmasked: their
        // products stay finite and their outputs are never written.
        const int npg = min(4, nblk - 4 * k);
        const int b0 = blk0 + 4 * k;
        const bool interior = npg == 4 && b0 + 3 < b_causal &&
                              (unsigned)(b_hist_part - b0) > 3u && (unsigned)(b_live_part - b0) > 3u;
        if (!interior) {
#pragma unroll
          for (int pg = 0; pg < 4; ++pg) {
            const BlockRange br = block_range(si, b0 + min(pg, npg - 1));
#pragma unroll
            for (int i = 0; i < PS; ++i) {
              const bool v = pg < npg && i >= br.lo && i < br.hi && br.base + i <= qlog;
              float& x = s[pg * PS + i];
              x = (v || !live) ? x : -INFINITY;
            }
          }
        }
        // Row maximum over 8 independent chains.
        float m8[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) m8[i] = s[i];
#pragma unroll
        for (int i = 8; i < NK; i += 16)
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            if (i + 8 + c < NK) m8[c] = fmaxf(fmaxf(m8[c], s[i + c]), s[i + 8 + c]);
            else m8[c] = fmaxf(m8[c], s[i + c]);
          }
        float mx = fmaxf(fmaxf(fmaxf(m8[0], m8[1]), fmaxf(m8[2], m8[3])),
                         fmaxf(fmaxf(m8[4], m8[5]), fmaxf(m8[6], m8[7])));
        if (!live) mx = -INFINITY;
        // The group's previous product is complete: its O may be rescaled and its P
        // overwritten.
        if (j > 0) wait(&bars[B_PV + grp], (j - 1) & 1);
        if (dead) break;
        // Rescale O (in TMEM) and l only when the row maximum grows by > 2^8.  Every lane
        // of the warp takes part in the TMEM accesses; lanes that need no rescale use
        // factor 1.
        const bool need = mx > m_used + RESCALE_LOG2;
        const bool have_o = k > k_first && m_used != -INFINITY;
        if (__any_sync(FULL, need && have_o)) {
          tc_fence_after();
          const float f = (need && have_o) ? exp2f(m_used - mx) : 1.f;
#pragma unroll 1
          for (int c = 0; c < D / 16; ++c) {
            float o[16];
            tmem_ld16(trow + O_COL + grp * D + c * 16, o);
#pragma unroll
            for (int i = 0; i < 16; ++i) o[i] *= f;
            tmem_st16(trow + O_COL + grp * D + c * 16, o);
          }
        }
        if (need) {
          if (have_o) l *= exp2f(m_used - mx);
          m_used = mx;
        }
        // P = exp2(s - m_used) as bfloat16 pairs.  Masked keys are -inf and give 0; a row
        // with no finite key yet uses 0 as its reference so that no -inf - -inf appears;
        // padding rows get weight 0.
        const float mref = !live ? INFINITY : (m_used == -INFINITY ? 0.f : m_used);
        const float2 nref = make_float2(-mref, -mref);
        float2 rs[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f),
                        make_float2(0.f, 0.f)};
        uint32_t pw[NK / 2];
#pragma unroll
        for (int i = 0; i < NK; i += 2) {
          const float2 x = __fadd2_rn(make_float2(s[i], s[i + 1]), nref);
          const float2 p = make_float2(ex2(x.x), ex2(x.y));
          rs[(i / 2) & 3] = __fadd2_rn(rs[(i / 2) & 3], p);
          pw[i / 2] = pack_bf16(p.x, p.y);
        }
        const float2 r2 = __fadd2_rn(__fadd2_rn(rs[0], rs[1]), __fadd2_rn(rs[2], rs[3]));
        l += r2.x + r2.y;
        __syncwarp();
        tmem_st32(trow + P_COL + grp * (NK / 2), pw);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars[B_P_FULL + grp]);
      }
      // Epilogue: every product of the segment complete, both groups' (max, sum) known.
      if (k_first < n_st) {
        const uint32_t j = (n + ((n_st - 1 - k_first) & ~1) + k_first) >> 1;  // last own stage
        wait(&bars[B_PV + grp], j & 1);
      }
      n += n_st;
      s_ml[grp * M + r] = make_float2(dead ? -INFINITY : m_used, l);
      tc_fence_before();
      cp_async_wait_all();
      sync_groups();
      tc_fence_after();
      if (u < u_end) start_segment(seg);
      const float2 ml0 = s_ml[r], ml1 = s_ml[M + r];
      // A segment of one stage has the state of one group only.
      const bool has0 = n_st > 1 || k_first == grp, has1 = n_st > 1 || k_first != grp;
      const float Mr = fmaxf(has0 ? ml0.x : -INFINITY, has1 ? ml1.x : -INFINITY);
      const float f0 = has0 ? exp2_safe(ml0.x, Mr) : 0.f, f1 = has1 ? exp2_safe(ml1.x, Mr) : 0.f;
      const float Lr = (has0 ? ml0.y * f0 : 0.f) + (has1 ? ml1.y * f1 : 0.f);
      // Columns [64 grp + 32 c, + 32) of this row, both groups' parts summed.
      auto own = [&](int c, float sc, float (&o)[32]) {
        __syncwarp();  // (rows that are not live skip the stores of the columns before)
        const uint32_t col = trow + O_COL + 64 * grp + 32 * c;
        const float a0 = f0 * sc, a1 = f1 * sc;
        if (has0) {
          tmem_ld32(col, o);
#pragma unroll
          for (int i = 0; i < 32; ++i) o[i] *= a0;
        } else {
#pragma unroll
          for (int i = 0; i < 32; ++i) o[i] = 0.f;
        }
        if (has1) {
#pragma unroll
          for (int h = 0; h < 32; h += 16) {
            float o1[16];
            tmem_ld16(col + D + h, o1);
#pragma unroll
            for (int i = 0; i < 16; ++i) o[h + i] = fmaf(o1[i], a1, o[h + i]);
          }
        }
      };
      const bool write = live && !dead;
      // Output rows leave through the staging rows: store() puts 32 normalised columns of this
      // thread's row there, flush() writes the rows out whole.
      auto store = [&](int c, const float (&o)[32]) {
        if (!live) return;
#pragma unroll
        for (int i = 0; i < 32; i += 8)
          *reinterpret_cast<uint4*>(st_out + r * ST_PITCH + 128 * grp + 64 * c + 2 * i) =
              make_uint4(pack_bf16(o[i], o[i + 1]), pack_bf16(o[i + 2], o[i + 3]),
                         pack_bf16(o[i + 4], o[i + 5]), pack_bf16(o[i + 6], o[i + 7]));
      };
      auto flush = [&] {
        sync_groups();
        for (int i = ts; i < R * 16 && !dead; i += SM_THREADS) {
          const int row = i >> 4, c = i & 15;
          __nv_bfloat16* orow =
              out + ((size_t)(si.q_row0 + row / G) * d.q_heads + head * G + row % G) * D;
          reinterpret_cast<uint4*>(orow)[c] =
              *reinterpret_cast<const uint4*>(st_out + row * ST_PITCH + c * 16);
        }
      };
      if (CLUSTER ? k_slices == 1 : cur.whole()) {
        const float inv = 1.f / Lr;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          float o[32];
          own(c, inv, o);
          store(c, o);
        }
        flush();
      } else if constexpr (CLUSTER) {
        // The partial rows into the ring's place (every copy and product is complete); they
        // are sent from there below.
        float* prow = reinterpret_cast<float*>(smem + OFF_KV + r * ROW_PITCH);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          float o[32];
          own(c, 1.f, o);
          if (write) {
#pragma unroll
            for (int i = 0; i < 32; i += 4)
              *reinterpret_cast<float4*>(prow + 64 * grp + 32 * c + i) =
                  make_float4(o[i], o[i + 1], o[i + 2], o[i + 3]);
          }
        }
        if (live && grp == 0) *reinterpret_cast<float2*>(prow + D) = make_float2(Mr, Lr);
      } else {
        // Split-K: publish this part's (O, max, sum); the last CTA to arrive for the
        // (session, head) merges every part, half a query row per thread.  Every softmax
        // warp reaches the same named barriers.
        const bool deferred = first && defer, last = u >= u_end;
        if (last) wait(&bars[B_PEEK], 0);
        const bool alone = last && !dead && s_peek;  // every other part is there
        const int cf = us.owner(cur.pair_start), nch = us.owner(cur.pair_end - 1) - cf + 1;
        if (!__any_sync(FULL, alone)) {
          const int slot = 2 * cta + (first ? 0 : 1);
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            float o[32];
            own(c, 1.f, o);
            if (write) {
#pragma unroll
              for (int i = 0; i < 8; ++i)
                part_rows(d, slot)[(16 * grp + 8 * c + i) * M + r] =
                    make_float4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
            }
          }
          if (write && grp == 0) d.pf_part_ml[(size_t)slot * M + r] = make_float2(Mr, Lr);
        }
        sync_groups();
        if (deferred) {
          if (ts == 0) mbar_arrive(&bars[B_PUB]);
        } else {
          if (ts == 0)
            s_last = alone || arrive_acq_rel(&d.pf_count[cur.seq * H + head], nch);
          sync_groups();
        }
        if (!deferred && s_last) {
          // This CTA's own part is still in the O columns.  Every lane takes part in the
          // tensor-memory accesses; rows that are padding (or of a warp whose wait gave up)
          // write nothing.
          merge_parts(d, us, cur, cf, nch, cta - cf, write, r, grp, Mr, Lr,
                      [&](int c, float sc, float (&o)[32]) { own(c, sc, o); }, store);
          flush();
          if (ts == 0) d.pf_count[cur.seq * H + head] = 0;
        }
      }
      // Both groups have read O and the (max, sum) pairs before either goes on.
      tc_fence_before();
      sync_groups();
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 2) tmem_dealloc(tmem, TMEM_COLS);
  if (!CLUSTER && s_first_last && warp >= 4) {
    // The first segment's pair was complete when this CTA arrived for it: every part,
    // this CTA's own too, comes from its slot.
    const int grp = (warp >> 2) - 1, r = (warp & 3) * 32 + lane, ts = tid - (THREADS - SM_THREADS);
    const PSeg s = segment_at(info(seq0), seq0, u_begin, u_end);
    const SeqInfo& si = info(seq0);
    const int R = si.t * G, cf = us.owner(s.pair_start), nch = cta - cf + 1;
    uint8_t* st_out = smem + off_out(ring, max_t);
    merge_parts(
        d, us, s, cf, nch, -1, r < R, r, grp, -INFINITY, 0.f,
        [](int, float, float (&o)[32]) {
#pragma unroll
          for (int i = 0; i < 32; ++i) o[i] = 0.f;
        },
        [&](int c, const float (&o)[32]) {
          if (r >= R) return;
#pragma unroll
          for (int i = 0; i < 32; i += 8)
            *reinterpret_cast<uint4*>(st_out + r * ST_PITCH + 128 * grp + 64 * c + 2 * i) =
                make_uint4(pack_bf16(o[i], o[i + 1]), pack_bf16(o[i + 2], o[i + 3]),
                           pack_bf16(o[i + 4], o[i + 5]), pack_bf16(o[i + 6], o[i + 7]));
        });
    __syncwarp();
    asm volatile("bar.sync 1, %0;" ::"n"(SM_THREADS) : "memory");
    for (int i = ts; i < R * 16; i += SM_THREADS) {
      const int row = i >> 4, c = i & 15;
      __nv_bfloat16* orow =
          out + ((size_t)(si.q_row0 + row / G) * d.q_heads + s.head * G + row % G) * D;
      reinterpret_cast<uint4*>(orow)[c] =
          *reinterpret_cast<const uint4*>(st_out + row * ST_PITCH + c * 16);
    }
    if (ts == 0) d.pf_count[seq0 * H + s.head] = 0;
  }
  if constexpr (CLUSTER) {
    if (k_slices == 1) return;
    const int k = k_slices, slice = cta % k;
    const SeqInfo& si = info(seg.seq);
    const int R = si.t * G, per = (R + k - 1) / k;
    const int r0 = slice * R / k, n_rows = (slice + 1) * R / k - r0;
    const uint32_t s_recv = smem_u32(smem + off_out(ring, max_t));
    // Every part of another CTA's rows goes to slot `slice` of its received rows.
    for (int i = tid; u_begin == u_end && i < R; i += THREADS)  // no page: weighs nothing
      *reinterpret_cast<float2*>(smem + OFF_KV + i * ROW_PITCH + D * 4) = make_float2(-INFINITY, 0.f);
    fence_proxy_async_smem();
    __syncthreads();
    cluster_wait();  // every CTA of the cluster has started
    if (tid < k) {
      const int f = tid * R / k, nf = (tid + 1) * R / k - f;
      if (nf > 0 && tid != slice)
        bulk_s2cluster(cluster_map(s_recv + slice * per * ROW_PITCH, tid), sKV + f * ROW_PITCH,
                       nf * ROW_PITCH, cluster_map(smem_u32(&bars[B_RECV]), tid));
    }
    __syncwarp();
    pdl_wait();
    const bool got = mbar_wait(d, &bars[B_RECV], 0);
    __syncwarp();
    cluster_arrive();
    // Merge and write this CTA's rows.
    const uint8_t* rows = smem + off_out(ring, max_t);
    const uint8_t* own = smem + OFF_KV + r0 * ROW_PITCH;
    auto out_row = [&](int rl) {
      const int row = r0 + rl;
      return out + ((size_t)(si.q_row0 + row / G) * d.q_heads + seg.head * G + row % G) * D;
    };
    if (got) {
      if (k <= 2)
        merge_rows<2>(rows, own, slice, k, per, n_rows, tid, out_row);
      else if (k <= 4)
        merge_rows<4>(rows, own, slice, k, per, n_rows, tid, out_row);
      else
        merge_rows<PF_MAX_SLICES>(rows, own, slice, k, per, n_rows, tid, out_row);
    }
    __syncwarp();
    cluster_wait();  // every part was received: no copy still reads this CTA's rows
  }
}

using TcFn = void (*)(Dev, int, const CUtensorMap, const CUtensorMap, const __nv_bfloat16*,
                      __nv_bfloat16*, float, int, int, int, int, const __nv_bfloat16*,
                      const __nv_bfloat16*);
TcFn tc_kernel(bool fused, bool cluster) {
  return cluster ? (fused ? &attn_prefill_tc_kernel<true, true> : &attn_prefill_tc_kernel<false, true>)
                 : (fused ? &attn_prefill_tc_kernel<true, false> : &attn_prefill_tc_kernel<false, false>);
}

cudaError_t set_attributes() {
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < 4 && e == cudaSuccess; ++i)
    e = cudaFuncSetAttribute(reinterpret_cast<const void*>(tc_kernel(i & 1, i & 2)),
                             cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_MAX);
  return e;
}

}  // namespace

cudaError_t prefill_tc_limits(Limits* lim) {
  cudaError_t e = set_attributes();
  if (e != cudaSuccess) return e;
  const void* fn = reinterpret_cast<const void*>(tc_kernel(false, false));
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, THREADS, SMEM_MAX);
  if (e != cudaSuccess) return e;
  lim->pf_stream_k = max(1, per_sm) * lim->sms;
  for (int k = 1; k <= PF_MAX_SLICES; ++k) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(k);
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = SMEM_MAX;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = k;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    e = cudaOccupancyMaxActiveClusters(&n, tc_kernel(false, true), &cfg);
    lim->pf_clusters[k] = e == cudaSuccess ? n : 0;
    if (e != cudaSuccess) cudaGetLastError();  // (a size that the device does not take: no error)
  }
  return cudaSuccess;
}

cudaError_t launch_attn_prefill_tc(const Dev& d, int layer, const CUtensorMap& lo,
                                   const CUtensorMap& hi, const void* q, void* out, int grid,
                                   int k, int max_t, bool early, cudaStream_t s, const void* new_k,
                                   const void* new_v) {
  const float scale = LOG2E / sqrtf((float)d.head_dim);
  // The deepest ring that leaves room for the rows sent to a CTA (k parts of its share).
  const int recv = k > 1 ? (max_t * G + k - 1) / k * k : 0;
  int ring = MAX_RING;
  while (tc_smem(ring, max_t, recv) > SMEM_MAX) --ring;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = tc_smem(ring, max_t, recv);
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
  return cudaLaunchKernelEx(&cfg, tc_kernel(new_k != nullptr, k > 0), d, layer, lo, hi,
                            static_cast<const __nv_bfloat16*>(q),
                            static_cast<__nv_bfloat16*>(out), scale, ring, max_t, k, (int)early,
                            static_cast<const __nv_bfloat16*>(new_k),
                            static_cast<const __nv_bfloat16*>(new_v));
}

}  // namespace kvc
