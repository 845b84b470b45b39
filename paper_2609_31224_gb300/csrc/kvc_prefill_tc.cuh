// Tile constants, tensor-memory and MMA helpers of the tcgen05 prefill kernel
// (kvc_attn_prefill_tc.cu), and its fused write of the chunk's K and V rows.
#pragma once

#include "kvc_launch.cuh"
#include "kvc_rope.cuh"

namespace kvc {

namespace {

constexpr int G = 4;
constexpr int D = 128;
constexpr int M = 128;                       // MMA rows (query rows, padded)
constexpr int NK = 64;                       // keys per stage (4 pages)
constexpr int KV_PANEL = NK * 128;           // 64 rows x 128 B = 8 KiB
constexpr int STAGE = 4 * KV_PANEL;          // K lo, K hi, V lo, V hi = 32 KiB
constexpr float LOG2E = 1.4426950408889634f;
constexpr float RESCALE_LOG2 = 8.f;          // rescale O only when the max grows by > 2^8
constexpr unsigned FULL = 0xFFFFFFFFu;

// Whether a phase is complete, without waiting (mbarrier.try_wait may suspend the thread).
__device__ inline bool mbar_test(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait for two barriers: both are tested first, back to back, so that their latencies
// overlap when both are ready.
__device__ inline bool mbar_wait2(const Dev& d, uint64_t* a, uint32_t pa, uint64_t* b, uint32_t pb) {
  const bool ra = mbar_test(a, pa), rb = mbar_test(b, pb);
  return (ra || mbar_wait(d, a, pa)) && (rb || mbar_wait(d, b, pb));
}

// -- tcgen05 helpers ------------------------------------------------------------------
__device__ inline void tmem_alloc(uint32_t* smem_dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_u32(smem_dst)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ inline void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
               : "memory");
}
__device__ inline void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ inline void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ inline void tc_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}
// D (TMEM) (+)= A B with A read from tensor memory (M lanes, K/2 columns of
// bfloat16 pairs) and B from shared memory.
__device__ inline void tc_mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc,
                                 uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Each thread of the warp reads 32 consecutive fp32 columns of its TMEM lane.
__device__ inline void tmem_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
      "%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
        "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
        "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
        "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
// 64 consecutive columns, one wait.
__device__ inline void tmem_ld64(uint32_t taddr, float* v) {
  uint32_t r[64];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x64.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32,%33,%34,%35,%36,%37,%38,%39,%40,%41,%42,%43,%44,%45,%46,%47,%48,%49,%50,%51,%52,%53,%54,%55,%56,%57,%58,%59,%60,%61,%62,%63}, [%64];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]), "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]), "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]), "=r"(r[48]), "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]), "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 64; ++i) v[i] = __uint_as_float(r[i]);
}
// The same for 16 columns.
__device__ inline void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ inline void tmem_st16(uint32_t taddr, const float* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
      "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])), "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])), "r"(__float_as_uint(v[8])), "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])), "r"(__float_as_uint(v[11])), "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])), "r"(__float_as_uint(v[15]))
      : "memory");
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
__device__ inline void tmem_st16(uint32_t taddr, const uint32_t* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
      "r"((v[0])), "r"((v[1])), "r"((v[2])), "r"((v[3])), "r"((v[4])), "r"((v[5])), "r"((v[6])), "r"((v[7])), "r"((v[8])), "r"((v[9])), "r"((v[10])), "r"((v[11])), "r"((v[12])), "r"((v[13])), "r"((v[14])), "r"((v[15]))
      : "memory");
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
__device__ inline void tmem_st32(uint32_t taddr, const uint32_t* w) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,"
      "%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(
          taddr),
      "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]),
      "r"(w[8]), "r"(w[9]), "r"(w[10]), "r"(w[11]), "r"(w[12]), "r"(w[13]), "r"(w[14]),
      "r"(w[15]), "r"(w[16]), "r"(w[17]), "r"(w[18]), "r"(w[19]), "r"(w[20]), "r"(w[21]),
      "r"(w[22]), "r"(w[23]), "r"(w[24]), "r"(w[25]), "r"(w[26]), "r"(w[27]), "r"(w[28]),
      "r"(w[29]), "r"(w[30]), "r"(w[31])
      : "memory");
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
// Shared-memory matrix descriptor, 128-byte swizzle: `sbo` bytes between 8-row
// groups; `lbo` bytes between 64-element groups of the contiguous dimension
// (MN-major operands only).
__device__ inline uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;  // descriptor version of this architecture
  d |= (uint64_t)2 << 61;  // 128-byte swizzle
  return d;
}

// The descriptor `bytes` further on (a multiple of 16; the address field does not
// overflow within one CTA's shared memory).
__device__ inline uint64_t desc_at(uint64_t desc, uint32_t bytes) { return desc + (bytes >> 4); }

// The per-layer write of the chunk rows of tokens [t0, t1) of a session (its call
// row q_row0, positions from pos_first) for KV head `head`, by the n_threads
// softmax threads (thread index ts): V rows copied, K rows rotated at their positions, in
// 16-byte chunks, every load of an item issued before its stores.  Each thread then
// orders its writes before later tensor copies (async proxy).
__device__ inline void write_chunk_rows(const Dev& d, int layer, const SeqInfo& si, int head,
                                        const __nv_bfloat16* new_k, const __nv_bfloat16* new_v,
                                        int t0, int t1, int ts, int n_threads) {
  // Item (token, c): 16-byte chunk c of the first half of the K row with its
  // rotate-half partner, and chunks c and c + 8 of the V row.
  constexpr int VEC = 8, HALF = D / 2, KC = HALF / VEC;
  __nv_bfloat16* pool = reinterpret_cast<__nv_bfloat16*>(d.pool);
  const int H = d.kv_heads;
  const int n = (t1 - t0) * KC;
  for (int idx = ts; idx < n; idx += n_threads) {
    const int t = t0 + idx / KC, c = idx % KC;
    const size_t in_row = ((size_t)(si.q_row0 + t) * H + head) * D + c * VEC;
    const uint4 ka = *reinterpret_cast<const uint4*>(new_k + in_row);
    const uint4 kb = *reinterpret_cast<const uint4*>(new_k + in_row + HALF);
    const uint4 va = *reinterpret_cast<const uint4*>(new_v + in_row);
    const uint4 vb = *reinterpret_cast<const uint4*>(new_v + in_row + HALF);
    const float2* t2 = d.rope + (size_t)(si.pos_first + t) * HALF + c * VEC;
    float2 cs[VEC];
#pragma unroll
    for (int e = 0; e < VEC; ++e) cs[e] = t2[e];
    const int gs = d.tok_slot[si.q_row0 + t];
    float xa[VEC], xb[VEC], ya[VEC], yb[VEC];
    Chunk16<__nv_bfloat16>::unpack(ka, xa);
    Chunk16<__nv_bfloat16>::unpack(kb, xb);
#pragma unroll
    for (int e = 0; e < VEC; ++e) rope_pair(xa[e], xb[e], cs[e], ya[e], yb[e]);
    __nv_bfloat16* kd = pool + pool_offset_elems(d, gs / PS, layer, 0, head, gs % PS) + c * VEC;
    __nv_bfloat16* vd = pool + pool_offset_elems(d, gs / PS, layer, 1, head, gs % PS) + c * VEC;
    *reinterpret_cast<uint4*>(kd) = Chunk16<__nv_bfloat16>::pack(ya);
    *reinterpret_cast<uint4*>(kd + HALF) = Chunk16<__nv_bfloat16>::pack(yb);
    *reinterpret_cast<uint4*>(vd) = va;
    *reinterpret_cast<uint4*>(vd + HALF) = vb;
  }
  asm volatile("fence.proxy.async.global;" ::: "memory");
}

// Chunk tokens [t0, t1) of a session whose slots lie in its blocks [b_lo, b_hi).
__device__ inline void chunk_tokens_in(const SeqInfo& si, int b_lo, int b_hi, int& t0, int& t1) {
  const int sl_first = si.live_head + si.n_live - si.t;  // live slot of the first token
  const int lo = (b_lo - si.n_hist_pages) * PS, hi = (b_hi - si.n_hist_pages) * PS;
  t0 = max(0, lo - sl_first);
  t1 = min(si.t, hi - sl_first);
}

// Instruction descriptor, kind::f16: D fp32, A and B bf16, A K-major, B K- or MN-major.
__host__ __device__ constexpr uint32_t instr_desc(int n, int m, bool b_mn_major) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((b_mn_major ? 1u : 0u) << 16) |
         ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

__device__ inline uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

__device__ inline float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

}  // namespace

}  // namespace kvc
