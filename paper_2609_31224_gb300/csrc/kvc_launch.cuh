// Host-side launchers of the kvc kernels (defined in the .cu files) and the
// argument blocks they pass by value.
#pragma once

#include "kvc_decode_slices.h"
#include "kvc_internal.cuh"

namespace kvc {

// ---------------------------------------------------------------------------
// Launchers (defined in the .cu files).
// ---------------------------------------------------------------------------
// Session lists of a call, by value.  Calls of up to FEW sessions pass the small block: the
// driver copies a launch's arguments, and 4 KB of them cost more than the rest of a launch.
constexpr int FEW = 32;
template <int N>
struct AppendArgsT {
  int32_t n_seq;
  int32_t total;
  int32_t sessions[N];
  int32_t cu[N + 1];
};
using AppendArgs = AppendArgsT<MAX_SEQ>;

template <int N>
struct SeqArgsT {
  int32_t n_seq;
  int32_t sessions[N];
};
using SeqArgs = SeqArgsT<MAX_SEQ>;

// What the device runs at once, for each kernel whose launch shape follows from it.  kvc_create
// looks it up for the current CUDA context; the first time for a context and element type (about
// 3 ms) that also sets the kernels' attributes, which belong to the CUDA context too.
constexpr int PF_MAX_SLICES = 8;  // CTAs of a bfloat16 prefill cluster, at most
struct Limits {
  int sms;                         // SMs
  int dec_stream_k;                // CTAs of the stream-K decode's grid
  int dec_wide, dec_narrow;        // CTAs of the 16-warp and 4-warp pair split in one wave
  int pf_stream_k;                 // CTAs of the stream-K prefill (bfloat16)
  int pf_clusters[PF_MAX_SLICES + 1];  // [k] clusters of k CTAs of the prefill's pair split
  int f32_cluster[2][2];           // largest cluster of the binary32 prefill: [rows][spread]
};
cudaError_t query_limits(const Dev& d, Limits* lim);
// Id of the current CUDA context (never reused: a context that replaces a destroyed one at the
// same address has another).
cudaError_t current_context_id(unsigned long long* id);

cudaError_t launch_init(const Dev& d, double rope_base, cudaStream_t s);
// single: every session of the call gets exactly one token (one session: plan and K/V write in
// one launch).
cudaError_t launch_append(const Dev& d, const AppendArgs& a, const uint8_t* types, const void* k,
                          const void* v, bool single, cudaStream_t s);
// after_plan: launched right behind the plan kernel of the same append.
cudaError_t launch_append_layers(const Dev& d, int total, int layer0, int n_layers, const void* k,
                                 const void* v, bool after_plan, cudaStream_t s);
cudaError_t launch_evict(const Dev& d, const SeqArgs& a, int64_t* resident_out, int64_t* used_out,
                         int sms, cudaStream_t s);
cudaError_t launch_release(const Dev& d, const SeqArgs& a, int64_t* used_out, cudaStream_t s);
cudaError_t launch_transcript(const Dev& d, int session, int cap, int32_t* pos_out, void* k_out,
                              void* v_out, int32_t* count, cudaStream_t s);
// Attention launches may start while the kernel before them in the stream finishes.  early:
// they may also read what the append wrote before that (an attention launch of the same
// append came before, so the append is complete).
// new_k / new_v (optional): the fused per-layer write of the new tokens' K/V.
// epoch: tag of this launch's partial states (nonzero, never reused while tags
// of it may remain in the slots); 0 selects the fenced arrival instead.
// pages: estimate of the longest session's pages, for the choice of the split only.
cudaError_t launch_attn_decode(const Dev& d, const Limits& lim, int layer, const void* q,
                               void* out, int n_seq, int pages, bool early, cudaStream_t s,
                               uint32_t epoch, const void* new_k = nullptr,
                               const void* new_v = nullptr);
// Stream-K decode kernel (kvc_attn_decode.cu): its grid (resident CTAs, capped by
// the partial slots; sets its attributes) and its launch.
int decode_stream_k_grid(const Dev& d);
cudaError_t launch_attn_decode_streamk(const Dev& d, int layer, const CUtensorMap& map_lo,
                                       const CUtensorMap& map_hi, const void* q, void* out,
                                       float scale, int grid, int min_units, const void* new_k,
                                       const void* new_v, bool early, cudaStream_t s);
// Pair-split decode kernel (kvc_attn_decode_split.cu).  wide: the 16-warp shape
// (one CTA per SM; tensor-core pages for bfloat16), else the 4-warp shape.  k_most: CTAs per
// pair; fit: how the 4-warp shape counts those that work.
// Resident CTAs in one wave (sets its attributes).
int decode_split_slots(int esz, bool wide, int sms);
bool decode_split_uses_tma(int esz, bool wide);      // needs the pool's tensor maps
cudaError_t launch_attn_decode_split(const Dev& d, bool wide, int layer, const CUtensorMap& map_lo,
                                     const CUtensorMap& map_hi, const void* q, void* out,
                                     float scale, int k_most, const NarrowFit& fit,
                                     uint32_t epoch, const void* new_k, const void* new_v,
                                     int n_pairs, bool early, cudaStream_t s);
// new_k / new_v (optional, bfloat16 only): the chunk's rows of this layer, written
// into the pool by the launch itself (the per-layer order).
// pages_max, pages_sum: estimates of the sessions' resident pages (largest, sum over the
// call), for the choice of the split only.
cudaError_t launch_attn_prefill(const Dev& d, const Limits& lim, int layer, const void* q,
                                void* out, int n_seq, int max_t, int pages_max,
                                int64_t pages_sum, bool early, cudaStream_t s,
                                const void* new_k = nullptr, const void* new_v = nullptr);
// k = 0: stream-K over `grid` CTAs; k >= 1: pair split, grid = pairs * k CTAs.
cudaError_t launch_attn_prefill_tc(const Dev& d, int layer, const CUtensorMap& lo,
                                   const CUtensorMap& hi, const void* q, void* out, int grid,
                                   int k, int max_t, bool early, cudaStream_t s, const void* new_k,
                                   const void* new_v);
// Sets its attributes; CTAs of the stream-K split and clusters of the pair split at once.
cudaError_t prefill_tc_limits(Limits* lim);
// binary32; pages_max as in launch_attn_prefill.
cudaError_t prefill_f32_limits(Limits* lim);
cudaError_t launch_attn_prefill_f32(const Dev& d, const Limits& lim, int layer, const void* q,
                                    void* out, int n_seq, int max_t, int pages_max, bool early,
                                    cudaStream_t s);
// Two 2-D views of the bfloat16 pool as rows of 128 elements (columns 0-63 and
// 64-127), 16-row boxes, 128-byte swizzle; cached per pool.  False if the driver
// entry point is missing or the encoding fails.
bool pool_tensor_maps(const Dev& d, CUtensorMap* lo, CUtensorMap* hi);
int noalloc_max_pairs();
cudaError_t launch_attn_decode_noalloc(const Dev& d, int layer, const void* q, void* out,
                                       int n_seq, cudaStream_t s);

}  // namespace kvc
