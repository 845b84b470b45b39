// Dispatch of a decode attention call (one token per session) between the three
// kernel shapes, by the number of (session, KV head) pairs it has and the pages of its
// longest session (estimated on the host):
//   - pair split, 16-warp CTAs (one per SM): sessions of 55 pages or more of which each
//     warp gets one at most, and long bfloat16 sessions when every pair gets 6 CTAs in one
//     wave (at most 3 sessions of 8 KV heads on 152 SMs); for bfloat16 the pages run on the
//     tensor cores;
//   - pair split, 4-warp CTAs (three per SM, tensor-core pages for bfloat16): every
//     other call whose pairs each get k >= 1 CTAs in one wave (with k = 1 a pair needs no
//     merge), unless one slice each would leave many slots empty for long; k follows the
//     pages on the device (kvc_decode_slices.h);
//   - stream-K over (session, KV head, page) units, tensor-core pages for bfloat16:
//     the rest (e.g. rounds of 30-50 long sessions, and calls of more pairs than the
//     4-warp shape's resident CTAs, like the full-batch rounds of 64 sessions).
#include <cstring>
#include <mutex>

#include "kvc_launch.cuh"

namespace kvc {

namespace {

constexpr float LOG2E = 1.4426950408889634f;
// Minimum (session, kv head, page) units per CTA of the stream-K split.
constexpr int DEC_MIN_UNITS = 12;
// The pair-split kernel takes calls whose pairs each get a CTA in one wave: the 16-warp CTAs
// (one per SM) where they are the better shape, else stream-K's 4-warp CTAs (three per SM).
// Only the 16-warp shape uses tagged partial states: with 4-warp CTAs the fenced arrival
// measured faster.
//
// The 16-warp shape is the better one while each of its warps has one page at most and most
// of them have one (us, bfloat16, 16-warp against the best slices of the 4-warp one):
//   pages       8 pairs       16 pairs      20 pairs      24 pairs
//   52          6.5 / 5.8     6.5 / 6.3     6.5 / 6.5     6.7 / 6.6
//   63          6.6 / 6.4     6.5 / 6.6     6.6 / 6.8     6.8 / 6.8
//   76          6.7 / 6.5     6.7 / 6.9     6.8 / 7.1     7.2 / 7.2
//   101         6.9 / 7.0     6.9 / 7.1     7.3 / 7.3     8.6 / 7.5
//   157         6.9 / 7.5     9.4 / 8.5     9.5 / 8.6    10.0 / 8.9
//   257         7.5 / 9.5    10.5 / 10.5   12.0 / 11.1   12.6 / 11.9
// Long sessions leave both shapes' warps many pages each.  Of 257 and 501 binary32 pages, 8
// pairs take 7.9 and 11.1 us against 10.8 and 15.8, 16 pairs 11.2 and 16.7 against 11.2 and
// 16.6, 24 pairs 13.9 and 22.3 against 12.4 and 19.0: the 16-warp shape up to a ninth of the
// SMs.  bfloat16 stays with it up to a sixth, at up to 6 % more for 24 pairs, so that calls
// of one to three long sessions run one kernel; at 28 pairs the 4-warp shape is 7-12 % faster.
constexpr int WIDE_MIN_PAGES = 55;
constexpr int WIDE_LONG_K = 6, WIDE_LONG_K_F32 = 9, WIDE_LONG_PAGES = 256;
bool use_wide(int slots, int n_pairs, int pages, int esz) {
  if (pages >= WIDE_LONG_PAGES)
    return n_pairs * (esz == 2 ? WIDE_LONG_K : WIDE_LONG_K_F32) <= slots;
  return pages >= WIDE_MIN_PAGES && pages + 2 <= slots / n_pairs * WIDE_WARPS;
}

// One slice per pair against stream-K, 257 pages, 8 KV heads: 92.9 against 77.5 us at 30
// sessions (a slice's CTA takes 63 us by itself), 104.7 against 100.7 at 40, 121.4 against
// 119.7 at 48, but 128.3 against 129.4 at 52 and 137.8 against 139.8 at 57; with 38 pages
// one slice is faster throughout (14.9 against 18.1 at 30, 17.7 against 20.8 at 40).
constexpr int STREAM_K_MIN_PAGES = 128;
bool one_slice_too_few(int slots, int n_pairs, int pages) {
  return pages >= STREAM_K_MIN_PAGES && n_pairs <= slots * 7 / 8;
}

}  // namespace

cudaError_t launch_attn_decode(const Dev& d, const Limits& lim, int layer, const void* q,
                               void* out, int n_seq, int pages, bool early, cudaStream_t s,
                               uint32_t epoch, const void* new_k, const void* new_v) {
  const int esz = d.esz, slots = lim.dec_wide, slots4 = lim.dec_narrow;
  const float scale = LOG2E / sqrtf((float)d.head_dim);
  const int n_pairs = n_seq * d.kv_heads;
  const bool wide = use_wide(slots, n_pairs, pages, esz);
  const int most = n_pairs <= slots4 ? narrow_most(slots4, n_pairs) : 0;
  const bool narrow = !wide && most > 0 && !(most == 1 && one_slice_too_few(slots4, n_pairs, pages));
  // Tensor maps of the pool for the tensor-core page loop (bfloat16).
  CUtensorMap map_lo, map_hi;
  memset(&map_lo, 0, sizeof(map_lo));
  memset(&map_hi, 0, sizeof(map_hi));
  // (The stream-K kernel's bfloat16 pages also run on the tensor cores.)
  if (((wide && decode_split_uses_tma(esz, true)) || (narrow && decode_split_uses_tma(esz, false)) ||
       (!wide && !narrow && esz == 2)) &&
      !pool_tensor_maps(d, &map_lo, &map_hi))
    return cudaErrorInvalidValue;
  if (wide) {
    const int k = wide_slices(slots, n_pairs, pages);
    const uint32_t tag = n_pairs * k <= d.dec_tag_slots ? epoch : 0u;
    return launch_attn_decode_split(d, true, layer, map_lo, map_hi, q, out, scale, k, {}, tag, new_k,
                                    new_v, n_pairs, early, s);
  }
  if (narrow)
    return launch_attn_decode_split(d, false, layer, map_lo, map_hi, q, out, scale, most,
                                    narrow_fit(slots4, n_pairs), 0u, new_k, new_v, n_pairs, early, s);
  return launch_attn_decode_streamk(d, layer, map_lo, map_hi, q, out, scale, lim.dec_stream_k,
                                    DEC_MIN_UNITS, new_k, new_v, early, s);
}

namespace {

struct KnownLimits {
  unsigned long long ctx_id;
  int esz;
  Limits lim;
};
constexpr int MAX_KNOWN = 64;
KnownLimits g_known[MAX_KNOWN];
int g_n_known = 0;
std::mutex g_known_mu;

}  // namespace

cudaError_t query_limits(const Dev& d, Limits* lim) {
  std::lock_guard<std::mutex> lock(g_known_mu);
  unsigned long long id = 0;
  const bool known = current_context_id(&id) == cudaSuccess;  // (else worked out each time)
  for (int i = 0; known && i < g_n_known; ++i)
    if (g_known[i].ctx_id == id && g_known[i].esz == d.esz) {
      *lim = g_known[i].lim;
      return cudaSuccess;
    }
  memset(lim, 0, sizeof(*lim));
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&lim->sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  lim->dec_stream_k = decode_stream_k_grid(d);
  lim->dec_wide = decode_split_slots(d.esz, true, lim->sms);
  lim->dec_narrow = decode_split_slots(d.esz, false, lim->sms);
  e = d.esz == 2 ? prefill_tc_limits(lim) : prefill_f32_limits(lim);
  // A full table only means that later contexts repeat this for every kvc_create.
  if (e == cudaSuccess && known && g_n_known < MAX_KNOWN) g_known[g_n_known++] = {id, d.esz, *lim};
  return e;
}

}  // namespace kvc
