// Dispatch of a decode attention call (one token per session) between the three
// kernel shapes, by the number of (session, KV head) pairs it has and the pages of its
// longest session (estimated on the host):
//   - pair split, 16-warp CTAs (one per SM): sessions of 100 pages or more when every
//     pair gets k >= 5 CTAs in one wave (at most 3 sessions of 8 KV heads on 152 SMs); for
//     bfloat16 the pages run on the tensor cores;
//   - pair split, 4-warp CTAs (three per SM, tensor-core pages for bfloat16): every
//     other call whose pairs each get k >= 1 CTAs in one wave (with k = 1 a pair needs no
//     merge), unless one slice each would leave many slots empty for long;
//   - stream-K over (session, KV head, page) units, tensor-core pages for bfloat16:
//     the rest (e.g. rounds of 30-50 long sessions, and calls of more pairs than the
//     4-warp shape's resident CTAs, like the full-batch rounds of 64 sessions).
#include <cstring>

#include "kvc_launch.cuh"

namespace kvc {

namespace {

constexpr int MAX_PARTS = 64;      // partial states per pair (both pair-split shapes)
constexpr float LOG2E = 1.4426950408889634f;
// Minimum (session, kv head, page) units per CTA of the stream-K split.
constexpr int DEC_MIN_UNITS = 12;
// The pair-split kernel takes calls whose pairs each get at least this many CTAs
// in one wave: with 16-warp CTAs (one per SM) first, else with stream-K's 4-warp
// CTAs (three per SM).  Only the 16-warp shape uses tagged partial states: with
// 4-warp CTAs the fenced arrival measured faster.  Against the 16-warp shape, the 4-warp
// one measured faster from 4 sessions on (15.4 against 16.7 us at 4, 26.4 against 28.1 at
// 9) and slower below (11.7 against 8.1 at 1).
constexpr int SPLIT_MIN_K = 5, SPLIT4_MIN_K = 1;
// Below this many pages the 16-warp shape leaves most of its warps without one
// (64 pages, 8 pairs: 6.8 us against 6.4-6.7 with 4 warps; 20 pages: 6.7 against 5.2).
constexpr int WIDE_MIN_PAGES = 100;

// One slice per pair against stream-K, 257 pages, 8 KV heads: 92.9 against 77.5 us at 30
// sessions (a slice's CTA takes 63 us by itself), 104.7 against 100.7 at 40, 121.4 against
// 119.7 at 48, but 128.3 against 129.4 at 52 and 137.8 against 139.8 at 57; with 38 pages
// one slice is faster throughout (14.9 against 18.1 at 30, 17.7 against 20.8 at 40).
constexpr int STREAM_K_MIN_PAGES = 128;
bool one_slice_too_few(int slots, int n_pairs, int pages) {
  return pages >= STREAM_K_MIN_PAGES && n_pairs <= slots * 7 / 8;
}

// Slices per pair of the 16-warp shape: no more than give each warp a page (257 pages, 8
// pairs: 7.6 us at 17 slices, 7.9 at 19, 8.9 at 15; 4 pairs: 7.2 at 19, 8.4 at 38).
int wide_slices(int slots, int n_pairs, int pages) {
  return min(MAX_PARTS, min(slots / n_pairs, (pages + 15) / 16));
}

// ... and of the 4-warp shape: up to 5/6 of the slots for as long as that leaves 6 slices or
// more, all of them beyond (257 pages: 14.5 us at 12 slices of 32 pairs, 15.0 at 14; 18.9 at 8
// of 48, 19.6 at 9; but 26.0 at 6 of 72, 26.5 at 5), and about three pages per slice at least
// (33 pages, one binary32 pair: 4.7 us at 12 slices, 9.9 at 64; 20 pages, 8 pairs: 5.2 at 8,
// 6.1 at 12; 17 pages: 4.5 at 6, 9.3 at 64).  The CUDA-core pages of binary32 are bound by
// the pages of a warp: there more slices are taken if they save a warp one (48 pairs of 130
// pages: 12.0 us at 9 slices, 12.5 at 8).
int narrow_slices(int slots, int n_pairs, int pages, bool cuda_cores) {
  const int five_sixths = (slots * 5 / 6 + n_pairs / 2) / n_pairs;
  int fit = five_sixths >= 6 ? five_sixths : slots / n_pairs;
  // (Two more pages than estimated: the partly filled ones of both regions.)
  auto warp_pages = [&](int k) { return ((pages + 2 + k - 1) / k + 3) / 4; };
  for (int k = fit + 1; cuda_cores && k <= slots / n_pairs; ++k)
    if (warp_pages(k) < warp_pages(fit)) fit = k;
  return max(1, min(MAX_PARTS, min(fit, (pages + 2) / 3)));
}

}  // namespace

cudaError_t launch_attn_decode(const Dev& d, int layer, const void* q, void* out, int n_seq,
                               int pages, bool early, cudaStream_t s, uint32_t epoch,
                               const void* new_k, const void* new_v) {
  const int esz = d.esz;
  // Grid sizes of the three shapes, per element type (their CTA shapes differ), worked
  // out on a thread's first call with that type.
  struct Shapes {
    int grid = 0, slots = 0, slots4 = 0;
  };
  static thread_local Shapes shapes[2];
  Shapes& sh = shapes[esz == 2 ? 1 : 0];
  if (sh.grid == 0) {
    sh.grid = decode_stream_k_grid(d);
    sh.slots = decode_split_slots(esz, true);
    sh.slots4 = decode_split_slots(esz, false);
  }
  const int grid = sh.grid, slots = sh.slots, slots4 = sh.slots4;
  const float scale = LOG2E / sqrtf((float)d.head_dim);
  const int n_pairs = n_seq * d.kv_heads;
  const int k = n_pairs * SPLIT_MIN_K <= slots && pages >= WIDE_MIN_PAGES
                    ? wide_slices(slots, n_pairs, pages) : 0;
  int k4 = k == 0 && n_pairs * SPLIT4_MIN_K <= slots4
               ? narrow_slices(slots4, n_pairs, pages, esz == 4) : 0;
  if (k4 == 1 && one_slice_too_few(slots4, n_pairs, pages)) k4 = 0;
  // Tensor maps of the pool for the tensor-core page loop (bfloat16).
  CUtensorMap map_lo, map_hi;
  memset(&map_lo, 0, sizeof(map_lo));
  memset(&map_hi, 0, sizeof(map_hi));
  // (The stream-K kernel's bfloat16 pages also run on the tensor cores.)
  if (((k > 0 && decode_split_uses_tma(esz, true)) ||
       (k4 > 0 && decode_split_uses_tma(esz, false)) || (k == 0 && k4 == 0 && esz == 2)) &&
      !pool_tensor_maps(d, &map_lo, &map_hi))
    return cudaErrorInvalidValue;
  if (k > 0) {
    const uint32_t tag = n_pairs * k <= d.dec_tag_slots ? epoch : 0u;
    return launch_attn_decode_split(d, true, layer, map_lo, map_hi, q, out, scale, k, tag, new_k,
                                    new_v, n_pairs, early, s);
  }
  if (k4 > 0)
    return launch_attn_decode_split(d, false, layer, map_lo, map_hi, q, out, scale, k4, 0u, new_k,
                                    new_v, n_pairs, early, s);
  return launch_attn_decode_streamk(d, layer, map_lo, map_hi, q, out, scale, grid, DEC_MIN_UNITS,
                                    new_k, new_v, early, s);
}

}  // namespace kvc
