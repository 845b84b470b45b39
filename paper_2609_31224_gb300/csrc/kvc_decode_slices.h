// Slices per (session, KV head) pair of the two pair-split decode shapes.  Those of the 4-warp
// shape range from 1 to 14 and follow from the pages of the pair's session: the host launches as
// many CTAs as any number of pages can want, each counts the slices for itself, and those past
// the count leave at once.  So a launch that was captured with short sessions, or one whose
// sessions the host estimates wrong, is cut right (8 pairs captured at one page and replayed at
// 250: 48.2 us with the host's count), and a captured launch is cut like an eager one.  (The count
// in the append kernels cost each of them 0.3 us; from the call's longest session, one address
// that every CTA reads, it cost a decode launch up to 0.3.)
// Those of the 16-warp shape hardly depend on the pages: they are the host's, as CTAs without a
// slice would keep the next launch's off their SM (8 pairs of 257 pages: 7.5 us with 17 slices
// launched, 7.9 with 19 of which 17 work).  Plain C++ beside CUDA, so that it is tested on the CPU.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define KVC_HD __host__ __device__
#else
#define KVC_HD
#endif

namespace kvc {

constexpr int SLICES_MAX = 64;                 // partial states per pair that a merge takes
constexpr int WIDE_WARPS = 16, NARROW_WARPS = 4;
constexpr int NARROW_MAX = 14, ALL_MIN_PAGES = 300;

KVC_HD inline int at_most(int a, int b) { return a < b ? a : b; }
KVC_HD inline int at_least(int a, int b) { return a > b ? a : b; }
KVC_HD inline int div_up(int a, int b) { return ((unsigned)a + b - 1) / (unsigned)b; }  // a, b > 0

// The most slices of a call with n_pairs pairs, whatever its pages (slots: CTAs in one wave).
KVC_HD inline int narrow_most(int slots, int n_pairs) { return at_most(NARROW_MAX, slots / n_pairs); }

// 16-warp shape: 17, which gives 272 pages a warp each, and more for longer sessions (8 pairs
// of 257 pages: 7.5 us at 17 slices, 8.2 at 19, 8.8 at 15; of 157: 6.9 at 17, 7.1 at 11; 4
// pairs of 257: 7.2 at 19, 8.4 at 38).
KVC_HD inline int wide_slices(int slots, int n_pairs, int pages) {
  return at_most(at_most(SLICES_MAX, slots / n_pairs), at_least(17, div_up(pages + 2, WIDE_WARPS)));
}

// 4-warp shape.  Up to 5/6 of the slots for as long as that leaves 6 slices or more, all of them
// beyond (257 pages: 14.5 us at 12 slices of 32 pairs, 15.0 at 14; 18.9 at 8 of 48, 19.6 at 9;
// but 26.0 at 6 of 72, 26.5 at 5), from 300 pages on as long as it leaves 8 (64 pairs: 39.9 us
// at 7 slices of 501 pages, 41.4 at 6, but 24.0 and 23.1 of 257); and no more than 14, as the
// merge is the dearer part beyond (8 pairs of 52 pages: 5.8 us at 14 slices, 6.3 at 16, 6.7 at
// 18; of 76: 6.5, 7.1, 7.2).
// bfloat16 takes a page per warp at least, and the fewest slices, from 5 on, that leave a warp as
// few pages (72 pairs of 76 pages: 9.9 us at 5 slices, 10.7 at 6; 32 of 157: 10.2 at 10, 10.7 at
// 12; 16 of 29: 5.7 at 8, 6.3 at 10).  The CUDA-core pages of binary32 are bound by the pages
// of a warp: about two pages per slice at least (20 pages, 16 pairs: 4.9 us at 11 slices, 5.2
// at 8; 24 pairs: 5.0 and 5.2), and more slices if they save a warp one (48 pairs of 130
// pages: 12.0 us at 9 slices, 12.5 at 8).
//
// What follows from the pairs alone is the host's part.  A kernel is left with one division, for
// long sessions: it comes before a CTA's first load, and three of them took 0.1-0.4 us.
struct WarpPages {  // pages of a warp with k slices: n / (4 k) rounded up, as a product
  int d;            // 4 k
  uint32_t inv;     // 2^32 / d rounded up: exact up to 2^32 / d pages
  KVC_HD int of(int n) const { return (int)(((uint64_t)(uint32_t)(n + d - 1) * inv) >> 32); }
};
inline WarpPages warp_pages(int k) {
  const int d = NARROW_WARPS * (k > 0 ? k : 1);
  return {d, (uint32_t)(((1ull << 32) + d - 1) / d)};
}
struct NarrowFit {
  int most;         // slices that the slots and NARROW_MAX allow
  int below, from;  // of sessions below, and from, ALL_MIN_PAGES pages on
  WarpPages w_most, w_below, w_from;
};
inline NarrowFit narrow_fit(int slots, int n_pairs) {
  const int most = narrow_most(slots, n_pairs);
  const int five_sixths = (slots * 5 / 6 + n_pairs / 2) / n_pairs, some = at_most(most, five_sixths);
  const int below = five_sixths >= 6 ? some : most, from = five_sixths >= 8 ? some : most;
  return {most, below, from, warp_pages(most), warp_pages(below), warp_pages(from)};
}
KVC_HD inline int narrow_slices(const NarrowFit& fit, int pages, bool cuda_cores) {
  const int n = pages + 1;  // (the figures above count whole pages)
  const bool shorter = pages < ALL_MIN_PAGES;
  const int k = shorter ? fit.below : fit.from;
  const int w = (shorter ? fit.w_below : fit.w_from).of(n);
  const int quarter = (n + NARROW_WARPS - 1) / NARROW_WARPS;  // slices with a page per warp
  if (cuda_cores) {
    const int w_most = fit.w_most.of(n);
    const int more = w_most >= w ? k : w_most == 1 ? quarter : div_up(quarter, w_most);
    return at_least(1, at_most(more, n / 2));
  }
  if (quarter <= k) return quarter;
  return k > 5 ? at_least(5, div_up(quarter, w)) : at_least(1, k);
}

}  // namespace kvc
