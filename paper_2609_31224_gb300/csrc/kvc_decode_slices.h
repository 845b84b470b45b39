// Slices per (session, KV head) pair of the two pair-split decode shapes, by the pages of the
// call's longest session.  Those of the 4-warp shape range from 1 to 14 and follow from the pages
// that are there (nb_max of the append): the host launches as many CTAs as any number of pages
// can want, and CTAs past the count leave at once.  So a launch that was captured with short
// sessions, or one whose sessions the host estimates wrong, is cut right (8 pairs captured at one
// page and replayed at 250: 48.2 us with the host's count), and a captured launch is cut like an
// eager one.  Each CTA counts for itself; that and the CTAs without a slice cost up to 0.1 us of
// a launch, 0.4 where one slice in six is spare (72 pairs of 76 pages: 9.9 -> 10.3 us).  In the
// append kernels the count cost each of them 0.3 us.
// Those of the 16-warp shape hardly depend on the pages: they are the host's, as CTAs without a
// slice would keep the next launch's off their SM (8 pairs of 257 pages: 7.5 us with 17 slices
// launched, 7.9 with 19 of which 17 work).  Plain C++ beside CUDA, so that it is tested on the CPU.
#pragma once

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
// What follows from the pairs alone is the host's part, so that a kernel is left with two divisions.
struct NarrowFit {
  int most;         // slices that the slots and NARROW_MAX allow
  int below, from;  // of sessions below, and from, ALL_MIN_PAGES pages on
};
KVC_HD inline NarrowFit narrow_fit(int slots, int n_pairs) {
  const int most = narrow_most(slots, n_pairs);
  const int five_sixths = (slots * 5 / 6 + n_pairs / 2) / n_pairs, some = at_most(most, five_sixths);
  return {most, five_sixths >= 6 ? some : most, five_sixths >= 8 ? some : most};
}
KVC_HD inline int narrow_slices(const NarrowFit& fit, int pages, bool cuda_cores) {
  if (fit.most < 1) return 1;
  const int n = pages + 1;  // (the figures above count whole pages)
  int k = pages < ALL_MIN_PAGES ? fit.below : fit.from;
  // Pages of a warp: ceil(ceil(n / k) / NARROW_WARPS).
  if (cuda_cores) {
    const int w = div_up(n, NARROW_WARPS * fit.most);
    if (w < div_up(n, NARROW_WARPS * k)) k = div_up(n, NARROW_WARPS * w);
    return at_least(1, at_most(k, n / 2));
  }
  k = at_least(1, at_most(k, div_up(n, NARROW_WARPS)));
  return k > 5 ? at_least(5, div_up(n, NARROW_WARPS * div_up(n, NARROW_WARPS * k))) : k;
}

}  // namespace kvc
