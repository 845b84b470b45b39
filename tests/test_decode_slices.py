"""Slices per pair of the pair-split decode (csrc/kvc_decode_slices.h), over every number of pairs
and pages: the rule in closed form, as the kernels evaluate it, against the rule as a search,
and within what the host launches.
"""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include "kvc_decode_slices.h"
#include <algorithm>
#include <cstdio>
using namespace kvc;

// The 4-warp rule by trying slice after slice.
int narrow_search(int slots, int n_pairs, int pages, bool cuda_cores) {
  const int all = std::min(NARROW_MAX, slots / n_pairs), x = pages + 1;
  auto warp_pages = [&](int k) { return ((x + k - 1) / k + 3) / 4; };
  const int five_sixths = (slots * 5 / 6 + n_pairs / 2) / n_pairs;
  int k = std::min(all, five_sixths >= (pages < 300 ? 6 : 8) ? five_sixths : all);
  if (cuda_cores) {
    for (int more = k + 1; more <= all; ++more)
      if (warp_pages(more) < warp_pages(k)) k = more;
    return std::max(1, std::min(k, x / 2));
  }
  k = std::max(1, std::min(k, (x + 3) / 4));
  while (k > 5 && warp_pages(k - 1) == warp_pages(k)) --k;
  return k;
}

int main() {
  for (int sms : {152, 148, 132, 7}) {
    for (int n_pairs = 1; n_pairs <= 3 * sms; ++n_pairs)
      for (int at = 1; at <= 1120; ++at) {
        const int pages = at <= 1100 ? at : (1 << 20) + 3 * at - 3400;  // (a session has 2^20 and a few)
        for (int cc = 0; cc < 2; ++cc) {
          const int k = narrow_slices(narrow_fit(3 * sms, n_pairs), pages, cc);
          if (k != narrow_search(3 * sms, n_pairs, pages, cc) || k < 1 ||
              k > narrow_most(3 * sms, n_pairs)) {
            std::printf("4 warps, %d SMs, %d pairs, %d pages: %d\n", sms, n_pairs, pages, k);
            return 1;
          }
        }
        if (n_pairs > sms) continue;
        const int k = wide_slices(sms, n_pairs, pages);
        if (k != std::min(std::min(64, sms / n_pairs), std::max(17, (pages + 17) / 16)) || k < 1 ||
            k > SLICES_MAX) {
          std::printf("16 warps, %d SMs, %d pairs, %d pages: %d\\n", sms, n_pairs, pages, k);
          return 1;
        }
      }
  }
  return 0;
}
"""


def test_slices(tmp_path):
    src, exe = tmp_path / "slices.cpp", tmp_path / "slices"
    src.write_text(PROGRAM)
    inc = os.path.join(ROOT, "paper_2609_31224_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", inc, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
