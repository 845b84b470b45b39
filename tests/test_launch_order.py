"""Which attention launches may read pages before the kernels in front of them are complete
(csrc/kvc_order.h): never one that would read rows that an overlapping launch writes.  The
header is plain C++, so the rule is run here without a GPU, over every short sequence of calls.
"""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "kvc_order.h"
#include <cstdio>
#include <vector>

// Launches in stream order with what each writes and reads from the pool; `early` ones may
// overlap every launch back to the last one that waited before it let others start.
struct Model {
  kvc::LaunchOrder order;
  bool append_done = false;        // some launch behind the append has waited for it
  std::vector<int> fused_open;     // layers of fused launches that no launch has waited for
  bool attention(int layer, bool fused) {
    const bool early = order.early(layer, fused);
    if (!early) {
      append_done = true;
      fused_open.clear();
    } else {
      if (!append_done) return false;
      for (int l : fused_open)
        if (l == layer && !fused) return false;
    }
    if (fused) fused_open.push_back(layer);
    order.launched(layer, fused);
    return order.layer_written(layer);
  }
  bool op(int o) {  // 0-1 plain, 2-3 fused, 4-5 layer write, 6 append
    if (o < 4) return attention(o & 1, o >= 2);
    if (o < 6) {
      order.layer_write(o & 1);
      fused_open.clear();  // (the write itself starts behind everything before it)
    } else {
      order.append(true, 2);
    }
    append_done = false;
    if (o == 6) fused_open.clear();
    return true;
  }
};

int main() {
  for (int len = 1; len <= 6; ++len) {
    long n = 1;
    for (int i = 0; i < len; ++i) n *= 7;
    for (long s = 0; s < n; ++s) {
      Model m;
      m.op(6);
      long x = s;
      for (int i = 0; i < len; ++i, x /= 7)
        if (!m.op((int)(x % 7))) {
          std::printf("sequence %ld of length %d fails at call %d\n", s, len, i);
          return 1;
        }
    }
  }
  // What overlaps still does: layer after layer, of either kind.
  kvc::LaunchOrder o;
  o.append(false, 64);
  if (o.layer_written(0) || o.layer_written(63) || o.early(0, true)) return 2;
  for (int l = 0; l < 64; ++l) {
    if (o.early(l, true) != (l > 0)) return 3;
    o.launched(l, true);
  }
  if (o.early(63, false) || !o.early(63, true) || !o.layer_written(63)) return 4;
  o.launched(63, false);
  for (int l = 0; l < 64; ++l)
    if (!o.early(l, false)) return 5;
  o.append(true, 64);
  return o.layer_written(63) && !o.early(0, false) ? 0 : 6;
}
"""


def test_no_early_read_of_rows_in_flight(tmp_path):
    src, exe = tmp_path / "order.cpp", tmp_path / "order"
    src.write_text(PROGRAM)
    inc = os.path.join(ROOT, "paper_2609_31224_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", inc, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_the_library_asks_it():
    """No attention call decides by itself: each passes order.early() and reports back."""
    text = open(os.path.join(ROOT, "paper_2609_31224_gb300", "csrc", "kvc_api.cu")).read()
    calls = text.count("launch_attn_decode(") + text.count("launch_attn_prefill(")
    assert calls == 5
    assert text.count("order.early(") == calls and text.count("order.launched(") == calls
