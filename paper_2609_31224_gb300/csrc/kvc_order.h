// Order of the attention launches of one append (host side, no CUDA): which layers' K/V of
// the append are in the pool, and whether an attention launch may read pages before the
// kernels in front of it in the stream are complete ("early").
//
// Every attention launch lets the next one start before it has finished, so a chain of early
// launches may overlap.  The first launch after an append, or after a layer write, waits for
// it before it lets anything else start.  A fused launch writes its layer's rows itself and
// reads them from the caller's buffers, so launches on other layers may overlap it, and so may
// a fused launch on the same layer; a plain launch on that layer reads the rows from the pool
// and has to wait, after which no fused write is pending any more.
#pragma once

#include <stdint.h>

namespace kvc {

class LaunchOrder {
 public:
  // An append: of all layers' K/V, or of none (layers follow one by one).
  void append(bool with_kv, int layers) {
    written_ = !with_kv ? 0 : layers >= 64 ? ~0ull : (1ull << layers) - 1;
    settle();
  }
  // A separate write of one layer's K/V, complete before the launch behind it starts.
  void layer_write(int layer) {
    written_ |= 1ull << layer;
    settle();
  }
  bool layer_written(int layer) const { return (written_ >> layer) & 1; }

  bool early(int layer, bool fused) const {
    return waited_ && (fused || !((pending_ >> layer) & 1));
  }
  // The attention launch that early(layer, fused) was asked for is in the stream.
  void launched(int layer, bool fused) {
    if (!early(layer, fused)) pending_ = 0;
    if (fused) {
      pending_ |= 1ull << layer;
      written_ |= 1ull << layer;
    }
    waited_ = true;
  }

 private:
  void settle() {
    pending_ = 0;
    waited_ = false;
  }
  uint64_t written_ = 0;  // layers whose K/V of the append are in the pool, or will be
  uint64_t pending_ = 0;  // layers with a fused write that no launch has waited for
  bool waited_ = false;   // an attention launch has waited for the append (or layer write)
};

}  // namespace kvc
