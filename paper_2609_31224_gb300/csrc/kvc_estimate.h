// Estimate of a session's resident positions (host side, no CUDA).  The host knows how many
// tokens it feeds, not their types, and so not what eviction leaves; the device's counts are
// not waited for.  The estimate guides the shape of the attention launches only, whose kernels
// take their ranges from the device's page lists.
//
// What the unit and position rules cannot remove bounds it from below: transcripts, text and
// the W newest units stay whatever the budget is.  Duplex speech as synth/script.py makes it
// keeps a sixth of what it feeds (0.16-0.17) and has about 19 positions of a unit to evict.
// Streams of other proportions are estimated off, sessions at their budget or below it are not.
#pragma once

#include <algorithm>
#include <cstdint>

#include "../../include/kvc.h"

namespace kvc {

class ResidentEstimate {
 public:
  int64_t positions() const { return resident_; }
  void append(int tokens) {
    fed_ += tokens;
    resident_ += tokens;
  }
  void evict(const kvc_config& c) { resident_ = std::min(resident_, kept(c, fed_)); }
  void release() { fed_ = resident_ = 0; }

  // Positions that an eviction leaves of a session of `fed`, as far as it has as many.
  static int64_t kept(const kvc_config& c, int64_t fed) {
    if (c.policy == KVC_POLICY_SINK_RECENT) return (int64_t)c.sink + c.recent;
    if (c.budget < 0) return fed;
    return std::max<int64_t>(c.budget, fed / KEPT_OF + (int64_t)c.window * EVICTABLE_PER_UNIT);
  }

 private:
  static constexpr int KEPT_OF = 6, EVICTABLE_PER_UNIT = 19;
  int64_t fed_ = 0, resident_ = 0;
};

}  // namespace kvc
