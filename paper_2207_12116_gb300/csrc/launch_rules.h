// launch_rules.h -- arithmetic of the launch planners that needs no device
// (plain C++: checked on the host).
#pragma once

#include <algorithm>
#include <cstdint>

namespace pccp {

// Threads of a team that evaluates `rows` propagator rows at `per_thread` rows a
// thread, where `teams` teams share a CTA of at most `cta` threads: whole warps
// (teams synchronise by named barriers over whole warps, and their warps vote
// and shuffle with full masks), at least one.
inline int team_for_rows(int64_t rows, int64_t per_thread, int cta, int teams) {
  const int64_t most = std::max(32, (cta / teams) & ~31);
  const int64_t want = ((rows + per_thread - 1) / per_thread + 31) & ~static_cast<int64_t>(31);
  return static_cast<int>(std::min(most, std::max<int64_t>(32, want)));
}

}  // namespace pccp
