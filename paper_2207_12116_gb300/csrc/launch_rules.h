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

// Threads of a team of the mask form's propagation, for n_stores stores of `words`
// words of Booleans on `sms` SMs.  A team takes a whole store, and an SM holds 1,024
// threads and 16 teams, so
//   - the stores that an SM gets take as few turns as they can (a batch that just
//     misses one turn pays for two), and share its 32 warps evenly;
//   - a warp for at most every pair of words (two words are evaluated together), and in
//     batches of several turns for every second one: there the SM is busy anyway; at
//     least two warps: the two directions of the temporal levels;
//   - stores of more than 40 pairs at least four warps and of more than 100 eight, since
//     a hard one in few warps holds up the end.  Where that is more than their share,
//     turns are many whatever the width, and wider teams leave less of the last one
//     empty: eight warps for four, sixteen for eight when a second turn would be at most
//     a third full.
// Measured (us of kernel; a team as wide as left every warp two and a half, until
// now): 608 stores of 20 tasks 23.5 -> 12.2, 1,216 23.9 -> 14.1, 1,700 of 14 33.8 -> 23.1,
// 1,216 of 30 37.6 -> 31.3, 300 of 60 38.1 -> 23.3, 608 of 120 127 -> 104, 777 of 120 179 ->
// 161; slower 1,700 of 45 48.5 -> 51.2.  Means over six models, 2 / 3 / 4 / 5 / 6 / 8 / 16
// warps: 620 of 62 tasks 71 / 55 / 47 / 43 / 43 / 44 / 49, 1,000 87 / 66 / 56 / 67 / 70 / 61 /
// 64, 1,314 104 / 79 / 91 / 90 / 83 / 74 / 81, 2,300 99 / 110 / 96 / 96 / 95 / 90 / 109; 1,200 of
// 80 133 / 99 / 83 / 100 / 95 / 86 / 90; 1,314 of 48 62 / 48 / 59 / 58 / 55 / 52 / 61.
inline int propagation_team(int64_t n_stores, int64_t sms, int words) {
  const int64_t per_sm = std::max<int64_t>(1, (n_stores + sms - 1) / sms);
  const int64_t turns = (per_sm + 15) / 16, at_once = (per_sm + turns - 1) / turns;
  const int64_t pairs = (words + 1) / 2, share = 32 / at_once;
  int64_t least = pairs > 100 ? 8 : pairs > 40 ? 4 : 2;
  while (least < 32 && 32 * least < pairs) least *= 2;
  if (share < least) {
    const int64_t held = sms * std::min<int64_t>(16, 32 / least);
    const bool few = n_stores > held && 3 * (n_stores - held) <= held;
    if (least < 32 && (few || (least == 4 && turns <= 2))) least *= 2;
    return static_cast<int>(32 * least);
  }
  const int64_t most = std::max(least, turns == 1 ? pairs : pairs / 2);
  return static_cast<int>(32 * std::min(most, share));
}

// Stores of which the default chunks of host-memory propagation are multiples, for
// the mask form (whose teams take their size from the chunk, so that only the copies
// size it): at most eight an SM; with page-locked stores at most kHostUnitBytes of
// bounds, so that a batch of large stores is several chunks whose copies overlap
// (pageable copies do not, and every chunk more costs them a round trip).
// Whole multiples of 64 stores: each chunk of a 256-byte-aligned array then starts
// 256-byte aligned whatever the variables.  Copies that start at odd 32 bytes are slow
// (10,000 stores of 30 tasks in chunks of 2,128: 731 us, of 2,432: 635).
// Calls by the most bytes of a unit, us (9 / 12 / 18 / 24 MB, eight stores an SM alone):
// 1,216 of 60 tasks 355 / 347 / 360 / 394, 433; 1,700 464 / 450 / 451 / 486, 526; 1,216 of 40
// 197 / 205 / 225 / 224, 226; 10,000 of 30 all 636.
constexpr int64_t kHostUnitBytes = int64_t(12) << 20;

inline int64_t host_chunk_unit(int64_t store_bytes, int64_t sms, bool locked) {
  int64_t unit = 8 * sms;
  if (locked) unit = std::min(unit, kHostUnitBytes / store_bytes);
  return std::max<int64_t>(64, unit & ~static_cast<int64_t>(63));
}

}  // namespace pccp
