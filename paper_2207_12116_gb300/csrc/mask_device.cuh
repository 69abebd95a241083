// mask_device.cuh -- the mask form of a model and its fixed point.
//
// A model whose Booleans appear only as the b of one reified row each and in
// all-positive 0/1 linear rows (overlap Booleans and resource sums) has a
// second packed table.  Its Booleans are bits, 32 to a store slot {lower
// bits, upper bits}, and the Booleans that share linear rows (one column of
// the overlap matrix) share words, so that
//   - a linear row sum a_k x_k <= c is the bit planes of its coefficients:
//     S = sum_p 2^p popc(lower & plane_p), one thread per row, four planes and
//     one slot per load instead of a term and an interval per term;
//   - a warp evaluates the reified rows of a word together, a lane a bit: both
//     operands are one load each, the Boolean's bits are a broadcast, and the
//     Booleans decided are two ballots joined by one atomic each.
// Rows of one word repeat from column to column (the same tasks and
// durations), so words share patterns, and linear rows share planes: the
// table of 120 tasks and 4 resources is 30 KB instead of 570 KB and its store
// 4.7 KB instead of 116 KB.  The rules are those of eval_reified and
// eval_linear_thread_at, so the fixed point is theirs (Sec. 3).
//
// What bounds it: instruction issue.  Per 32 reified rows about 30 warp
// instructions (a pair of rows took about 100 thread instructions with
// intervals), per resource row about 25 thread instructions (520).
#pragma once

#include <cstddef>

#include "pccp_device.cuh"

namespace pccp {

// Sections of a mask image, read through 32-bit shared-memory addresses.  Slots
// and variables are byte offsets into the store (8 bytes a slot, so at most
// 8,191 slots).
//   temporal rows and levels  uint2 {x | y << 16, d}
//   word descriptor  uint4 {lanes with a row, slot, y of every row or 0,
//                           byte offset of its pattern}; in pairs, the last
//                           pair filled with one that has no lanes
//   pattern          uint2 [32] {x | y << 16, d}, a lane each; y is added to the
//                           descriptor's (one of the two is 0)
//   mask row         uint4 {c, first full word's slot | full words << 16 |
//                           slots from one to the next << 24 (its only word's
//                           slot when one_word),
//                           byte offset of its planes,
//                           slot of the partial word or kNoSlot | largest coefficient << 16}
//   planes           uint4 [words][n_pq]: planes 4q .. 4q + 3, least
//                           significant first; full words, then the partial one
// A row's group of Booleans fills `full` words; its rest sits in a
// partial word that other groups may share.
constexpr uint32_t kNoSlot = 0xffffu;
constexpr int kRowFullMax = 255, kRowStrideMax = 255;  // what a mask row can hold
// Units of an interval variable (searches) and its paths (see pack_mask).
constexpr uint16_t kUnitNone = 0xffffu, kUnitCross = 0x8000u;
constexpr int16_t kNoPath = INT16_MIN;

// Map entry of one of the caller's variables (staging and write-back): its
// slot, its bit in the slot, whether it is an interval, its root bounds when it is a bit.
constexpr uint32_t kMapInterval = 1u << 21, kMapRootLb = 1u << 22, kMapRootUb = 1u << 23;

// A staged mask image: every phase reads the header fields it needs from
// shared memory (a broadcast load each), so that they hold no registers between phases.
struct MTab {
  uint32_t img;  // shared-memory address of the image
  bool levels;   // the temporal rows run in levels
};

// What a phase of the fixed point found (joined over the team's threads).
constexpr uint32_t kEvFail = 1u;   // an interval or a Boolean is empty
constexpr uint32_t kEvTime = 2u;   // an interval moved
constexpr uint32_t kEvRaise = 4u;  // a Boolean became 1
constexpr uint32_t kEvClear = 8u;  // a mask row set a Boolean to 0
constexpr uint32_t kEvError = 16u;  // the iteration budget ran out

// Per-team control words of the fixed point (shared memory), followed by the
// words' watch masks (a word per word of Booleans: those that would tell
// something if they became 0, as of the word phase; 0 for a word without a
// reified row, cleared by the kernel) and two bitmaps over the
// words: those in which a mask row cleared a watched Boolean (written in one
// round's row phase, read in the next round's word phase).
struct MaskCtrl {
  uint32_t ev[3];  // events of the phases, in rotation
  uint32_t evals;  // rows evaluated in dirty words
};
static_assert(sizeof(MaskCtrl) == 16, "control words");

__host__ __device__ __forceinline__ int mask_ctrl_words(int n_words) {
  return 4 + ((n_words + 2 * ((n_words + 31) / 32) + 3) & ~3);
}

// Table loads (constant while the kernel runs) and store loads (relaxed, as ld_dom).
__device__ __forceinline__ uint4 lds128(uint32_t p) {
  uint4 r;
  asm("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "r"(p));
  return r;
}

__device__ __forceinline__ uint2 lds64(uint32_t p) {
  uint2 r;
  asm("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(r.x), "=r"(r.y) : "r"(p));
  return r;
}

__device__ __forceinline__ int lds32(uint32_t p) {
  int r;
  asm("ld.shared.s32 %0, [%1];" : "=r"(r) : "r"(p));
  return r;
}

__device__ __forceinline__ uint32_t lds16(uint32_t p) {
  uint16_t r;
  asm("ld.shared.u16 %0, [%1];" : "=h"(r) : "r"(p));
  return r;
}

__device__ __forceinline__ int lds16s(uint32_t p) {
  int16_t r;
  asm("ld.shared.s16 %0, [%1];" : "=h"(r) : "r"(p));
  return r;
}

__device__ __forceinline__ int lds32v(uint32_t p) {  // a word that the team writes
  int r;
  asm volatile("ld.shared.s32 %0, [%1];" : "=r"(r) : "r"(p) : "memory");
  return r;
}

__device__ __forceinline__ int2 ld_slot(uint32_t p) {
  int2 r;
  asm volatile("ld.relaxed.cta.shared::cta.v2.s32 {%0, %1}, [%2];" : "=r"(r.x), "=r"(r.y) : "r"(p));
  return r;
}

__device__ __forceinline__ void red_max_at(uint32_t p, int v) {
  asm volatile("red.relaxed.cta.shared::cta.max.s32 [%0], %1;" ::"r"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void red_min_at(uint32_t p, int v) {
  asm volatile("red.relaxed.cta.shared::cta.min.s32 [%0], %1;" ::"r"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void red_add_at(uint32_t p, uint32_t v) {
  asm volatile("red.relaxed.cta.shared::cta.add.u32 [%0], %1;" ::"r"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void red_or_at(uint32_t p, uint32_t v) {
  asm volatile("red.relaxed.cta.shared::cta.or.b32 [%0], %1;" ::"r"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void red_and_at(uint32_t p, uint32_t v) {
  asm volatile("red.relaxed.cta.shared::cta.and.b32 [%0], %1;" ::"r"(p), "r"(v) : "memory");
}

// Header field of a mask image; m_sec: shared-memory address of a section.
__device__ __forceinline__ int m_field(const MTab& tb, size_t offset) {
  return lds32v(tb.img + static_cast<uint32_t>(offset));
}
#define PCCP_MF(field) m_field(tb, offsetof(TableHeader, field))
#define PCCP_MSEC(field) (tb.img + static_cast<uint32_t>(PCCP_MF(field)))

__device__ __forceinline__ MTab make_mtab(const uint8_t* img, int levels) {
  MTab tb{smem_u32(img), false};
  tb.levels = levels && PCCP_MF(n_tlev) > 0;
  return tb;
}

// Team barriers: a one-warp team needs no named barrier.
template <bool kWarp>
__device__ __forceinline__ void mbar_team(const Team& tm) {
  if (kWarp)
    __syncwarp();
  else
    team_bar(tm.bar, tm.nthr);
}

template <bool kWarp>
__device__ __forceinline__ bool mbar_team_or(const Team& tm, bool p) {
  if (kWarp) {
    __syncwarp();
    return __any_sync(0xffffffffu, p);
  }
  return team_bar_or(tm.bar, tm.nthr, p);
}

// Marks a told interval in the bitmap of moved variables (searches; 0: none).
template <bool kMark>
__device__ __forceinline__ void m_moved(uint32_t st, uint32_t p, uint32_t moved) {
  if (kMark) {
    const uint32_t v = (p - st) >> 3;
    red_or_at(moved + 4 * (v >> 5), 1u << (v & 31u));
  }
}

// Joins of a bound of the variable at p, seen by this thread as `seen`, without
// the old value: the event may also report a move that another thread made
// further meanwhile.
template <bool kMark = false>
__device__ __forceinline__ void m_raise(uint32_t p, int cand, int2 seen, uint32_t& ev,
                                        uint32_t st = 0u, uint32_t moved = 0u) {
  if (cand <= seen.x) return;
  if (cand > seen.y) {
    ev |= kEvFail;
  } else {
    red_max_at(p, cand);
    m_moved<kMark>(st, p, moved);
    ev |= kEvTime;
  }
}

template <bool kMark = false>
__device__ __forceinline__ void m_lower(uint32_t p, int cand, int2 seen, uint32_t& ev,
                                        uint32_t st = 0u, uint32_t moved = 0u) {
  if (cand >= seen.y) return;
  if (cand < seen.x) {
    ev |= kEvFail;
  } else {
    red_min_at(p + 4, cand);
    m_moved<kMark>(st, p, moved);
    ev |= kEvTime;
  }
}

// Ends a phase: the team's events since the last one.  `at` rotates over the
// three event words: the next phase's is cleared a phase ahead, after every
// reader of its last use has passed a barrier.
template <bool kWarp>
__device__ __forceinline__ uint32_t m_events(const Team& tm, MaskCtrl* mc, uint32_t ev, int& at) {
  ev = __reduce_or_sync(0xffffffffu, ev);
  if (kWarp) {
    __syncwarp();
    return ev;
  }
  const int next = at == 2 ? 0 : at + 1;
  if (tm.tid == 0) mc->ev[next] = 0u;
  const uint32_t p = smem_u32(&mc->ev[at]);
  if (tm.lane == 0 && ev) red_or_at(p, ev);
  team_bar(tm.bar, tm.nthr);
  at = next;
  return static_cast<uint32_t>(ld_relaxed(reinterpret_cast<const int*>(&mc->ev[next == 0 ? 2 : next - 1])));
}

// The reified rows of K words by one warp: row of lane l is
// b <=> (x <= y and y < x + d) with b bit l of the word's slot.  With
// g1 = lb y - ub x and g2 = ub y - lb x the conjunction is entailed when
// g1 >= 0 and g2 < d, its negation when g2 < 0 or g1 >= d; a Boolean already
// decided the way its entailed side says tells nothing on non-empty intervals
// (an empty one is found by the final scan).  What the lanes found meets in
// three ballots, so a word with nothing to tell (two thirds of them on search
// nodes of 30 tasks) ends at one warp-uniform branch.  The loads of the K
// words come before their first use.  watch: address of slot 0's watch mask (a
// word a slot).  kMark (searches): moved intervals go to the bitmap `moved`,
// words with a raised Boolean to the bitmap `raised` (slot 0's word a bit).
template <int K, bool kMark = false>
__device__ __forceinline__ void m_words(uint32_t st, const uint4 (&D)[K], const uint2 (&row)[K],
                                        uint32_t lane_bit, uint32_t watch, uint32_t& ev,
                                        uint32_t moved = 0u, uint32_t raised = 0u, uint32_t bit0 = 0u) {
  int2 W[K], X[K], Y[K];
  uint32_t px[K], py[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    px[k] = st + (row[k].x & 0xffffu);
    py[k] = st + D[k].z + (row[k].x >> 16);
    W[k] = ld_slot(st + D[k].y);
    X[k] = ld_slot(px[k]);
    Y[k] = ld_slot(py[k]);
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int d = static_cast<int>(row[k].y);
    const int g1 = Y[k].x - X[k].y, g2 = Y[k].y - X[k].x;
    const bool a = g1 >= 0, b = g2 < d;
    const bool n = g2 < 0 || g1 >= d;
    const uint32_t ent = __ballot_sync(0xffffffffu, a && b);
    const uint32_t neg = __ballot_sync(0xffffffffu, n);
    const uint32_t half = __ballot_sync(0xffffffffu, (a || b) && !n);
    const uint32_t lo = static_cast<uint32_t>(W[k].x), up = static_cast<uint32_t>(W[k].y);
    const uint32_t raise = D[k].x & ent & ~lo, clear = D[k].x & neg & up;
    const uint32_t act = D[k].x & ((lo & ~ent) | (~up & half));
    if (lane_bit == 1u && D[k].x != 0u)  // (a filler has another descriptor's slot)
      asm volatile("st.shared.u32 [%0], %1;" ::"r"(watch + (D[k].y >> 1)), "r"(half & D[k].x)
                   : "memory");
    if (raise | clear | act) {
      if (raise | clear) {
        if (raise) ev |= kEvRaise;
        if ((raise & ~up) | (clear & lo)) ev |= kEvFail;
        if (lane_bit == 1u) {
          if (raise) {
            red_or_at(st + D[k].y, raise);
            if (kMark) {
              const uint32_t w = (D[k].y >> 3) - bit0;
              red_or_at(raised + 4 * (w >> 5), 1u << (w & 31u));
            }
          }
          if (clear) red_and_at(st + D[k].y + 4, ~clear);
        }
      }
      if (act & lane_bit) {
        int nlx = X[k].x, nux = X[k].y, nly = Y[k].x, nuy = Y[k].y;
        if (lo & lane_bit) {  // b: x <= y and y <= x + d - 1
          nux = min(nux, Y[k].y);
          nly = max(nly, X[k].x);
          nuy = min(nuy, X[k].y + d - 1);
          nlx = max(nlx, Y[k].x - d + 1);
        }
        if (!(up & lane_bit) && a) {  // not b, x <= y holds: x + d <= y
          nly = max(nly, X[k].x + d);
          nux = min(nux, Y[k].y - d);
        }
        if (!(up & lane_bit) && b) {  // not b, y < x + d holds: y + 1 <= x
          nlx = max(nlx, Y[k].x + 1);
          nuy = min(nuy, X[k].y - 1);
        }
        if (nlx > X[k].x || nux < X[k].y || nly > Y[k].x || nuy < Y[k].y) {
          m_raise<kMark>(px[k], nlx, X[k], ev, st, moved);
          m_lower<kMark>(px[k], nux, X[k], ev, st, moved);
          m_raise<kMark>(py[k], nly, Y[k], ev, st, moved);
          m_lower<kMark>(py[k], nuy, Y[k], ev, st, moved);
        }
      }
    }
  }
}

// Bits of one quad of planes whose coefficients exceed slack's digits, given
// those equal so far (bit-sliced comparison, most significant plane first).
__device__ __forceinline__ void m_above(uint4 p, int slack, uint32_t& gt, uint32_t& eq) {
  const uint32_t pl[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
  for (int k = 3; k >= 0; --k) {
    const uint32_t s = static_cast<uint32_t>(-((slack >> k) & 1));  // all ones: the digit is 1
    gt |= eq & pl[k] & ~s;
    eq &= ~(pl[k] ^ s);
  }
}

__device__ __forceinline__ int m_sum(uint4 p, uint32_t lo) {
  return __popc(lo & p.x) + 2 * __popc(lo & p.y) + 4 * __popc(lo & p.z) + 8 * __popc(lo & p.w);
}

// The mask row cleared Booleans of the word at slot address `slot`: the word
// runs again when one of them is watched.
__device__ __forceinline__ void m_cleared(const MTab& tb, uint32_t st, uint32_t slot, uint32_t bits,
                                          uint32_t watch, uint32_t dirty, uint32_t& ev) {
  red_and_at(slot + 4, ~bits);
  if (!(static_cast<uint32_t>(lds32v(watch + ((slot - st) >> 1))) & bits)) return;
  const uint32_t w = ((slot - st) >> 3) - static_cast<uint32_t>(PCCP_MF(bit0));
  red_or_at(dirty + 4 * (w >> 5), 1u << (w & 31u));
  ev |= kEvClear;
}

// Mask row sum a_k x_k <= c by one thread: S from the lower bits; a Boolean
// still open whose coefficient exceeds c - S is lowered to 0.  kOne: every row
// of the model has one word and one quad of planes.
template <bool kOne>
__device__ __forceinline__ void m_row(const MTab& tb, uint32_t planes, int n_pq, uint32_t st, uint4 R,
                                      uint32_t watch, uint32_t dirty, uint32_t& ev) {
  const int c = static_cast<int>(R.x), top = static_cast<int>(R.w >> 16);
  const uint32_t P = planes + R.z;
  if (kOne) {
    const uint32_t slot = st + R.y;
    const int2 W = ld_slot(slot);
    const uint4 p = lds128(P);
    const int slack = c - m_sum(p, static_cast<uint32_t>(W.x));
    if (slack >= top) return;
    if (slack < 0) {
      ev |= kEvFail;
      return;
    }
    uint32_t gt = 0u, eq = 0xffffffffu;
    m_above(p, slack, gt, eq);
    const uint32_t tell = gt & static_cast<uint32_t>(W.y) & ~static_cast<uint32_t>(W.x);
    if (tell) m_cleared(tb, st, slot, tell, watch, dirty, ev);
    return;
  }
  const uint32_t rest = R.w & 0xffffu;
  const int full = static_cast<int>((R.y >> 16) & 255u);
  const uint32_t slot0 = st + (R.y & 0xffffu), stride = 8u * (R.y >> 24);
  const int words = full + (rest != kNoSlot ? 1 : 0);
  int S = 0;
  for (int w = 0; w < words; ++w) {
    const uint32_t lo = static_cast<uint32_t>(ld_slot(w < full ? slot0 + stride * w : st + rest).x);
    for (int q = 0; q < n_pq; ++q) S += m_sum(lds128(P + 16 * (w * n_pq + q)), lo) << (4 * q);
  }
  const int slack = c - S;
  if (slack >= top) return;
  if (slack < 0) {
    ev |= kEvFail;
    return;
  }
  for (int w = 0; w < words; ++w) {
    const uint32_t slot = w < full ? slot0 + stride * w : st + rest;
    const int2 W = ld_slot(slot);
    uint32_t gt = 0u, eq = static_cast<uint32_t>(W.y) & ~static_cast<uint32_t>(W.x);
    if (eq == 0u) continue;
    for (int q = n_pq - 1; q >= 0; --q) m_above(lds128(P + 16 * (w * n_pq + q)), slack >> (4 * q), gt, eq);
    if (gt) m_cleared(tb, st, slot, gt, watch, dirty, ev);
  }
}

// One temporal row x + d <= y.
__device__ __forceinline__ void m_temporal(uint32_t st, uint2 row, uint32_t& ev) {
  const uint32_t px = st + (row.x & 0xffffu), py = st + (row.x >> 16);
  const int d = static_cast<int>(row.y);
  const int2 X = ld_slot(px), Y = ld_slot(py);
  m_lower(px, Y.y - d, X, ev);
  m_raise(py, X.x + d, Y, ev);
}

// The temporal rows in topological levels (temporal_levels) by one warp:
// lower bounds up the levels by its first kUp lanes, upper bounds down them by
// its other kDown lanes.  A team of one warp runs both at once with half a warp
// each, a larger one a warp for each direction.
template <int kUp, int kDown>
__device__ __forceinline__ void m_levels(const MTab& tb, uint32_t st, int lane, uint32_t& ev) {
  const int n = PCCP_MF(n_tlev);
  const uint32_t tlev_off = PCCP_MSEC(off_tlev);
  const uint32_t tlev = tlev_off + static_cast<uint32_t>(align16_dev(4 * (n + 1)));
  const bool up = lane < kUp;
  const int first = up ? lane : lane - kUp, step = up ? kUp : kDown;
  uint32_t off = tlev_off + (up ? 0u : 4u * static_cast<uint32_t>(n - 1));
  int lo = lds32(off), hi = lds32(off + 4);
  for (int k = 1; k <= n; ++k) {
    off += up ? 4 : -4;
    int nlo = 0, nhi = 0;
    if (k < n) {
      nlo = lds32(off);
      nhi = lds32(off + 4);
    }
    for (int r = lo + first; r < hi; r += step) {
      const uint2 row = lds64(tlev + 8 * static_cast<uint32_t>(r));
      const uint32_t px = st + (row.x & 0xffffu), py = st + (row.x >> 16);
      const int d = static_cast<int>(row.y);
      const int2 X = ld_slot(px), Y = ld_slot(py);
      if (up)
        m_raise(py, X.x + d, Y, ev);
      else
        m_lower(px, Y.y - d, X, ev);
    }
    __syncwarp();
    lo = nlo;
    hi = nhi;
  }
}

// Rounds and rows of a fixed point (team-uniform; dirty words' rows aside).
struct MaskWork {
  int rounds, t, words, rows;  // rounds, passes over the temporal rows, the words, the mask rows
};

// Fixed-point loop of one team; st is staged and published.  `at` (team-uniform,
// kept from one fixed point of the team to the next) starts at 0 with the
// control words and the watch masks cleared.  A round is three phases, each ended by the
// team's events: the temporal rows to their closure, the words, the mask rows.
// A later phase sees what the earlier ones told, so a phase runs again only
// after an event that can give it something to tell:
//   - temporal rows and all words after a word moved an interval (the
//     temporal phase ends closed, and the words follow it);
//   - words in which a mask row cleared a Boolean that then tells something (a
//     Boolean that a word itself decides is entailed by the intervals it was
//     decided from, so that word tells nothing more for it);
//   - mask rows after a Boolean was raised (clearing one moves no sum).
// The last round of a plain sweep loop, which changes nothing, is most of its
// work here on search nodes: 10,000 of 30 tasks take 1.87 such sweeps.
// rows_first: the mask rows run in the first round whatever the words told
// (false for a fixed point of which only intervals moved since).
template <bool kWarp>
__device__ __forceinline__ int m_fixpoint(const MTab& tb, int2* store, const Team& tm, MaskCtrl* mc,
                                          bool rows_first, int max_iter, int& at, MaskWork& work) {
  const uint32_t st = smem_u32(store);
  const uint32_t lane_bit = 1u << tm.lane;
  // watch masks and bitmaps by word of Booleans; `watch` is where slot 0's would be
  uint32_t watch, dirty, spare;
  {
    const int bit0 = PCCP_MF(bit0), n_words = PCCP_MF(n_slots) - bit0;
    dirty = smem_u32(mc + 1) + 4 * static_cast<uint32_t>(n_words);
    spare = dirty + 4 * static_cast<uint32_t>((n_words + 31) / 32);
    watch = smem_u32(mc + 1) - 4 * static_cast<uint32_t>(bit0);
  }
  bool full = true;
  work.rounds = work.t = work.words = work.rows = 0;
  for (;;) {
    ++work.rounds;
    uint32_t ev = 0u;
    const int n_t = full ? PCCP_MF(n_t) : 0;
    if (n_t > 0) {
      if (tb.levels) {
        if (kWarp) {
          m_levels<16, 16>(tb, st, tm.lane, ev);
        } else {
          if (tm.warp == 0) m_levels<32, 0>(tb, st, tm.lane, ev);
          if (tm.warp == (tm.nwarps > 1 ? 1 : 0)) m_levels<0, 32>(tb, st, tm.lane, ev);
        }
        ++work.t;
        ev = m_events<kWarp>(tm, mc, ev, at);
      } else {
        const uint32_t rows = PCCP_MSEC(off_t);
        int pass = 0;
        do {
          ev = 0u;
          for (int r = tm.tid; r < n_t; r += tm.nthr)
            m_temporal(st, lds64(rows + 8 * static_cast<uint32_t>(r)), ev);
          ++work.t;
          ev = m_events<kWarp>(tm, mc, ev, at);
        } while (ev == kEvTime && ++pass < max_iter);
        if (ev == kEvTime) return kError;
      }
      if (ev & kEvFail) return kFailed;
      ev = 0u;
    }
    const int n_wd = PCCP_MF(n_wd);
    const uint32_t wd = PCCP_MSEC(off_wd), wp = PCCP_MSEC(off_wp) + 8 * static_cast<uint32_t>(tm.lane);
    for (int i = tm.tid; i < (static_cast<int>(spare > dirty ? spare - dirty : dirty - spare) >> 2);
         i += tm.nthr)  // this round's rows mark it
      asm volatile("st.shared.u32 [%0], %1;" ::"r"(spare + 4 * i), "r"(0u) : "memory");
    if (full) {
      ++work.words;
      for (int w = 2 * tm.warp; w < n_wd; w += 2 * tm.nwarps) {
        const uint32_t p = wd + 16 * static_cast<uint32_t>(w);
        const uint4 D[2] = {lds128(p), lds128(p + 16)};
        const uint2 row[2] = {lds64(wp + D[0].w), lds64(wp + D[1].w)};
        m_words<2>(st, D, row, lane_bit, watch, ev);
      }
    } else {
      uint32_t evals = 0u;
      const uint32_t bit0 = static_cast<uint32_t>(PCCP_MF(bit0));
      for (int w = tm.warp; w < n_wd; w += tm.nwarps) {
        const uint4 D[1] = {lds128(wd + 16 * static_cast<uint32_t>(w))};
        const uint32_t q = (D[0].y >> 3) - bit0;
        if (!((lds32v(dirty + 4 * (q >> 5)) >> (q & 31u)) & 1)) continue;
        const uint2 row[1] = {lds64(wp + D[0].w)};
        m_words<1>(st, D, row, lane_bit, watch, ev);
        evals += __popc(D[0].x);
      }
      if (lane_bit == 1u && evals) atomicAdd(&mc->evals, evals);
    }
    ev = m_events<kWarp>(tm, mc, ev, at);
    if (ev & kEvFail) return kFailed;
    full = ev & kEvTime;
    const uint32_t swap = dirty;
    dirty = spare;
    spare = swap;
    ev &= kEvRaise;
    if (rows_first || ev) {
      rows_first = false;
      ++work.rows;
      ev = 0u;
      const int n_mr = PCCP_MF(n_mr), n_pq = PCCP_MF(n_pq);
      const uint32_t rows = PCCP_MSEC(off_mr), planes = PCCP_MSEC(off_mp);
      if (PCCP_MF(one_word)) {
        for (int r = tm.tid; r < n_mr; r += tm.nthr)
          m_row<true>(tb, planes, 1, st, lds128(rows + 16 * static_cast<uint32_t>(r)), watch, dirty, ev);
      } else {
        for (int r = tm.tid; r < n_mr; r += tm.nthr)
          m_row<false>(tb, planes, n_pq, st, lds128(rows + 16 * static_cast<uint32_t>(r)), watch, dirty,
                       ev);
      }
      ev = m_events<kWarp>(tm, mc, ev, at);
      if (ev & kEvFail) return kFailed;
    }
    if (!full && ev == 0u) break;
    if (work.rounds >= max_iter) return kError;
  }
  uint32_t ev = 0u;
  const int n_slots = PCCP_MF(n_slots), bit0 = PCCP_MF(bit0);
  for (int sl = tm.tid; sl < n_slots; sl += tm.nthr)
    if (slot_empty(ld_slot(st + 8 * static_cast<uint32_t>(sl)), sl, bit0)) ev = kEvFail;
  return m_events<kWarp>(tm, mc, ev, at) ? kFailed : kFixpoint;
}

// Rows evaluated and their algorithmic bytes (thread 0, after the fixed point).
__device__ __forceinline__ void m_work(const TableHeader* h, const MaskWork& w, const MaskCtrl* mc,
                                       long long& evals, long long& bytes) {
  const long long lin = h->bytes_sweep - 20ll * h->n_t - 40ll * h->n_rf;
  evals = static_cast<long long>(w.t) * h->n_t + static_cast<long long>(w.words) * h->n_rf + mc->evals +
          static_cast<long long>(w.rows) * h->n_mr;
  bytes = 20ll * w.t * h->n_t + 40ll * (static_cast<long long>(w.words) * h->n_rf + mc->evals) +
          w.rows * lin;
}

}  // namespace pccp
