// k_propagate_mask.cuh -- the batched propagation kernel for models in mask
// form (mask_device.cuh; included by pccp.cu).
//
// As k_propagate: persistent CTAs, the table image staged once per CTA by TMA
// bulk copies, teams of warps that take stores from a counter (the first one
// by team number, so a batch of at most one store per team needs no counter).
// A store in shared memory is the root's slots with the variables that
// differ from the root joined in: the caller's arrays are read four variables
// a load through a map in the caller's order, and most Booleans of a search
// node are still the root's, so a quad usually costs its loads and eight
// compares.  A store that fails is not written back (its contents are
// unspecified).
//
// What bounds it: instruction issue, and for batches of few stores the hardest
// store's chain of phases.  Kernel times against k_propagate on the same stores (one
// GB300): 10,000 of 30 tasks 169 -> 81 us.  Whole passes, with the caller's copy of
// the stores: 777 of 60 tasks 159 -> 88 us, 1,216 of 120 tasks 936 -> 306 us.
#pragma once

#include "mask_device.cuh"
#include "k_propagate.cuh"

namespace pccp {

// One Boolean of the caller's joined into the store: l, u its input bounds.
__device__ __forceinline__ void m_join(uint32_t st, int l, int u, uint32_t e, bool& empty) {
  const int rl = (e & kMapRootLb) ? 1 : 0, ru = (e & kMapRootUb) ? 1 : 0;
  if ((l <= rl && u >= ru) || (e & kMapInterval)) return;
  const uint32_t slot = st + (e & 0xffffu), m = 1u << ((e >> 16) & 31u);
  const int L = max(l, rl), U = min(u, ru);
  empty |= L > U;
  if (L > 0) red_or_at(slot, m);
  if (U < 1) red_and_at(slot + 4, ~m);
}

// Starts bringing bytes [p, p + bytes) into L2 (whole 16-byte units inside).
__device__ __forceinline__ void prefetch_l2(const void* p, size_t bytes) {
  const uintptr_t a = (reinterpret_cast<uintptr_t>(p) + 15u) & ~static_cast<uintptr_t>(15);
  const uintptr_t b = (reinterpret_cast<uintptr_t>(p) + bytes) & ~static_cast<uintptr_t>(15);
  if (b > a)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a),
                 "r"(static_cast<uint32_t>(b - a))
                 : "memory");
}

// One Boolean of the store (an interval's entry reads slot 0: its owner writes it after).
__device__ __forceinline__ int2 m_bit(uint32_t st, uint32_t e) {
  const int2 W = ld_slot(st + (e & 0xffffu));
  const int sh = static_cast<int>((e >> 16) & 31u);
  return make_int2((W.x >> sh) & 1, (W.y >> sh) & 1);
}

template <bool kWarp, int kMaxThreads, int kMinBlocks>
__global__ void __launch_bounds__(kMaxThreads, kMinBlocks) k_propagate_mask(PropArgs a) {
  extern __shared__ __align__(128) uint8_t smem[];
  // [table image][mbarrier 16 B] then per team [next store 16 B][MaskCtrl, bitmaps][store]
  uint64_t* mbar = reinterpret_cast<uint64_t*>(smem + a.image_bytes);
  const int team_id = static_cast<int>(threadIdx.x) / a.team_size;
  uint8_t* slot = smem + a.image_bytes + 16 + static_cast<size_t>(a.slot_bytes) * team_id;
  int* next_store = reinterpret_cast<int*>(slot);
  MaskCtrl* mc = reinterpret_cast<MaskCtrl*>(slot + 16);
  int2* st = reinterpret_cast<int2*>(slot + 16 + 4 * a.track_words);
  if (threadIdx.x == 0) mbar_init(mbar, 1);
  const bool ok = load_image(smem, a.image, a.image_bytes, mbar, 0);
  Team tm;
  tm.tid = static_cast<int>(threadIdx.x) - team_id * a.team_size;
  tm.nthr = a.team_size;
  tm.bar = (1 + team_id) & 15;  // a 16th team takes barrier 0, free after the image is in
  tm.lane = static_cast<int>(threadIdx.x & 31u);
  tm.warp = tm.tid >> 5;
  tm.nwarps = a.team_size >> 5;
  const int nv = a.n_vars;
  const int n_teams = static_cast<int>(gridDim.x) * a.teams;
  int s = static_cast<int>(blockIdx.x) + team_id * static_cast<int>(gridDim.x);
  if (!ok) {  // the image never arrived: nothing of it is read, the stores are reported
    for (; tm.tid == 0 && s < a.n_stores; s = a.counter ? n_teams + atomicAdd(a.counter, 1) : a.n_stores) {
      a.status[s] = kError;
      if (a.iters) a.iters[s] = 0;
      if (a.work) {
        a.work[2 * static_cast<size_t>(s)] = 0;
        a.work[2 * static_cast<size_t>(s) + 1] = 0;
      }
    }
    return;
  }
  const MTab tb = make_mtab(smem, a.levels & 1);
  const uint32_t sb = smem_u32(st);
  const TableHeader* h = reinterpret_cast<const TableHeader*>(smem);
  // events, counts, and the watch masks, of which those of words without a
  // reified row are never written; published by the first store's barrier
  for (int i = tm.tid; i < a.track_words; i += tm.nthr) reinterpret_cast<uint32_t*>(mc)[i] = 0u;
  int at = 0;
  while (s < a.n_stores) {
    int32_t* lbs = a.lb + static_cast<size_t>(s) * nv;
    int32_t* ubs = a.ub + static_cast<size_t>(s) * nv;
    // the team's next store
    int next = a.n_stores;
    if (a.counter && tm.tid == 0) next = n_teams + atomicAdd(a.counter, 1);
    // quads of variables at 16-byte addresses of both arrays, from `head` on
    const int head = static_cast<int>((16u - (reinterpret_cast<uintptr_t>(lbs) & 15u)) & 15u) >> 2;
    const bool quads = ((reinterpret_cast<uintptr_t>(lbs) ^ reinterpret_cast<uintptr_t>(ubs)) & 15u) == 0u;
    const uint32_t* map = a.map + head * a.map_stride + ((4 - head) & 3);
    const int nq = quads && nv > head ? (nv - head) >> 2 : 0;
    // the root's slots, the intervals joined with the input (a thread each)
    bool empty = false;
    const int32_t* user_of = reinterpret_cast<const int32_t*>(a.root + nv) + nv;
    const int2* rs = reinterpret_cast<const int2*>(smem + h->off_rs);
    const int n_slots = h->n_slots, bit0 = h->bit0;
    for (int sl = tm.tid; sl < n_slots; sl += tm.nthr) {
      int2 r = rs[sl];
      if (sl < bit0) {
        const int x = __ldg(user_of + sl);
        r = make_int2(max(lbs[x], r.x), min(ubs[x], r.y));
        empty |= r.x > r.y;
      }
      st[sl] = r;
    }
    mbar_team<kWarp>(tm);
    int status = kFailed;
    MaskWork work{0, 0, 0, 0};
    // a quad whose lower bounds are at most the root's and whose upper
    // bounds are at least 1 leaves the root's bits (nothing is read from the map)
    const uint32_t rl = smem_u32(smem) + static_cast<uint32_t>(h->off_rl + 4 * head * h->rl_words);
#pragma unroll 4
    for (int q = tm.tid; q < nq; q += tm.nthr) {
      const int x = head + 4 * q;
      const int4 l = __ldcs(reinterpret_cast<const int4*>(lbs + x));
      const int4 u = __ldcs(reinterpret_cast<const int4*>(ubs + x));
      const int r = lds32(rl + 4 * (q >> 3)) >> (4 * (q & 7));
      const bool over = (l.x > (r & 1)) | (l.y > ((r >> 1) & 1)) | (l.z > ((r >> 2) & 1)) |
                        (l.w > ((r >> 3) & 1));
      if (over | (min(min(u.x, u.y), min(u.z, u.w)) < 1)) {
        const uint4 e = __ldg(reinterpret_cast<const uint4*>(map + x));
        m_join(sb, l.x, u.x, e.x, empty);
        m_join(sb, l.y, u.y, e.y, empty);
        m_join(sb, l.z, u.z, e.z, empty);
        m_join(sb, l.w, u.w, e.w, empty);
      }
    }
    for (int k = tm.tid; k < nv - 4 * nq; k += tm.nthr) {  // before and after the quads
      const int x = nq == 0 || k < head ? k : k + 4 * nq;
      m_join(sb, lbs[x], ubs[x], __ldg(map + x), empty);
    }
    if (tm.tid == 0 && next < a.n_stores) {
      prefetch_l2(a.lb + static_cast<size_t>(next) * nv, 4 * static_cast<size_t>(nv));
      prefetch_l2(a.ub + static_cast<size_t>(next) * nv, 4 * static_cast<size_t>(nv));
    }
    if (!mbar_team_or<kWarp>(tm, empty))
      status = m_fixpoint<kWarp>(tb, st, tm, mc, true, a.max_iter, at, work);
    if (status != kFailed) {
#pragma unroll 2
      for (int q = tm.tid; q < nq; q += tm.nthr) {
        const int x = head + 4 * q;
        const uint4 e = __ldg(reinterpret_cast<const uint4*>(map + x));
        const int2 v0 = m_bit(sb, e.x), v1 = m_bit(sb, e.y), v2 = m_bit(sb, e.z),
                   v3 = m_bit(sb, e.w);
        *reinterpret_cast<int4*>(lbs + x) = make_int4(v0.x, v1.x, v2.x, v3.x);
        *reinterpret_cast<int4*>(ubs + x) = make_int4(v0.y, v1.y, v2.y, v3.y);
      }
      for (int k = tm.tid; k < nv - 4 * nq; k += tm.nthr) {
        const int x = nq == 0 || k < head ? k : k + 4 * nq;
        const int2 v = m_bit(sb, __ldg(map + x));
        lbs[x] = v.x;
        ubs[x] = v.y;
      }
      mbar_team<kWarp>(tm);  // the intervals, over what the quads put there
      for (int v = tm.tid; v < bit0; v += tm.nthr) {
        const int x = __ldg(user_of + v);
        const int2 D = st[v];
        lbs[x] = D.x;
        ubs[x] = D.y;
      }
    }
    if (tm.tid == 0) {
      a.status[s] = status;
      if (a.iters) a.iters[s] = work.rounds;
      if (a.work) {
        long long ev, by;
        m_work(h, work, mc, ev, by);
        a.work[2 * static_cast<size_t>(s)] = ev > 0x7fffffffll ? 0x7fffffff : static_cast<int>(ev);
        a.work[2 * static_cast<size_t>(s) + 1] =
            by > 0x7fffffffll ? 0x7fffffff : static_cast<int>(by);
      }
      mc->evals = 0u;
      *next_store = next;
    }
    mbar_team<kWarp>(tm);  // every warp is done with the store
    s = *next_store;
  }
}

}  // namespace pccp
