// svv_pull.cuh -- one pull pass over the transposed graph (layout:
// svv_layout.cu), shared by the single solve (KL = 1) and the group solves
// (KL = 2, 4, 8 value lanes per vertex).
//
// A lane owns a target: it streams the target's in-edges, keeps the best
// candidate of every value lane in registers, and updates the target once per
// item.  Nothing is exchanged between lanes except for hubs (one fold per item
// of up to 512 edges), so an edge costs its 8-byte load, one gather of the
// source's row and the relaxation.
//
// A random gather takes one cache-line lookup per CUDA lane, and an SM's L1
// does about one lookup per clock: 16.1M gathers (scale 20) are 55 us on 152
// SMs however few instructions surround them, and that is what a round took
// with this layout before the in-edges were sorted by weight.  Sorted, most targets look
// at one weight and gather nothing: a round at scale 20 takes 20-26 us (SSSP
// and SSWP; 63-78 us with target-sorted edges folded by match.any and redux),
// a two-lane round of SSSP and SSWP 37-44 us (110-118).  What is left is the
// latency of an item (descriptor, targets, values) and the slowest warp.
#pragma once

#include "svv_device.cuh"

namespace svv {

// plain (L1-cacheable) load of a vertex's lane row; values only improve, so a
// stale row gives worse candidates (see ld_val)
template <int KL>
__device__ __forceinline__ void ld_row(const uint32_t* p, uint32_t (&r)[KL]) {
  if constexpr (KL == 1) {
    r[0] = ld_val(p);
  } else if constexpr (KL == 2) {
    const uint2 x = *reinterpret_cast<const uint2*>(p);
    r[0] = x.x;
    r[1] = x.y;
  } else {
    const uint4* q = reinterpret_cast<const uint4*>(p);
#pragma unroll
    for (int i = 0; i < KL / 4; ++i) {
      const uint4 x = q[i];
      r[4 * i] = x.x;
      r[4 * i + 1] = x.y;
      r[4 * i + 2] = x.z;
      r[4 * i + 3] = x.w;
    }
  }
}

// Ordering key of a value: larger = closer to the source, so one atomicMax
// per round finds the frontier's best value in both lattices.
template <class Op>
__device__ __forceinline__ uint32_t nf_key(uint32_t v) {
  return Op::better(0u, 1u) ? ~v : v;
}

struct PullRound {
  uint32_t* val;        // [V * KL]
  uint32_t* stamp;
  uint32_t stamp_next, it;
  uint32_t mask;        // value lanes of this pass
  uint32_t kinds;       // mixed groups: relaxation kind per lane
  uint32_t best;        // no source changed since it was last taken has a better value
  bool bottom_up;       // BFS from the source: see below
};

// One half of a pull round: every item of `P`, warps in turn.  `pres(slot)`
// gives the value lanes in which the edge of a slot is present (kAll: every
// edge is, and pres is not called).  Returns this lane's number of improved
// (target, item) pairs: zero over the grid exactly when nothing changed; `key`
// takes the best of the improved values (nf_key), lane 0's `edges` the slots
// read for targets that could still improve.  kStride: words per vertex (the KL
// lanes of the pass are the first ones of a row).
//
// A target's in-edges come in the order of their weights, the best first
// (ascending; kDesc: from the end, for widest paths).  The best that an edge
// of weight w can give is relax(r.best, w): an edge for which that is no
// improvement does not gather its source, and the first such edge ends the
// target, since all further ones give less.
// Bottom-up BFS: round `it` sets level `it` exactly when it only takes
// in-neighbours reached before it, and every improvement is `it` (r.best =
// it - 1), so a target is done when it has been reached.
template <class Op, int KL, int kStride, bool kAll, bool kDesc, class Pres>
__device__ __forceinline__ uint32_t pull_items(const PullGraph& P, const PullRound& r, uint32_t gwarp, uint32_t nwarps,
                                               unsigned lane, unsigned long long& edges, uint32_t& key, Pres pres) {
  constexpr int U = KL == 8 ? 2 : 4;  // edges in flight per lane
  uint32_t changed = 0, seen = 0;
  for (uint32_t i = gwarp; i < P.nitems; i += nwarps) {
    const uint2 d = ld_stream(P.items + (kDesc ? P.nitems - 1u - i : i));
    const uint32_t slice = d.y >> 4, steps = (d.y & 15u) + 1u;
    const uint32_t t = ld_stream(P.tgt + (size_t)slice * 32u + lane);
    const size_t slot0 = (size_t)d.x * 32u + lane;
    const bool own = t != kNone, hub = slice < P.nhub;
    uint32_t* xr = r.val + (size_t)(own ? t : 0u) * kStride;
    uint32_t tv[KL], acc[KL];
    ld_row<KL>(xr, tv);
#pragma unroll
    for (int k = 0; k < KL; ++k) {
      if (KL > 1 && !((r.mask >> k) & 1u)) tv[k] = Op::kSource;  // a lane that takes no part: nothing beats it
      acc[k] = tv[k];
    }
    // could an edge of weight w improve some value lane of the target?
    auto gains = [&](uint32_t w) {
      if constexpr (is_mixed<Op>::value) {
        bool any = false;
#pragma unroll
        for (int k = 0; k < KL; ++k) any |= Op::better(lane_relax<Op>(r.kinds, k, r.best, w), acc[k]);
        return any;
      } else {
        uint32_t worst = acc[0];
#pragma unroll
        for (int k = 1; k < KL; ++k) worst = Op::better(worst, acc[k]) ? acc[k] : worst;
        return Op::better(Op::relax(r.best, w), worst);
      }
    };
    bool live = own;
    if (Op::kLevels && r.bottom_up) {
      live = live && gains(0u);
      if (!__any_sync(kFullMask, live)) continue;
    }
    uint32_t s = 0;
    for (; s < steps; s += U) {
      uint2 sw[U];
      auto slot_of = [&](int j) { return slot0 + (size_t)(kDesc ? steps - 1u - (s + j) : s + j) * 32u; };
#pragma unroll
      for (int j = 0; j < U; ++j) {
        sw[j] = make_uint2(0u, 0u);
        if (live && s + j < steps) sw[j] = ld_stream(P.cw + slot_of(j));
      }
      live = live && gains(sw[0].y);
      const unsigned on = __ballot_sync(kFullMask, live);
      if (!on) break;
      seen += __popc(on) * min((uint32_t)U, steps - s);
      uint32_t pm[U];
#pragma unroll
      for (int j = 0; j < U; ++j) {
        pm[j] = 0u;
        if (live && s + j < steps && (j == 0 || gains(sw[j].y))) pm[j] = kAll ? r.mask : (pres(slot_of(j)) & r.mask);
      }
      uint32_t su[U][KL];
#pragma unroll
      for (int j = 0; j < U; ++j) {
#pragma unroll
        for (int k = 0; k < KL; ++k) su[j][k] = Op::kIdentity;
        if (pm[j]) ld_row<KL>(r.val + (size_t)sw[j].x * kStride, su[j]);
      }
#pragma unroll
      for (int j = 0; j < U; ++j) {
#pragma unroll
        for (int k = 0; k < KL; ++k) {
          bool on = (pm[j] >> k) & 1u;
          if (Op::kLevels) on = on && (!r.bottom_up || su[j][k] < r.it);
          const uint32_t cand = lane_relax<Op>(r.kinds, k, su[j][k], sw[j].y);
          if (on && Op::better(cand, acc[k])) acc[k] = cand;
        }
      }
      live = live && s + U < steps && gains(sw[U - 1].y);
      if (Op::kLevels && hub) live = __all_sync(kFullMask, live);
      if (!__any_sync(kFullMask, live)) break;
    }
    if (hub) {
#pragma unroll
      for (int k = 0; k < KL; ++k)
        acc[k] = Op::better(0u, 1u) ? __reduce_min_sync(kFullMask, acc[k]) : __reduce_max_sync(kFullMask, acc[k]);
    }
    if (own && (!hub || lane == 0)) {
      bool imp = false;
#pragma unroll
      for (int k = 0; k < KL; ++k) {
        if (Op::better(acc[k], tv[k])) {
          Op::red(xr + k, acc[k]);
          key = max(key, nf_key<Op>(acc[k]));
          imp = true;
        }
      }
      if (imp) {
        // a plain store: the next round finds the changed vertices from the
        // stamps, so the count only needs to be zero exactly when nothing changed
        r.stamp[t] = r.stamp_next;
        ++changed;
      }
    }
  }
  if (lane == 0) edges += seen;
  return changed;
}

}  // namespace svv
