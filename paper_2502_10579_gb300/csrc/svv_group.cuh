// svv_group.cuh -- the bound solves of several queries in one set of frontier
// rounds (a query-oblivious frontier over a group of same-type queries).
//
// Section 4.2 relaxes every snapshot of a window with one frontier that does
// not tell snapshots apart, and cites work that shares one frontier between
// queries; this is that idea applied to the bound solves of Section 3 Step 1:
// up to KL queries of one type, each with its own source and its own window,
// keep their values side by side in one row per vertex (val[v*KL + k] is lane
// k's value of v).  A vertex joins the frontier when any lane improved, and a
// frontier vertex relaxes its out-edges for every lane in which the edge is
// present, so each round reads each edge once and ends at one team barrier for
// all the queries of the group.  Each lane computes exactly what the solve of
// its own query computes (the fixed point is per lane and unique), so lanes
// never change one another's values.
//
// Edge presence per lane: an edge present in every one of the S snapshots is
// present in every lane's intersection and union graph; for the others a
// per-edge lane word is computed once per group (group_lanes_kernel): bits
// 0..15 = lanes whose whole window holds the edge (intersection graph), bits
// 16..31 = lanes whose window holds it at least once (union graph).
#pragma once

#include "svv_device.cuh"
#include "svv_pull.cuh"
#include "svv_push.cuh"
#include "svv_team.cuh"

namespace svv {

template <int KL>
__device__ __forceinline__ void st_row(uint32_t* p, const uint32_t (&r)[KL]) {
  if constexpr (KL == 2) {
    *reinterpret_cast<uint2*>(p) = make_uint2(r[0], r[1]);
  } else {
    uint4* q = reinterpret_cast<uint4*>(p);
#pragma unroll
    for (int i = 0; i < KL / 4; ++i) q[i] = make_uint4(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
  }
}

// lanes in which an edge takes part: every lane for an edge present in all S
// snapshots, else the intersection (PRED == kPredAll) or union half of its
// lane word
template <int PRED>
__device__ __forceinline__ uint32_t lanes_of(uint32_t word) {
  return PRED == kPredAll ? (word & 0xFFFFu) : (word >> 16);
}

// relax every lane of edge (u -> x, w) whose bit is set in `pm`, from the
// source row `su`, against the target row at `xr`; returns true if some lane
// of x was lowered (raised, for SSWP) by this edge, and keeps the best of the
// improved values in `key` (per lane, or one for all of them)
template <class Op, int KL, int NK>
__device__ __forceinline__ bool relax_lanes(const uint32_t (&su)[KL], uint32_t w, uint32_t pm, uint32_t* xr,
                                            uint32_t kinds, uint32_t (&key)[NK]) {
  uint32_t cur[KL];
  ld_row<KL>(xr, cur);
  bool imp = false;
#pragma unroll
  for (int k = 0; k < KL; ++k) {
    if ((pm >> k) & 1u) {
      const uint32_t cand = lane_relax<Op>(kinds, k, su[k], w);
      if (Op::better(cand, cur[k])) {
        Op::red(xr + k, cand);
        key[NK > 1 ? k : 0] = max(key[NK > 1 ? k : 0], nf_key<Op>(cand));
        imp = true;
      }
    }
  }
  return imp;
}

template <bool B>
struct Flag {
  static constexpr bool value = B;
};

template <class Op, int KL, int PRED>
__device__ bool group_solve_team(const GroupArgs& a, const Team& t, StageMem* stage) {
  const DevGraph& g = a.g;
  TeamCtl* c = a.ctl;
  const unsigned lane = threadIdx.x & 31u;
  const unsigned nthreads = t.nthreads();
  const unsigned gtid = t.tid();
  // neighbouring work goes to different SMs, so that a small round is spread
  // over all of them
  const unsigned gwarp = (threadIdx.x >> 5) * t.nblocks + t.rank, nwarps = nthreads >> 5;
  if (a.qerr && cta_read(a.qerr) != 0u) return false;
  PushStage st(stage, true);
  // The best improved value of every round goes to a ring as in the single
  // solve: one for the whole group (a bound for each of its lanes), or one per
  // lane for the two lanes of a mixed pair, whose values do not compare.
  constexpr int NK = is_mixed<Op>::value && KL == 2 ? 2 : 1;
  constexpr uint32_t kRing[2] = {0u, 8u};  // words of c->aux
  __shared__ uint32_t s_changed, s_key[NK];  // this CTA's improvements of a pull round; its best value
  if (threadIdx.x == 0) {
    s_changed = 0u;
    for (int k = 0; k < NK; ++k) s_key[k] = 0u;
  }
  uint32_t key[NK] = {};
  auto fold_keys = [&]() {  // a CTA barrier comes between this and publish_keys
#pragma unroll
    for (int k = 0; k < NK; ++k) {
      const uint32_t m = __reduce_max_sync(kFullMask, key[k]);
      if (lane == 0 && m) atomicMax(&s_key[k], m);
      key[k] = 0u;
    }
  };
  auto publish_keys = [&](uint32_t slot) {
    if (threadIdx.x == 0)
      for (int k = 0; k < NK; ++k)
        if (s_key[k]) {
          atomicMax(&c->aux[kRing[k] + slot], s_key[k]);
          s_key[k] = 0u;
        }
  };
  const uint32_t allmask = (1u << a.nlanes) - 1u;  // lanes in use (nlanes <= KL <= 8)

  // round 0: starting rows and stamps
  if (a.init == kInitSource) {
    uint32_t id[KL];
#pragma unroll
    for (int k = 0; k < KL; ++k) id[k] = Op::kIdentity;
    for (uint32_t v = gtid; v < g.V; v += nthreads) {
      st_row<KL>(a.val + (size_t)v * KL, id);
      a.stamp[v] = 0u;
    }
  } else {
    for (uint32_t v = gtid; v < g.V; v += nthreads) {
      uint32_t r[KL];
      ld_row<KL>(a.base + (size_t)v * KL, r);
      st_row<KL>(a.val + (size_t)v * KL, r);
      a.stamp[v] = 0u;
    }
  }
  if (!t.sync()) return false;
  if (a.trace && gtid == 0 && a.trace_cap) a.trace[0] = global_ns() & 0xFFFFFFFFFFull;

  // round 0: first frontier (stamp 1, queue q1, count qn[1])
  if (a.init == kInitSource) {
    if (gwarp == 0) {
      // every lane's source, queued once even when lanes share a source
      const bool mine = lane < a.nlanes;
      const uint32_t src = mine ? a.source[lane] : 0u;
      if (mine) a.val[(size_t)src * KL + lane] = Op::kSource;
#pragma unroll
      for (int k = 0; k < NK; ++k) key[k] = nf_key<Op>(Op::kSource);
      __syncwarp();
      bool push = false;
      uint32_t deg = 0;
      if (mine && atomicExch(a.stamp + src, 1u) != 1u) {
        push = true;
        deg = g.rp[src + 1] - g.rp[src];
      }
      stage_push_units(push, src, deg, a.cshift, st, a.q1, &c->qn[1], a.qcap, c, a.qerr, lane);
    }
  } else {
    // edges present in some but not all of a lane's window snapshots (that
    // lane's addition batches), from the intersection values of every lane
    for (uint32_t k0 = gwarp * 32u; k0 < g.NF; k0 += nwarps * 32u) {
      const uint32_t k = k0 + lane;
      bool push = false;
      uint32_t x = 0, deg = 0;
      if (k < g.NF) {
        const uint32_t lw = __ldg(a.nflanes + k);
        const uint32_t pm = (lw >> 16) & ~lw & allmask;  // any but not all
        if (pm) {
          const uint32_t u = __ldg(g.nfsrc + k);
          const uint2 e = __ldg(g.nfcw + k);
          x = e.x;
          uint32_t su[KL];
          ld_row<KL>(a.val + (size_t)u * KL, su);
          if (relax_lanes<Op, KL>(su, e.y, pm, a.val + (size_t)x * KL, a.kinds, key)) {
            const uint2 r = ld_row_span(g, x);
            push = atomicExch(a.stamp + x, 1u) != 1u;
            deg = r.y - r.x;
          }
        }
      }
      stage_push_units(push, x, deg, a.cshift, st, a.q1, &c->qn[1], a.qcap, c, a.qerr, lane);
    }
  }
  fold_keys();
  uint32_t queued = stage_flush_cta(st, a.q1, &c->qn[1], a.qcap, c, a.qerr, lane);
  publish_keys(1u);
  uint32_t n = 0;  // the round's frontier: units, or improved (target, item) pairs after a pull round
  bool dense = false;
  if (!t.sync(queued, n)) return false;

  unsigned long long relaxed = 0;
  uint32_t it = 1;
  for (;; ++it) {
    const uint32_t cur = it % 3u, nxt = (it + 1u) % 3u, clr = (it + 2u) % 3u;
    if (a.trace && gtid == 0 && it < a.trace_cap)
      a.trace[it] = ((unsigned long long)n << 40) | (global_ns() & 0xFFFFFFFFFFull);
    if (n == 0u) break;
    if (it > a.maxit) {
      if (gtid == 0) set_err(c, a.qerr, kErrTimeout);
      break;
    }
    n = min(n, a.qcap);
    // After a push round the frontier is a unit queue of n units; after a
    // pull round it is the vertices stamped with `it` (n counts as in the
    // single solve, once per pass).  A large frontier is pulled, a small one
    // pushed.
    const bool can_pull = g.pull != 0u && a.pull_units != 0u;
    const bool pull = can_pull && (dense ? (n > a.push_verts) : (n > a.pull_units));
    if (gtid == 0) {
      atomicExch(&c->qn[clr], 0u);
      atomicExch(&c->ticket[clr], 0u);
#pragma unroll
      for (int k = 0; k < NK; ++k) atomicExch(&c->aux[kRing[k] + clr], 0u);
      atomicExch(&c->aux[6 + ((it + 1u) & 1u)], 0u);  // compaction counter of the next round
    }
    unsigned long long* qin = (it & 1u) ? a.q1 : a.q0;
    unsigned long long* qout = (it & 1u) ? a.q0 : a.q1;
    unsigned* qn_out = &c->qn[nxt];
    const uint32_t stamp_next = it + 1u;

    if (pull) {
      // ---- pull round: one pass over every in-edge, a (CUDA) lane per target
      // and every value lane of the group in its registers
      const bool bottom_up = Op::kLevels && a.init == kInitSource;
      uint32_t best[2];
      cta_read2(&c->aux[kRing[0] + cur], &c->aux[kRing[NK - 1] + cur], best[0], best[1]);
#pragma unroll
      for (int k = 0; k < 2; ++k) best[k] = Op::better(0u, 1u) ? ~best[k] : best[k];
      // three or more lanes of several types have no common bound
      if (is_mixed<Op>::value && NK == 1) best[0] = Op::kSource;
      PullRound pr{a.val, a.stamp, stamp_next, it, allmask, a.kinds, bottom_up ? it - 1u : best[0], bottom_up};
      uint32_t changed = 0;
      auto pull_rows = [&](auto desc) {  // every value lane of pr.mask at once
        constexpr bool kDesc = decltype(desc)::value;
        changed += pull_items<Op, KL, KL, true, kDesc>(g.pf, pr, gwarp, nwarps, lane, relaxed, key[0],
                                                       [](size_t) { return ~0u; });
        changed += pull_items<Op, KL, KL, false, kDesc>(
            g.pp, pr, gwarp, nwarps, lane, relaxed, key[0],
            [&](size_t slot) { return lanes_of<PRED>(ld_stream(a.iplanes + slot)); });
      };
      if constexpr (is_mixed<Op>::value && KL == 2) {
        // two types: a pass per value lane, as in the single solve of its type
        for (uint32_t k = 0; k < a.nlanes; ++k) {
          pr.val = a.val + k;
          pr.mask = 1u;
          pr.best = best[k];
          uint32_t lkey = 0;
          auto pull_lane = [&](auto op, auto desc) {
            using LaneOp = decltype(op);
            constexpr bool kDesc = decltype(desc)::value;
            changed += pull_items<LaneOp, 1, 2, true, kDesc>(g.pf, pr, gwarp, nwarps, lane, relaxed, lkey,
                                                             [](size_t) { return 1u; });
            changed += pull_items<LaneOp, 1, 2, false, kDesc>(
                g.pp, pr, gwarp, nwarps, lane, relaxed, lkey,
                [&](size_t slot) { return (lanes_of<PRED>(ld_stream(a.iplanes + slot)) >> k) & 1u; });
          };
          switch ((a.kinds >> (2u * k)) & 3u) {
            case kKindSum: pull_lane(OpSSSP{}, Flag<false>{}); break;
            case kKindHop: pull_lane(OpBFS{}, Flag<false>{}); break;
            case kKindMax: pull_lane(OpSSNP{}, Flag<false>{}); break;
            default: pull_lane(OpSSWPNot{}, Flag<true>{}); break;
          }
          if (NK > 1) key[NK > 1 && k ? 1 : 0] = lkey;
        }
      } else if constexpr (is_mixed<Op>::value) {
        // widest-path lanes take the in-edges from the heaviest down, the
        // others from the lightest up
        uint32_t down = 0;
        for (uint32_t k = 0; k < a.nlanes; ++k)
          if (((a.kinds >> (2u * k)) & 3u) == kKindMaxNot) down |= 1u << k;
        pr.mask = allmask & ~down;
        if (pr.mask) pull_rows(Flag<false>{});
        pr.mask = allmask & down;
        if (pr.mask) pull_rows(Flag<true>{});
      } else {
        pull_rows(Flag<!Op::better(0u, 1u)>{});
      }
      fold_changes(changed, &s_changed, lane);
      fold_keys();
      __syncthreads();
      publish_keys(nxt);
      if (!t.sync(take_changes(&s_changed), n)) return false;
      dense = true;
      continue;
    }
    if (dense) {
      // ---- the last round pulled: queue the vertices it changed (stamp == it)
      unsigned* cnt_ctr = &c->aux[6 + (it & 1u)];
      for (uint32_t v0 = gwarp * 32u; v0 < g.V; v0 += nwarps * 32u) {
        const uint32_t v = v0 + lane;
        const bool take = v < g.V && ld_cg(a.stamp + v) == it;
        const uint32_t deg = take ? (__ldg(g.rp + v + 1) - __ldg(g.rp + v)) : 0u;
        stage_push_units(take, v, deg, a.cshift, st, qin, cnt_ctr, a.qcap, c, a.qerr, lane);
      }
      queued = stage_flush_cta(st, qin, cnt_ctr, a.qcap, c, a.qerr, lane);
      if (!t.sync(queued, n)) return false;
      n = min(n, a.qcap);
      dense = false;
    }

    // ---- push round: a warp takes up to 32 units, prefix-sums their edge
    // counts and walks the concatenated edges 32 at a time
    const bool levels = Op::kLevels && a.init == kInitSource;
    const Batches bt{n, batch_size(n, nwarps, 32u), nwarps, gwarp, &c->ticket[cur]};
    const uint32_t tk = bt.tk;
    for (uint32_t t0 = bt.first(); t0 < n; t0 = bt.next(lane)) {
      const uint32_t ui = t0 + lane;
      uint32_t beg = 0, cnt = 0, fe = 0, nfb = 0, vv = 0;
      if (lane < tk && ui < n) {
        const unsigned long long u = ld_cg(qin + ui);
        const uint32_t v = (uint32_t)u, ch = (uint32_t)(u >> 32);
        const uint4 rd = __ldg(g.rowd + v);
        const uint32_t r0 = rd.x, r1 = rd.y;
        fe = rd.z;
        nfb = rd.w;
        vv = v;
        beg = r0 + (ch << a.cshift);
        const uint32_t end = min(r1, beg + (1u << a.cshift));
        cnt = end > beg ? end - beg : 0u;
      }
      const uint32_t incl = warp_incl_scan(cnt, lane);
      const uint32_t total = __shfl_sync(kFullMask, incl, 31);
      if (lane == 0) relaxed += total;
      for (uint32_t p0 = 0; p0 < total; p0 += 32u) {
        const uint32_t p = p0 + lane;
        const int k = warp_owner(incl, p < total ? p : total - 1u);
        const uint32_t ik = __shfl_sync(kFullMask, incl, k);
        const uint32_t ck = __shfl_sync(kFullMask, cnt, k);
        const uint32_t bk = __shfl_sync(kFullMask, beg, k);
        const uint32_t fk = __shfl_sync(kFullMask, fe, k);
        const uint32_t nk = __shfl_sync(kFullMask, nfb, k);
        const uint32_t uk = __shfl_sync(kFullMask, vv, k);
        bool push = false;
        uint32_t x = 0, deg = 0;
        if (p < total) {
          const uint32_t e = bk + (p - (ik - ck));
          const uint2 ew = __ldg(g.cw + e);
          x = ew.x;
          uint32_t pm = e < fk ? allmask : (lanes_of<PRED>(__ldg(a.nflanes + nk + (e - fk))) & allmask);
          if (pm) {
            uint32_t su[KL];
            ld_row<KL>(a.val + (size_t)uk * KL, su);
            // BFS from the sources: a vertex can be in this round's frontier
            // for one lane while another lane's level of it is set in this
            // same round; pushing from that level would set the next level a
            // round early, and the pull rounds rely on round `it` setting
            // exactly level `it`.  So only levels set before this round push.
            if (levels) {
#pragma unroll
              for (int k = 0; k < KL; ++k)
                if (su[k] >= it) pm &= ~(1u << k);
            }
            if (pm && relax_lanes<Op, KL>(su, ew.y, pm, a.val + (size_t)x * KL, a.kinds, key)) {
              const uint2 r = ld_row_span(g, x);
              push = atomicExch(a.stamp + x, stamp_next) != stamp_next;
              deg = r.y - r.x;
            }
          }
        }
        stage_push_units(push, x, deg, a.cshift, st, qout, qn_out, a.qcap, c, a.qerr, lane);
      }
    }
    fold_keys();
    queued = stage_flush_cta(st, qout, qn_out, a.qcap, c, a.qerr, lane);
    publish_keys(nxt);
    if (!t.sync(queued, n)) return false;
  }
  if (lane == 0 && relaxed) atomicAdd(&c->relaxed, relaxed);
  if (gtid == 0) c->iters = it - 1u;
  return true;
}

}  // namespace svv
