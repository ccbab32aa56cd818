// svv_solve.cuh -- the single-value frontier solve as a team phase.
#pragma once

#include "svv_device.cuh"
#include "svv_pull.cuh"
#include "svv_push.cuh"
#include "svv_team.cuh"

namespace svv {

template <class Op, int PRED>
__device__ bool solve_team(const SolveArgs& a, const Team& t, StageMem* stage) {
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
  __shared__ uint32_t s_changed, s_key;  // this CTA's improvements of a round, and the best of them
  if (threadIdx.x == 0) s_changed = s_key = 0u;

  // round 0: starting values and stamps
  if (a.init == kInitSource) {
    for (uint32_t v = gtid; v < g.V; v += nthreads) {
      a.val[v] = Op::kIdentity;
      a.stamp[v] = 0u;
    }
  } else {
    for (uint32_t v = gtid; v < g.V; v += nthreads) {
      a.val[v] = a.base[v];
      a.stamp[v] = 0u;
    }
  }
  // no chunk has been relaxed yet: the identity is never a queued value
  if (a.procv)
    for (uint32_t k = gtid; k < a.pcap; k += nthreads) a.procv[k] = Op::kIdentity;
  if (a.skip_arrival && t.rank + 1u == a.skip_arrival) return false;  // test hook: never arrives
  if (!t.sync()) return false;
  if (a.trace && gtid == 0 && a.trace_cap) a.trace[0] = global_ns() & 0xFFFFFFFFFFull;

  // the best value of each round's frontier goes to aux[0..2], a ring: every
  // improvement of the round before counts, also those another lane beat
  uint32_t key = 0;
  auto fold_key = [&]() {  // a CTA barrier comes between this and publish_key
    const uint32_t m = __reduce_max_sync(kFullMask, key);
    if (lane == 0 && m) atomicMax(&s_key, m);
    key = 0;
  };
  auto publish_key = [&](unsigned* slot) {
    if (threadIdx.x == 0 && s_key) {
      atomicMax(slot, s_key);
      s_key = 0u;
    }
  };

  // round 0: first frontier (stamp 1, queue q1, count qn[1])
  if (a.init == kInitSource) {
    if (gwarp == 0) {
      uint32_t deg = 0;
      if (lane == 0) {
        a.val[a.source] = Op::kSource;
        a.stamp[a.source] = 1u;
        deg = g.rp[a.source + 1] - g.rp[a.source];
      }
      stage_push_units(lane == 0, a.source, deg, a.cshift, st, a.q1, &c->qn[1], a.qcap, c, a.qerr, lane);
      if (lane == 0) atomicMax(&c->aux[1], nf_key<Op>(Op::kSource));
    }
  } else {
    // edges present in some but not all window snapshots (the window's
    // addition batches); intersection edges cannot improve a fixed point of
    // the intersection graph, so they are skipped
    for (uint32_t k0 = gwarp * 32u; k0 < g.NF; k0 += nwarps * 32u) {
      const uint32_t k = k0 + lane;
      bool push = false;
      uint32_t x = 0, deg = 0;
      if (k < g.NF) {
        bool any, all;
        window_any_all(g.nfmask + (size_t)k * g.W, a.win, any, all);
        if (any && !all) {
          const uint32_t u = __ldg(g.nfsrc + k);
          const uint2 e = __ldg(g.nfcw + k);
          x = e.x;
          const uint32_t cand = Op::relax(ld_val(a.val + u), e.y);
          if (Op::better(cand, ld_val(a.val + x))) {
            Op::red(a.val + x, cand);
            key = max(key, nf_key<Op>(cand));
            const uint2 r = ld_row_span(g, x);
            if (atomicExch(a.stamp + x, 1u) != 1u) {
              push = true;
              deg = r.y - r.x;
            }
          }
        }
      }
      stage_push_units(push, x, deg, a.cshift, st, a.q1, &c->qn[1], a.qcap, c, a.qerr, lane);
    }
  }
  fold_key();
  uint32_t queued = stage_flush_cta(st, a.q1, &c->qn[1], a.qcap, c, a.qerr, lane);
  publish_key(&c->aux[1]);
  uint32_t n = 0;  // the round's frontier: units, or improved (target, item) pairs after a pull round
  bool dense = false;
  if (!t.sync(queued, n)) return false;

  unsigned long long relaxed = 0;
  uint32_t it = 1;
  for (;; ++it) {
    const uint32_t cur = it % 3u, nxt = (it + 1u) % 3u, clr = (it + 2u) % 3u;
    const bool far_on = a.delta != 0u;
    if (a.trace && gtid == 0 && it < a.trace_cap) a.trace[it] = ((unsigned long long)n << 40) | (global_ns() & 0xFFFFFFFFFFull);
    if (n == 0u) break;
    if (it > a.maxit) {
      if (gtid == 0) set_err(c, a.qerr, kErrTimeout);
      break;
    }
    n = min(n, a.qcap);
    // How this round runs.  After a push round the frontier is a unit queue of
    // n units; after a pull round it is the vertices stamped with `it`, and n
    // counts a vertex once, a hub once per item that improved it (so hubs keep
    // pulling a little longer).  A large frontier is pulled: every vertex takes
    // the best candidate over its in-edges (no queue, one reduction per target
    // and item); a small one is pushed.
    const bool can_pull = g.pull != 0u && a.pull_units != 0u;
    const bool pull = can_pull && (dense ? (n > a.push_verts) : (n > a.pull_units));
    if (gtid == 0) {
      atomicExch(&c->qn[clr], 0u);
      atomicExch(&c->ticket[clr], 0u);
      atomicExch(&c->aux[clr], 0u);
      atomicExch(&c->aux[6 + ((it + 1u) & 1u)], 0u);  // compaction counter of the next round
    }
    unsigned long long* qin = (it & 1u) ? a.q1 : a.q0;
    unsigned long long* qout = (it & 1u) ? a.q0 : a.q1;
    unsigned* qn_out = &c->qn[nxt];
    const uint32_t stamp_next = it + 1u;

    if (pull) {
      // ---- pull round: one pass over every in-edge, a lane per target
      const bool bottom_up = Op::kLevels && a.init == kInitSource;
      const uint32_t slot = cta_read(&c->aux[cur]);
      constexpr bool kDesc = !Op::better(0u, 1u);
      const PullRound pr{a.val, a.stamp, stamp_next, it, 1u, 0u,
                         bottom_up ? it - 1u : (kDesc ? slot : ~slot), bottom_up};
      uint32_t changed =
          pull_items<Op, 1, 1, true, kDesc>(g.pf, pr, gwarp, nwarps, lane, relaxed, key, [](size_t) { return 1u; });
      if (!(PRED == kPredAll && a.skip_nf))
        changed += pull_items<Op, 1, 1, false, kDesc>(g.pp, pr, gwarp, nwarps, lane, relaxed, key,
                                                   [&](size_t slot) -> uint32_t {
                                                     const uint64_t* m = g.ppmask + slot * g.W;
                                                     if (PRED == kPredAll) return window_all(m, a.win);
                                                     if (PRED == kPredAny) return window_any(m, a.win);
                                                     return mask_bit(m, a.bit);
                                                   });
      fold_changes(changed, &s_changed, lane);
      fold_key();
      __syncthreads();
      publish_key(&c->aux[nxt]);
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
    // near-far: relax only units whose value is within delta of the best
    // value queued for this round (that unit itself always qualifies, so every
    // round makes progress); the others are queued again unchanged
    uint32_t bound = 0;
    if (far_on) {
      const uint32_t slot = cta_read(&c->aux[cur]);
      if (Op::better(0u, 1u)) {
        const uint32_t best = ~slot;
        bound = best > kInf - a.delta ? kInf : best + a.delta;
      } else {
        bound = slot > a.delta ? slot - a.delta : 0u;
      }
    }

    // units per ticket: spread a small frontier over every warp, batch a
    // large one 32 units at a time
    const Batches bt{n, batch_size(n, nwarps, 32u), nwarps, gwarp, &c->ticket[cur]};
    const uint32_t tk = bt.tk;
    for (uint32_t t0 = bt.first(); t0 < n; t0 = bt.next(lane)) {
      const uint32_t ui = t0 + lane;
      uint32_t beg = 0, cnt = 0, fe = 0, nfb = 0, sv = Op::kIdentity;
      bool defer = false;
      uint32_t dv = 0, ddeg = 0;
      if (lane < tk && ui < n) {
        const unsigned long long u = ld_cg(qin + ui);
        const uint32_t v = (uint32_t)u, ch = (uint32_t)(u >> 32);
        const uint4 rd = __ldg(g.rowd + v);
        const uint32_t r0 = rd.x, r1 = rd.y;
        fe = rd.z;
        nfb = rd.w;
        beg = r0 + (ch << a.cshift);
        uint32_t end = min(r1, beg + (1u << a.cshift));
        if (PRED == kPredAll && a.skip_nf) end = min(end, fe);
        cnt = end > beg ? end - beg : 0u;
        sv = ld_cg(a.val + v);
        if (far_on && (Op::better(0u, 1u) ? sv > bound : sv < bound)) {
          // far: queue all of v's units again, once per round (stamp), and
          // skip this one now
          cnt = 0;
          if (atomicExch(a.stamp + v, stamp_next) != stamp_next) {
            defer = true;
            dv = v;
            ddeg = r1 - r0;
          }
        }
        if (a.procv && cnt) {
          // chunk ids v + rp[v]/C + ch are distinct across vertices; a
          // deferred chunk is not relaxed now, so it records nothing
          uint32_t* pv = a.procv + v + (r0 >> a.cshift) + ch;
          if (ld_cg(pv) == sv) cnt = 0;
          else *pv = sv;
        }
      }
      if (far_on) {
        stage_push_units(defer, dv, ddeg, a.cshift, st, qout, qn_out, a.qcap, c, a.qerr, lane);
        if (defer) key = max(key, nf_key<Op>(sv));
      }
      const uint32_t incl = warp_incl_scan(cnt, lane);
      const uint32_t total = __shfl_sync(kFullMask, incl, 31);
      if (lane == 0) relaxed += total;
      // two 32-edge steps in flight per iteration: their loads, checks and
      // atomics are independent, so each lane keeps two chains going
      for (uint32_t p0 = 0; p0 < total; p0 += 64u) {
        bool push[2];
        uint32_t x[2], deg[2];
        uint32_t sk[2], ew_w[2];
        bool act[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const uint32_t p = p0 + 32u * j + lane;
          const int k = warp_owner(incl, p < total ? p : total - 1u);
          const uint32_t ik = __shfl_sync(kFullMask, incl, k);
          const uint32_t ck = __shfl_sync(kFullMask, cnt, k);
          const uint32_t bk = __shfl_sync(kFullMask, beg, k);
          const uint32_t fk = __shfl_sync(kFullMask, fe, k);
          const uint32_t nk = __shfl_sync(kFullMask, nfb, k);
          sk[j] = __shfl_sync(kFullMask, sv, k);
          push[j] = false;
          x[j] = 0;
          deg[j] = 0;
          act[j] = false;
          ew_w[j] = 0;
          if (p < total) {
            const uint32_t e = bk + (p - (ik - ck));
            const uint2 ew = __ldg(g.cw + e);
            x[j] = ew.x;
            ew_w[j] = ew.y;
            bool present = true;
            if (e >= fk) {
              const uint64_t* m = g.nfmask + (size_t)(nk + (e - fk)) * g.W;
              if (PRED == kPredAll) present = window_all(m, a.win);
              else if (PRED == kPredAny) present = window_any(m, a.win);
              else present = mask_bit(m, a.bit);
            }
            act[j] = present;
          }
        }
        uint32_t cand[2], curv[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          cand[j] = Op::relax(sk[j], ew_w[j]);
          curv[j] = act[j] ? ld_val(a.val + x[j]) : cand[j];
        }
        bool imp[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          imp[j] = act[j] && Op::better(cand[j], curv[j]);
          if (imp[j]) {
            Op::red(a.val + x[j], cand[j]);
            key = max(key, nf_key<Op>(cand[j]));
          }
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          if (imp[j]) {
            const uint2 r = ld_row_span(g, x[j]);
            if (atomicExch(a.stamp + x[j], stamp_next) != stamp_next) {
              push[j] = true;
              deg[j] = r.y - r.x;
            }
          }
        }
        stage_push_units(push[0], x[0], deg[0], a.cshift, st, qout, qn_out, a.qcap, c, a.qerr, lane);
        stage_push_units(push[1], x[1], deg[1], a.cshift, st, qout, qn_out, a.qcap, c, a.qerr, lane);
      }
    }
    fold_key();
    queued = stage_flush_cta(st, qout, qn_out, a.qcap, c, a.qerr, lane);
    publish_key(&c->aux[nxt]);
    if (!t.sync(queued, n)) return false;
  }
  if (lane == 0 && relaxed) atomicAdd(&c->relaxed, relaxed);
  if (gtid == 0) c->iters = it - 1u;
  return true;
}

}  // namespace svv
