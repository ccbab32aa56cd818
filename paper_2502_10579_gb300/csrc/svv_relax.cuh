// svv_relax.cuh -- Algorithm 2 (concurrent relaxation of every window
// snapshot) and the output scatter as team phases (see svv_relax.cu).
#pragma once

#include "svv_device.cuh"
#include "svv_pull.cuh"
#include "svv_push.cuh"
#include "svv_team.cuh"

namespace svv {

// a value that improved a row: into the CTA's best of its snapshot
template <class Op>
__device__ __forceinline__ void note_best(uint32_t* s, uint32_t v) {
  const uint32_t k = nf_key<Op>(v);
  if (k > *reinterpret_cast<volatile uint32_t*>(s)) atomicMax(s, k);
}

// query q's relaxation: the op's own, or (a mixed pair) query q's kind
template <class Op>
__device__ __forceinline__ uint32_t relax_q(const RelaxArgs& a, bool q1, uint32_t sv, uint32_t w) {
  if constexpr (is_mixed<Op>::value) return OpMixed::relax_kind(q1 ? a.kind1 : a.kind0, sv, w);
  else return Op::relax(sv, w);
}

// ---------------------------------------------------------------------------
// Pull rounds.  When a large part of the rows is in the frontier, a round goes
// over the in-edges of the unstable vertices instead (the transposed graph of
// the solves, svv_layout.cu), sorted by weight: a warp keeps a target's row in
// registers (a lane per snapshot, K of them), takes the rows of its in-edges'
// sources that are in the frontier, best weight first, and stops at the first
// weight that can improve no snapshot any more.  The best value that the round
// before gave any row in snapshot i (RelaxArgs::best) bounds what an edge of
// weight w can give there: relax(best[i], w); it is what lets a target stop
// whose value in some snapshot stays unreachable.  A push round instead loads
// (and partly lowers) a target's row for every edge of the frontier.
// At scale 20 with 533K unstable vertices and 16M subgraph edges (136 MB of
// rows) push rounds took 270-775 us each.

// the edges of one item: 32 lanes hold the steps of 32 / sp targets at a time;
// `edges` counts those whose source's row was read
template <class Op, int K, bool kPart>
__device__ __forceinline__ uint32_t relax_pull_items(const PullGraph& P, const RelaxArgs& a, bool q1, uint32_t it,
                                                     const uint32_t (&best)[K], uint32_t* s_best, unsigned gwarp,
                                                     unsigned nwarps, unsigned lane, uint32_t& edges) {
  const uint32_t lps = __ffs(a.LP) - 1;
  const uint32_t* rowmap = q1 ? a.row1 : a.row;
  const uint32_t snap = (q1 ? a.win1.b : a.win.b) + a.s0;
  bool desc = !Op::better(0u, 1u);
  if constexpr (is_mixed<Op>::value) desc = (q1 ? a.kind1 : a.kind0) == kKindMaxNot;
  const uint64_t slab0 = a.ls >= 64u ? ~0ull : (1ull << a.ls) - 1ull;
  const uint64_t slab1 = a.ls >= 128u ? ~0ull : a.ls > 64u ? (1ull << (a.ls - 64u)) - 1ull : 0ull;
  constexpr int H = K <= 2 ? 4 : 2;  // source rows in flight
  uint32_t changed = 0;
  for (uint32_t i = gwarp; i < P.nitems; i += nwarps) {
    const uint2 d = ld_stream(P.items + (desc ? P.nitems - 1u - i : i));
    const uint32_t steps = (d.y & 15u) + 1u;
    const uint32_t t = ld_stream(P.tgt + (size_t)(d.y >> 4) * 32u + lane);
    const uint32_t rt = t != kNone ? rowmap[t] : kNone;
    if (!__any_sync(kFullMask, rt != kNone)) continue;
    const uint32_t sps = 32u - __clz(steps - 1u), sp = 1u << sps;  // steps <= sp <= 16
    for (uint32_t p = 0; p < sp; ++p) {
      const uint32_t tl = (p << (5u - sps)) + (lane >> sps), k = lane & (sp - 1u);
      const uint32_t rl = __shfl_sync(kFullMask, rt, tl);
      if (!__any_sync(kFullMask, rl != kNone)) continue;
      const size_t slot = ((size_t)d.x + (desc ? steps - 1u - k : k)) * 32u + tl;
      uint32_t ru = kNone, w = 0;
      uint64_t m0 = slab0, m1 = slab1;
      if (rl != kNone && k < steps) {
        const uint2 e = __ldg(P.cw + slot);
        w = e.y;
        ru = rowmap[e.x];
        if (ru != kNone && ld_cg(a.stamp + ru) < it) ru = kNone;  // not in the frontier (it + 1: changed meanwhile)
        if (kPart && ru != kNone) {
          const uint64_t* m = a.g.ppmask + slot * a.g.W;
          m0 = mask_extract(m, a.g.W, snap) & slab0;
          m1 = K > 2 ? mask_extract(m, a.g.W, snap + 64u) & slab1 : 0ull;
          if (!(m0 | m1)) ru = kNone;
        }
      }
      const unsigned on = __ballot_sync(kFullMask, ru != kNone);
      for (unsigned left = on; left;) {
        const unsigned first = __ffs(left) - 1u;
        const unsigned grp = (sp == 32u ? kFullMask : ((1u << sp) - 1u)) << (first & ~(sp - 1u));
        unsigned todo = left & grp;  // this target's edges, the best weight first
        left &= ~grp;
        const uint32_t r = __shfl_sync(kFullMask, rl, first);
        uint32_t* xr = a.val + ((size_t)r << lps) + lane;
        uint32_t tv[K], cur[K];
#pragma unroll
        for (int kk = 0; kk < K; ++kk) tv[kk] = cur[kk] = ld_val(xr + kk * 32);
        while (todo) {
          const uint32_t w0 = __shfl_sync(kFullMask, w, __ffs(todo) - 1);
          bool gain = false;
#pragma unroll
          for (int kk = 0; kk < K; ++kk) gain |= Op::better(relax_q<Op>(a, q1, best[kk], w0), cur[kk]);
          if (!__any_sync(kFullMask, gain)) break;
          edges += min((uint32_t)__popc(todo), (uint32_t)H);
          uint32_t su[H][K], ew[H];
          uint64_t e0[H], e1[H];
          bool ev[H];
#pragma unroll
          for (int h = 0; h < H; ++h) {
            ev[h] = todo != 0u;
            const int src = todo ? __ffs(todo) - 1 : 0;
            todo &= todo - 1u;
            const uint32_t rs = __shfl_sync(kFullMask, ru, src);
            ew[h] = __shfl_sync(kFullMask, w, src);
            e0[h] = slab0;
            e1[h] = slab1;
            if (kPart) {
              e0[h] = __shfl_sync(kFullMask, m0, src);
              if (K > 2) e1[h] = __shfl_sync(kFullMask, m1, src);
            }
            const uint32_t* sr = a.val + ((size_t)rs << lps) + lane;
#pragma unroll
            for (int kk = 0; kk < K; ++kk) su[h][kk] = ev[h] ? ld_val(sr + kk * 32) : Op::kIdentity;
          }
#pragma unroll
          for (int h = 0; h < H; ++h) {
#pragma unroll
            for (int kk = 0; kk < K; ++kk) {
              const uint32_t i2 = lane + 32u * kk;
              const bool bit = kk < 2 ? (e0[h] >> i2) & 1ull : (e1[h] >> (i2 - 64u)) & 1ull;
              const uint32_t cand = relax_q<Op>(a, q1, su[h][kk], ew[h]);
              if (ev[h] && bit && Op::better(cand, cur[kk])) cur[kk] = cand;
            }
          }
        }
        bool imp = false;
#pragma unroll
        for (int kk = 0; kk < K; ++kk) {
          if (Op::better(cur[kk], tv[kk])) {
            Op::red(xr + kk * 32, cur[kk]);
            note_best<Op>(s_best + lane + 32 * kk, cur[kk]);
            imp = true;
          }
        }
        if (__any_sync(kFullMask, imp) && lane == 0) {
          a.stamp[r] = it + 1u;
          ++changed;
        }
      }
    }
  }
  return changed;
}

// A whole pull round of both queries; returns this lane's improved (row, item)
// pairs.  Out of line, so that the push rounds' loop keeps its registers.
template <class Op, int K>
__device__ __noinline__ uint32_t relax_pull_round(const RelaxArgs& a, uint32_t it, StageMem* stage, unsigned gwarp,
                                                  unsigned nwarps) {
  const unsigned lane = threadIdx.x & 31u;
  uint32_t changed = 0, edges = 0;
  for (int qi = 0; qi < (a.counts1 ? 2 : 1); ++qi) {
    uint32_t best[K];
#pragma unroll
    for (int kk = 0; kk < K; ++kk) {
      const uint32_t key = ld_cg(a.best + ((it % 3u) * 2u + qi) * kBestSnaps + lane + 32u * kk);
      best[kk] = Op::better(0u, 1u) ? ~key : key;
    }
    changed += relax_pull_items<Op, K, false>(a.g.pf, a, qi != 0, it, best, stage->best[qi], gwarp, nwarps, lane,
                                              edges);
    changed += relax_pull_items<Op, K, true>(a.g.pp, a, qi != 0, it, best, stage->best[qi], gwarp, nwarps, lane,
                                             edges);
  }
  if (lane == 0 && edges) atomicAdd(&a.ctl->relaxed, (unsigned long long)edges);
  return changed;
}

// One push round (Algorithm 2 over the frontier's units) and its flush.  Out of
// line, so that the loop has the registers to itself (64; rows of 32 to 128
// values store 16 to 96 bytes of them on the stack all the same); kNote: also keep the best
// improved value of every snapshot, for the bound of a pull round that follows.
struct RelaxRound {
  uint32_t n, it, U0, gwarp, nwarps;
  const unsigned long long* qin;
  unsigned long long* qout;
};
struct RelaxDone {
  uint32_t queued, edges;  // units the CTA queued (thread 0); edges this lane counts
};

template <class Op, int P, int K, bool kNote>
__device__ __noinline__ RelaxDone relax_push_round(const RelaxArgs& a, const RelaxRound rr, StageMem* stage) {
  TeamCtl* c = a.ctl;
  const unsigned lane = threadIdx.x & 31u;
  const uint32_t n = rr.n, U0 = rr.U0, nwarps = rr.nwarps, gwarp = rr.gwarp, stamp_next = rr.it + 1u;
  const uint32_t cur = rr.it % 3u;
  const uint32_t lps = __ffs(a.LP) - 1;
  const unsigned long long* qin = rr.qin;
  unsigned long long* qout = rr.qout;
  unsigned* qn_out = &c->qn[stamp_next % 3u];
  constexpr int G = 32 / P;
  const unsigned grp = lane / P, gl = lane % P;
  const unsigned gmask = (P == 32) ? kFullMask : (((1u << P) - 1u) << (grp * P));
  RelaxDone done{0u, 0u};
  PushStage st(stage, false);
  // presence in 32-bit words: word kk holds snapshots 32 kk .. 32 kk + 31, so
  // a lane of a 32-lane group tests bit gl of word kk for its kk-th snapshot
  constexpr int NW = P * K > 32 ? P * K / 32 : 1;
  uint32_t slab[NW];
#pragma unroll
  for (int k = 0; k < NW; ++k) slab[k] = a.ls >= 32u * (k + 1) ? ~0u : a.ls > 32u * k ? (1u << (a.ls - 32u * k)) - 1u : 0u;
  // G units (one per lane group) per batch
  const Batches bt{n, (uint32_t)G, nwarps, gwarp, &c->ticket[cur]};
  for (uint32_t t0 = bt.first(); t0 < n; t0 = bt.next(lane)) {
    const uint32_t ui = t0 + grp;
    uint32_t beg = 0, end = 0;  // of the unit, counted over the row's all-window edges and then the others
    uint4 d = make_uint4(0u, 0u, 0u, 0u);
    uint32_t room_end = 0;
    bool q1 = false;  // the unit's row belongs to the second query
    uint32_t sv[K];
#pragma unroll
    for (int kk = 0; kk < K; ++kk) sv[kk] = Op::kIdentity;
    if (ui < n) {
      const unsigned long long u = qin[ui];  // written before the last barrier
      const uint32_t r = (uint32_t)u, ch = (uint32_t)(u >> 32);
      q1 = r >= U0;
      d = a.qrow[r];
      room_end = a.qrow[r + 1].x;
      beg = ch << a.cshift;
      end = min(d.z + d.w, beg + (1u << a.cshift));
      const uint32_t* src = a.val + ((size_t)r << lps) + gl;
#pragma unroll
      for (int kk = 0; kk < K; ++kk) sv[kk] = ld_val(src + kk * P);
    }
    const uint32_t cnt = end > beg ? end - beg : 0u;
    const uint32_t maxcnt = __reduce_max_sync(kFullMask, cnt);
    if (gl == 0) done.edges += cnt;
    for (uint32_t j0 = 0; j0 < maxcnt; j0 += P) {
      const uint32_t e = beg + j0 + gl;
      uint32_t xr = 0, w = 0;
      uint32_t mw[NW];
#pragma unroll
      for (int k = 0; k < NW; ++k) mw[k] = slab[k];
      if (e < end) {
        const bool full = e < d.z;
        const uint32_t m = e - d.z;  // of the others, which end the row's room
        const uint2 ew = a.qcw[full ? d.x + e : room_end - 1u - m];
        xr = ew.x;
        w = ew.y;
        if (!full) {
          const uint64_t* mp = a.qmask + (size_t)(d.y + m) * a.QW;
#pragma unroll
          for (int k = 0; k < NW; k += 2) {
            const uint64_t x = mask_extract(mp, a.QW, a.s0 + 32u * k);
            mw[k] &= (uint32_t)x;
            if (k + 1 < NW) mw[k + 1] &= (uint32_t)(x >> 32);
          }
        }
      }
      bool pend = false;
      uint32_t pend_x = 0;
      const uint32_t nj = min((uint32_t)P, maxcnt - j0);
      // H edges per iteration: every target row is loaded before any is
      // compared, so each lane keeps H load chains in flight
      constexpr int H = (K <= 2) ? 4 : 2;
      for (uint32_t jj = 0; jj < nj; jj += H) {
        uint32_t ex[H], ewt[H];
        uint32_t curv[H][K];
        bool want[H][K];
#pragma unroll
        for (int h = 0; h < H; ++h) {
          const uint32_t src = min(jj + h, (uint32_t)P - 1u);
          ex[h] = __shfl_sync(kFullMask, xr, src, P);
          ewt[h] = __shfl_sync(kFullMask, w, src, P);
          const bool ev = (jj + h < nj) && (beg + j0 + jj + h) < end;
          uint32_t em[NW];
#pragma unroll
          for (int k = 0; k < NW; ++k) em[k] = __shfl_sync(kFullMask, mw[k], src, P);
          const uint32_t* row = a.val + ((size_t)ex[h] << lps) + gl;
#pragma unroll
          for (int kk = 0; kk < K; ++kk) {
            const uint32_t i = gl + kk * P;
            want[h][kk] = ev && ((P == 32 ? em[kk < NW ? kk : 0] >> gl : em[NW > 1 ? i >> 5 : 0] >> (i & 31u)) & 1u);
            curv[h][kk] = want[h][kk] ? ld_val(row + kk * P) : 0u;
          }
        }
        bool imp[H];
#pragma unroll
        for (int h = 0; h < H; ++h) {
          imp[h] = false;
          uint32_t* row = a.val + ((size_t)ex[h] << lps) + gl;
#pragma unroll
          for (int kk = 0; kk < K; ++kk) {
            if (want[h][kk]) {
              const uint32_t cand = relax_q<Op>(a, q1, sv[kk], ewt[h]);
              if (Op::better(cand, curv[h][kk])) {
                Op::red(row + kk * P, cand);
                if (kNote) note_best<Op>(&stage->best[q1 ? 1 : 0][gl + kk * P], cand);
                imp[h] = true;
              }
            }
          }
        }
#pragma unroll
        for (int h = 0; h < H; ++h) {
          const unsigned bi = __ballot_sync(kFullMask, imp[h]) & gmask;
          if (gl == jj + h && bi) {
            pend = true;
            pend_x = ex[h];
          }
        }
      }
      bool push = false;
      uint32_t deg = 0;
      if (pend) {
        const uint4 dx = a.qrow[pend_x];  // issued alongside the stamp exchange
        if (atomicExch(a.stamp + pend_x, stamp_next) != stamp_next) {
          push = true;
          deg = dx.z + dx.w;
        }
      }
      stage_push_units(push, pend_x, deg, a.cshift, st, qout, qn_out, a.qcap, c, a.qerr, lane);
    }
  }
  done.queued = stage_flush_cta(st, qout, qn_out, a.qcap, c, a.qerr, lane);
  return done;
}

template <class Op, int P, int K>
__device__ bool relax_team(const RelaxArgs& a, const Team& t, StageMem* stage) {
  const DevGraph& g = a.g;
  TeamCtl* c = a.ctl;
  const unsigned lane = threadIdx.x & 31u;
  const unsigned nthreads = t.nthreads();
  const unsigned gtid = t.tid();
  // neighbouring work goes to different SMs, so that a small round is spread
  // over all of them
  const unsigned gwarp = (threadIdx.x >> 5) * t.nblocks + t.rank, nwarps = nthreads >> 5;
  if (cta_read(a.qerr) != 0u) return false;
  PushStage st(stage, true);
  // rows [0, U0) are the first query's, [U0, U) a second query's (a.counts1)
  const uint32_t U0 = a.counts[0];
  const uint32_t U = U0 + (a.counts1 ? a.counts1[0] : 0u);
  constexpr bool kPull = P == 32;  // rows of at least 32 snapshots: a lane per snapshot is worth it
  // A pull round looks at every in-edge of the unstable vertices (about U * E /
  // V), a push round at the frontier's share of the kept edges: pull when that
  // is more than 0.4 of the former (measured at 0.35-0.41: 308 us against 271,
  // 438 against 412; at 0.5: 531 against 579, at 0.7: 525 against 775; rounds of
  // one scale-20 query with 533K unstable vertices).  Where the unstable vertices'
  // mean in-degree is above E / V a pull costs more than this counts.
  // pull_above is that frontier in units; most queries never get there.
  const uint32_t all_units = U + (a.counts[2] >> a.cshift);
  const float few = 0.4f * (float)U * ((float)g.E / (float)g.V), kept = (float)a.counts[2];
  const bool may_pull = kPull && g.pull && kept > few;
  const uint32_t pull_above = may_pull ? (uint32_t)(few * ((float)all_units / kept)) : 0xFFFFFFFFu;
  uint32_t(&s_best)[2][kBestSnaps] = stage->best;
  if (kPull) {
    for (uint32_t i = threadIdx.x; i < 2u * kBestSnaps; i += blockDim.x) (&s_best[0][0])[i] = 0u;
    for (uint32_t i = gtid; i < 3u * 2u * kBestSnaps; i += nthreads) a.best[i] = 0u;
    if (threadIdx.x == 0) stage->changed = 0u;
  }
  // the CTA's best values into the ring slot of a round; a CTA barrier before and after
  auto publish_best = [&](uint32_t slot) {
    if (!may_pull) return;
    for (uint32_t i = threadIdx.x; i < 2u * kBestSnaps; i += blockDim.x) {
      uint32_t* s = &s_best[0][0] + i;
      if (*s) {
        atomicMax(a.best + slot * 2u * kBestSnaps + i, *s);
        *s = 0u;
      }
    }
  };
  const uint32_t LP = a.LP;
  const uint32_t lps = __ffs(LP) - 1;  // LP is a power of two

  // ---- round 0a: values and stamps.  A warp reads the starting values of
  // 32 rows at once (a lane per row), then writes those rows together (a
  // lane per column), so the dependent loads are paid once per 32 rows.
  for (uint32_t r0 = gwarp * 32u; r0 < U; r0 += nwarps * 32u) {
    const uint32_t r = r0 + lane;
    const uint32_t x = r < U ? ((r < U0 ? a.rI : a.rI1)[a.uv[r]] ^ ((a.flip >> (r < U0 ? 0 : 1)) & 1u ? ~0u : 0u))
                             : 0u;
    if (r < U) a.stamp[r] = 0u;
    const uint32_t nr = min(32u, U - r0);
    for (uint32_t k = 0; k < nr; ++k) {
      const uint32_t xv = __shfl_sync(kFullMask, x, k);
      uint32_t* row = a.val + ((size_t)(r0 + k) << lps);
      for (uint32_t i = lane; i < LP; i += 32u) row[i] = xv;
    }
  }
  if (!t.sync()) return false;
  if (a.trace && gtid == 0 && a.trace_cap) a.trace[0] = global_ns() & 0xFFFFFFFFFFull;

  // ---- round 0b: seed from addition edges with an unstable sink; four
  // qualifying edges per warp iteration, lanes over the slab's snapshots
  // each query's seeds (the second query's rows map to its own range)
  for (int qi = 0; qi < (a.counts1 ? 2 : 1); ++qi) {
    const uint32_t* srow = qi ? a.row1 : a.row;
    const uint32_t* srI = qi ? a.rI1 : a.rI;
    const Window swin = qi ? a.win1 : a.win;
    const uint32_t ssnap = swin.b + a.s0;
    const uint32_t sflip = ((a.flip >> qi) & 1u) ? ~0u : 0u;
    for (uint32_t k0 = gwarp * 32u; k0 < g.NF; k0 += nwarps * 32u) {
      const uint32_t k = k0 + lane;
      bool qual = false;
      uint32_t rx = kNone, cand = 0;
      if (k < g.NF) {
        const uint2 e = __ldg(g.nfcw + k);
        rx = srow[e.x];
        if (rx != kNone) {
          bool any, all;
          window_any_all(g.nfmask + (size_t)k * g.W, swin, any, all);
          qual = any && !all;
          if (qual) cand = relax_q<Op>(a, qi != 0, srI[__ldg(g.nfsrc + k)] ^ sflip, e.y);
        }
      }
      // the owner lane extracts the slab's presence bits once; the warp then
      // takes four qualifying edges at a time with the bits in registers
      uint64_t mlo = 0ull, mhi = 0ull;
      if (qual) {
        const uint64_t* mp = g.nfmask + (size_t)k * g.W;
        mlo = mask_extract(mp, g.W, ssnap);
        if (a.ls > 64u) mhi = mask_extract(mp, g.W, ssnap + 64u);
      }
      unsigned bq = __ballot_sync(kFullMask, qual);
      constexpr int HS = 4;
      while (bq) {
        int j[HS];
  #pragma unroll
        for (int h = 0; h < HS; ++h) {
          j[h] = bq ? __ffs(bq) - 1 : -1;
          if (bq) bq &= bq - 1u;
        }
        uint32_t ex[HS], ec[HS];
        uint64_t ml[HS], mh[HS];
  #pragma unroll
        for (int h = 0; h < HS; ++h) {
          const int src = j[h] < 0 ? j[0] : j[h];
          ex[h] = __shfl_sync(kFullMask, rx, src);
          ec[h] = __shfl_sync(kFullMask, cand, src);
          ml[h] = __shfl_sync(kFullMask, mlo, src);
          mh[h] = __shfl_sync(kFullMask, mhi, src);
        }
        bool imp[HS];
  #pragma unroll
        for (int h = 0; h < HS; ++h) imp[h] = false;
        for (uint32_t i = lane; i < a.ls; i += 32u) {
          bool want[HS];
          uint32_t curv[HS];
  #pragma unroll
          for (int h = 0; h < HS; ++h) {
            const uint64_t bit = i < 64u ? (ml[h] >> i) : (mh[h] >> (i - 64u));
            want[h] = j[h] >= 0 && (bit & 1ull);
            curv[h] = want[h] ? ld_val(a.val + ((size_t)ex[h] << lps) + i) : 0u;
          }
  #pragma unroll
          for (int h = 0; h < HS; ++h) {
            if (want[h] && Op::better(ec[h], curv[h])) {
              Op::red(a.val + ((size_t)ex[h] << lps) + i, ec[h]);
              if (may_pull) note_best<Op>(&s_best[qi][i], ec[h]);
              imp[h] = true;
            }
          }
        }
        // lane h claims edge h's target (the HS stamp exchanges run side by
        // side) and one warp append queues every claimed row
        unsigned anyb = 0;
  #pragma unroll
        for (int h = 0; h < HS; ++h) anyb |= (__any_sync(kFullMask, imp[h]) ? 1u : 0u) << h;
        uint32_t px = 0;
        bool claim = false;
  #pragma unroll
        for (int h = 0; h < HS; ++h)
          if (lane == (unsigned)h) {
            px = ex[h];
            claim = (anyb >> h) & 1u;
          }
        bool push = false;
        uint32_t deg = 0;
        if (claim) {
          const uint4 d = a.qrow[px];
          if (atomicExch(a.stamp + px, 1u) != 1u) {
            push = true;
            deg = d.z + d.w;
          }
        }
        stage_push_units(push, px, deg, a.cshift, st, a.q1, &c->qn[1], a.qcap, c, a.qerr, lane);
      }
    }
  }
  uint32_t queued = stage_flush_cta(st, a.q1, &c->qn[1], a.qcap, c, a.qerr, lane);
  publish_best(1u);
  uint32_t n = 0;  // the round's frontier: units, or improved (row, item part) pairs after a pull round
  bool dense = false;
  if (!t.sync(queued, n)) return false;

  // ---- rounds >= 1: Algorithm 2 while-loop over the frontier
  unsigned long long relaxed = 0;
  uint32_t it = 1;
  for (;; ++it) {
    const uint32_t cur = it % 3u, nxt = (it + 1u) % 3u, clr = (it + 2u) % 3u;
    if (a.trace && gtid == 0 && it < a.trace_cap) a.trace[it] = ((unsigned long long)n << 40) | (global_ns() & 0xFFFFFFFFFFull);
    if (n == 0u) break;
    if (it > a.maxit) {
      if (gtid == 0) set_err(c, a.qerr, kErrTimeout);
      break;
    }
    n = min(n, a.qcap);
    // after a pull round n counts a row once for every part of an item that
    // improved it; taken as a row, which has all_units / U units on average
    const bool pull = may_pull && (dense ? (float)n * ((float)all_units / (float)U) : (float)n) > (float)pull_above;
    if (gtid == 0) {
      atomicExch(&c->qn[clr], 0u);
      atomicExch(&c->ticket[clr], 0u);
      atomicExch(&c->aux[6 + ((it + 1u) & 1u)], 0u);  // compaction counter of the next round
    }
    if (may_pull && t.rank == 0)
      for (uint32_t i = threadIdx.x; i < 2u * kBestSnaps; i += blockDim.x) a.best[clr * 2u * kBestSnaps + i] = 0u;
    if constexpr (kPull) {
      if (pull) {
        const uint32_t changed = relax_pull_round<Op, K>(a, it, stage, gwarp, nwarps);
        fold_changes(changed, &stage->changed, lane);
        __syncthreads();
        publish_best(nxt);
        if (!t.sync(take_changes(&stage->changed), n)) return false;
        dense = true;
        continue;
      }
    }
    unsigned long long* qin = (it & 1u) ? a.q1 : a.q0;
    if (dense) {
      // ---- the last round pulled: queue the rows it changed (stamp == it)
      unsigned* cnt_ctr = &c->aux[6 + (it & 1u)];
      for (uint32_t r0 = gwarp * 32u; r0 < U; r0 += nwarps * 32u) {
        const uint32_t r = r0 + lane;
        const bool take = r < U && ld_cg(a.stamp + r) == it;
        uint32_t deg = 0;
        if (take) {
          const uint4 d = a.qrow[r];
          deg = d.z + d.w;
        }
        stage_push_units(take, r, deg, a.cshift, st, qin, cnt_ctr, a.qcap, c, a.qerr, lane);
      }
      queued = stage_flush_cta(st, qin, cnt_ctr, a.qcap, c, a.qerr, lane);
      if (!t.sync(queued, n)) return false;
      n = min(n, a.qcap);
      dense = false;
    }
    unsigned long long* qout = (it & 1u) ? a.q0 : a.q1;
    const RelaxRound rr{n, it, U0, gwarp, nwarps, qin, qout};
    RelaxDone rd;
    if (kPull && may_pull) rd = relax_push_round<Op, P, K, true>(a, rr, stage);
    else rd = relax_push_round<Op, P, K, false>(a, rr, stage);
    relaxed += rd.edges;
    publish_best(nxt);
    if (!t.sync(rd.queued, n)) return false;
  }
  if (relaxed) atomicAdd(&c->relaxed, relaxed);
  if (gtid == 0) c->iters = it - 1u;
  return true;
}

// Output scatter over a team: tiles of kScatterTV vertices x ls snapshots are
// staged in `tile` (ls * (kScatterTV + 1) words of shared memory) so the row
// reads and the snapshot-major writes both coalesce.
constexpr int kScatterTV = 64;

__device__ __forceinline__ void scatter_team(const ScatterArgs& a, const Team& t, uint32_t* tile) {
  const unsigned lane = threadIdx.x & 31u, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const uint32_t lps = __ffs(a.LP) - 1;
  const uint32_t ntiles = (a.V + kScatterTV - 1) / kScatterTV;
  for (uint32_t tl = t.rank; tl < ntiles; tl += t.nblocks) {
    const uint32_t v0 = tl * kScatterTV;
    for (uint32_t tv = wid; tv < (uint32_t)kScatterTV; tv += nw) {
      const uint32_t v = v0 + tv;
      if (v >= a.V) break;
      const uint32_t r = a.row[v];
      if (r == kNone) {
        const uint32_t x = a.rI[v];
        for (uint32_t i = lane; i < a.ls; i += 32u) tile[i * (kScatterTV + 1) + tv] = x;
      } else {
        const uint32_t* src = a.val + ((size_t)r << lps);
        for (uint32_t i = lane; i < a.ls; i += 32u) tile[i * (kScatterTV + 1) + tv] = __ldcg(src + i);
      }
    }
    __syncthreads();
    const uint32_t nv = min((uint32_t)kScatterTV, a.V - v0);
    for (uint32_t idx = threadIdx.x; idx < a.ls * (uint32_t)kScatterTV; idx += blockDim.x) {
      const uint32_t i = idx / kScatterTV, tv = idx % kScatterTV;
      if (tv < nv) a.out[(size_t)(a.s0 + i) * a.V + v0 + tv] = tile[i * (kScatterTV + 1) + tv];
    }
    __syncthreads();
  }
}

}  // namespace svv
