// svv_qrs.cuh -- stable-vertex compaction and Q-relevant subgraph extraction
// as a team phase (see svv_qrs.cu for what it computes).
#pragma once

#include "svv_device.cuh"
#include "svv_team.cuh"

namespace svv {



// what a range of vertices needs in the subgraph's arrays
struct QrsSum {
  uint32_t rows, units, deg, part;  // unstable vertices, their units, out-edges and partial out-edges
  __device__ __forceinline__ void add(const QrsSum& o) {
    rows += o.rows;
    units += o.units;
    deg += o.deg;
    part += o.part;
  }
};

__device__ __forceinline__ QrsSum warp_incl_scan(QrsSum x, unsigned lane) {
  return QrsSum{warp_incl_scan(x.rows, lane), warp_incl_scan(x.units, lane), warp_incl_scan(x.deg, lane),
                warp_incl_scan(x.part, lane)};
}

// sums over the warps before this one, and over the block
__device__ __forceinline__ void block_sums(const QrsSum& warp_total, QrsSum& before, QrsSum& total) {
  __shared__ QrsSum s[32];
  const unsigned lane = threadIdx.x & 31u, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (lane == 0) s[wid] = warp_total;
  __syncthreads();
  before = total = QrsSum{};
  for (unsigned i = 0; i < nw; ++i) {
    if (i < wid) before.add(s[i]);
    total.add(s[i]);
  }
  __syncthreads();
}

__device__ __forceinline__ QrsSum warp_sum(const QrsSum& x) {
  return QrsSum{__reduce_add_sync(kFullMask, x.rows), __reduce_add_sync(kFullMask, x.units),
                __reduce_add_sync(kFullMask, x.deg), __reduce_add_sync(kFullMask, x.part)};
}

// a vertex's share, if its bounds differ (with pruning off every vertex has a row)
__device__ __forceinline__ QrsSum vertex_share(const QrsArgs& a, uint32_t v, bool unstable) {
  if (!unstable) return QrsSum{};
  const uint4 rd = __ldg(a.g.rowd + v);
  const uint32_t deg = rd.y - rd.x;
  return QrsSum{1u, (deg + (1u << a.cshift) - 1u) >> a.cshift, deg, rd.y - rd.z};
}

// bit h of the result: vertex v + h (< hi) is unstable; v is a multiple of 4
__device__ __forceinline__ uint32_t unstable4(const QrsArgs& a, const uint32_t* I, const uint32_t* U, uint32_t v,
                                              uint32_t hi) {
  if (v >= hi) return 0u;
  const uint32_t in = hi - v < 4u ? (1u << (hi - v)) - 1u : 15u;
  if (!a.prune) return in;
  if (in == 15u) {
    const uint4 x = *reinterpret_cast<const uint4*>(I + v), y = *reinterpret_cast<const uint4*>(U + v);
    return (x.x != y.x ? 1u : 0u) | (x.y != y.y ? 2u : 0u) | (x.z != y.z ? 4u : 0u) | (x.w != y.w ? 8u : 0u);
  }
  uint32_t m = 0;
  for (uint32_t h = 0; h < hi - v; ++h) m |= (I[v + h] != U[v + h] ? 1u : 0u) << h;
  return m;
}

// Walk the edges of every unit in the queue (warp-balanced, as in the solve),
// classify each edge as all-window (F) or masked (M) kept edge, and write the
// kept ones next to those their rows already hold.  Returns (in lane 0) the
// numbers of kept and of masked edges.  With a second query (a.rI1), rows from
// U0 on are that query's: its edges are classified against its own row map and
// window.
__device__ __forceinline__ uint2 qrs_fill(const QrsArgs& a, const Team& t, uint32_t NU, uint32_t U0, unsigned* ticket) {
  uint2 kept = make_uint2(0u, 0u);
  const DevGraph& g = a.g;
  const unsigned lane = threadIdx.x & 31u;
  const unsigned lt = (1u << lane) - 1u;
  const uint32_t nwarps = t.nthreads() >> 5;
  const uint32_t gwarp = (threadIdx.x >> 5) * t.nblocks + t.rank;
  const Batches bt{NU, batch_size(NU, nwarps, 32u), nwarps, gwarp, ticket};
  const uint32_t tk = bt.tk;
  for (uint32_t t0 = bt.first(); t0 < NU; t0 = bt.next(lane)) {
    const uint32_t ui = t0 + lane;
    uint32_t r = 0, beg = 0, cnt = 0, fe = 0, nfb = 0;
    if (lane < tk && ui < NU) {
      const unsigned long long u = a.units[ui];  // earlier phases: ordered by the barrier
      r = (uint32_t)u;
      const uint32_t ch = (uint32_t)(u >> 32);
      const uint32_t v = a.uv[r];
      const uint4 rd = __ldg(g.rowd + v);
      const uint32_t r0 = rd.x, r1 = rd.y;
      fe = rd.z;
      nfb = rd.w;
      beg = r0 + (ch << a.cshift);
      const uint32_t end = min(r1, beg + (1u << a.cshift));
      cnt = end > beg ? end - beg : 0u;
    }
    const uint32_t incl = warp_incl_scan(cnt, lane);
    const uint32_t total = __shfl_sync(kFullMask, incl, 31);
    // two 32-edge steps per iteration: both steps' loads are issued before
    // either step's counts or writes
    for (uint32_t p0 = 0; p0 < total; p0 += 64u) {
      int kk[2];
      uint32_t rkk[2], rx[2], w[2];
      bool isF[2], isM[2];
      uint32_t mi[2];  // a partial edge's index in the partial list
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint32_t p = p0 + 32u * h + lane;
        const int k = warp_owner(incl, p < total ? p : total - 1u);
        const uint32_t ik = __shfl_sync(kFullMask, incl, k);
        const uint32_t ck = __shfl_sync(kFullMask, cnt, k);
        const uint32_t bk = __shfl_sync(kFullMask, beg, k);
        const uint32_t fk = __shfl_sync(kFullMask, fe, k);
        const uint32_t nk = __shfl_sync(kFullMask, nfb, k);
        kk[h] = k;
        rkk[h] = __shfl_sync(kFullMask, r, k);
        isF[h] = isM[h] = false;
        rx[h] = kNone;
        w[h] = 0;
        mi[h] = 0u;
        if (p < total) {
          const uint32_t e = bk + (p - (ik - ck));
          const uint2 ew = __ldg(g.cw + e);
          const bool q1 = a.rI1 && rkk[h] >= U0;
          rx[h] = (q1 ? a.row1 : a.row)[ew.x];
          w[h] = ew.y;
          if (rx[h] != kNone) {
            if (e < fk) {
              isF[h] = true;
            } else {
              mi[h] = nk + (e - fk);
              bool any, all;
              window_any_all(g.nfmask + (size_t)mi[h] * g.W, q1 ? a.win1 : a.win, any, all);
              isF[h] = all;
              isM[h] = any && !all;
            }
          }
        }
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint32_t p = p0 + 32u * h + lane;
        const uint32_t rk = rkk[h];
        const unsigned grp = __match_any_sync(kFullMask, p < total ? (uint32_t)kk[h] : 64u + lane);
        const unsigned bF = __ballot_sync(kFullMask, isF[h]), bM = __ballot_sync(kFullMask, isM[h]);
        const int leader = __ffs(grp) - 1;
        const uint32_t nF = __popc(grp & bF), nM = __popc(grp & bM);
        uint4* d = a.qrow + rk;
        uint32_t baseF = 0, baseM = 0, baseE = 0;  // baseE: where the row's masked edges go on, downwards
        if (lane == (unsigned)leader && p < total && (nF || nM)) {
          const uint2 at = __ldcg(reinterpret_cast<const uint2*>(d));  // {first slot, first mask}
          const uint32_t end = __ldcg(&d[1].x);
          const uint32_t oF = nF ? atomicAdd(&d->z, nF) : 0u, oM = nM ? atomicAdd(&d->w, nM) : 0u;
          baseF = at.x + oF;
          baseM = at.y + oM;
          baseE = end - 1u - oM;
        }
        baseF = __shfl_sync(kFullMask, baseF, leader);
        baseM = __shfl_sync(kFullMask, baseM, leader);
        baseE = __shfl_sync(kFullMask, baseE, leader);
        if (isF[h]) {
          a.qcw[baseF + __popc(grp & bF & lt)] = make_uint2(rx[h], w[h]);
        } else if (isM[h]) {
          const uint32_t k = __popc(grp & bM & lt);
          a.qcw[baseE - k] = make_uint2(rx[h], w[h]);
          uint64_t* out = a.qmask + (size_t)(baseM + k) * a.QW;
          const uint32_t wb = (a.rI1 && rk >= U0) ? a.win1.b : a.win.b;
          for (uint32_t j = 0; j < a.QW; ++j) {
            uint64_t word = mask_extract(g.nfmask + (size_t)mi[h] * g.W, g.W, wb + 64u * j);
            const uint32_t left = a.win.l - 64u * j;
            if (left < 64u) word &= (1ull << left) - 1ull;
            out[j] = word;
          }
        }
        kept.x += __popc(bF) + __popc(bM);
        kept.y += __popc(bM);
      }
    }
  }
  return kept;
}

__device__ inline bool qrs_team(const QrsArgs& a, const Team& t) {
  const DevGraph& g = a.g;
  TeamCtl* c = a.ctl;
  const unsigned nb = t.nblocks, b = t.rank, tid = threadIdx.x;
  if (cta_read(a.qerr) != 0u) return false;
  const uint32_t V = g.V;
  // A second query (a.rI1) is extracted in the same launch: its rows, units
  // and edges follow the first query's.
  const int nq = a.rI1 ? 2 : 1;

  // ---- P1: what each CTA's vertex range needs, per query
  if (a.trace && b == 0 && tid == 0) a.trace[0] = global_ns();
  const unsigned long long per = (((unsigned long long)V + nb - 1) / nb + 31ull) & ~31ull;
  const uint32_t lo = (uint32_t)min((unsigned long long)V, per * b);
  const uint32_t hi = (uint32_t)min((unsigned long long)V, per * b + per);
  for (int qi = 0; qi < nq; ++qi) {
    const uint32_t* qI = qi ? a.rI1 : a.rI;
    const uint32_t* qU = qi ? a.rU1 : a.rU;
    QrsSum sum{};
    for (uint32_t v = lo + 4u * tid; v < hi; v += 4u * blockDim.x) {
      uint32_t m = unstable4(a, qI, qU, v, hi);
      for (; m; m &= m - 1u) sum.add(vertex_share(a, v + __ffs(m) - 1, true));
    }
    QrsSum before, total;
    block_sums(warp_sum(sum), before, total);
    if (tid == 0) reinterpret_cast<uint4*>(a.part)[2 * b + qi] = make_uint4(total.rows, total.units, total.deg, total.part);
  }
  if (!t.sync()) return false;

  // ---- P2: rows and units in vertex order, the first query's then the
  // second's; a row has room for all its out-edges, so nothing is counted first
  if (a.trace && b == 0 && tid == 0) a.trace[1] = global_ns();
  QrsSum base{};  // the queries before
  uint32_t U0 = 0;
  for (int qi = 0; qi < nq; ++qi) {
    const uint32_t* qI = qi ? a.rI1 : a.rI;
    const uint32_t* qU = qi ? a.rU1 : a.rU;
    uint32_t* qrowmap = qi ? a.row1 : a.row;
    QrsSum mine{}, all{};
    for (uint32_t j = tid; j < nb; j += blockDim.x) {
      const uint4 x = __ldcg(reinterpret_cast<const uint4*>(a.part) + 2 * j + qi);
      const QrsSum s{x.x, x.y, x.z, x.w};
      all.add(s);
      if (j < b) mine.add(s);
    }
    QrsSum none, at, total;
    block_sums(warp_sum(mine), none, at);
    block_sums(warp_sum(all), none, total);
    at.add(base);  // where this CTA's range begins
    base.add(total);
    if (qi == 0) U0 = total.rows;
    if (b == 0 && tid == 0) {
      if (qi == 0) {
        c->aux[0] = total.rows;
        c->aux[1] = total.units;
      } else {
        a.counts1_out[0] = total.rows;
      }
    }
    if (base.units > a.ucap || base.rows > a.rowcap || base.deg > a.ecap ||
        (unsigned long long)base.part * a.QW > a.mcap) {
      if (tid == 0) set_err(c, a.qerr, kErrInternal);
      return false;  // every CTA sees the same totals and leaves here
    }
    const unsigned lane = tid & 31u;
    for (uint32_t v0 = lo; v0 < hi; v0 += 4u * blockDim.x) {
      const uint32_t v = v0 + 4u * tid;
      const uint32_t m = unstable4(a, qI, qU, v, hi);
      QrsSum sum{};
#pragma unroll
      for (uint32_t h = 0; h < 4u; ++h) sum.add(vertex_share(a, v + h, (m >> h) & 1u));
      const QrsSum incl = warp_incl_scan(sum, lane);
      const QrsSum wt{__shfl_sync(kFullMask, incl.rows, 31), __shfl_sync(kFullMask, incl.units, 31),
                      __shfl_sync(kFullMask, incl.deg, 31), __shfl_sync(kFullMask, incl.part, 31)};
      QrsSum before, btotal;
      block_sums(wt, before, btotal);
      QrsSum p = at;  // of this lane's first vertex
      p.add(before);
      p.rows += incl.rows - sum.rows;
      p.units += incl.units - sum.units;
      p.deg += incl.deg - sum.deg;
      p.part += incl.part - sum.part;
      at.add(btotal);
#pragma unroll 1
      for (uint32_t h = 0; h < 4u; ++h) {
        const bool on = (m >> h) & 1u;
        const QrsSum own = vertex_share(a, v + h, on);  // again: cheaper than keeping four
        if (v + h < hi) {
          qrowmap[v + h] = on ? p.rows : kNone;
          if (on) {
            a.uv[p.rows] = v + h;
            a.qrow[p.rows] = make_uint4(p.deg, p.part, 0u, 0u);
          }
        }
        // the warp writes its vertices' units together, so a hub's hundreds
        // of units do not serialise on one thread
        const uint32_t nu = own.units;
        const uint32_t ui = warp_incl_scan(nu, lane);
        const uint32_t wtot = __shfl_sync(kFullMask, ui, 31);
        for (uint32_t j0 = 0; j0 < wtot; j0 += 32u) {
          const uint32_t j = j0 + lane;
          const int k = warp_owner(ui, j < wtot ? j : wtot - 1u);
          const uint32_t ik = __shfl_sync(kFullMask, ui, k), nk = __shfl_sync(kFullMask, nu, k);
          const uint32_t rk = __shfl_sync(kFullMask, p.rows, k), ek = __shfl_sync(kFullMask, p.units, k);
          const uint32_t jj = j - (ik - nk);
          if (j < wtot) a.units[ek + jj] = (unsigned long long)rk | ((unsigned long long)jj << 32);
        }
        p.add(own);
      }
    }
  }
  if (b == 0 && tid == 0) a.qrow[base.rows] = make_uint4(base.deg, base.part, 0u, 0u);
  if (!t.sync()) return false;

  // ---- P3: fill
  if (a.trace && b == 0 && tid == 0) a.trace[2] = a.trace[3] = a.trace[4] = global_ns();
  const uint2 kept = qrs_fill(a, t, base.units, U0, &c->ticket[0]);
  QrsSum none, total;
  block_sums(QrsSum{kept.x, kept.y, 0u, 0u}, none, total);
  if (tid == 0) {
    if (total.rows) atomicAdd(&c->aux[2], total.rows);
    if (total.units) atomicAdd(&c->aux[3], total.units);
    if (a.trace) atomicMax(a.trace + 5, global_ns());  // the last CTA to finish
  }
  return true;
}

}  // namespace svv
