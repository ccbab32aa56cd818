// svv_push.cuh -- warp-cooperative frontier append.
#pragma once

#include "svv_device.cuh"

namespace svv {

// Every lane with `push` set appends the work units of vertex (or row) `x`:
// ceil(deg / 2^cshift) units "x | chunk << 32", none when deg == 0.  The warp
// reserves space with one atomic and writes the units cooperatively, so a hub
// with thousands of units costs its warp a few stores per lane, not one lane
// thousands.  All 32 lanes must call this.
__device__ __forceinline__ void warp_push_units(bool push, uint32_t x, uint32_t deg, uint32_t cshift,
                                                unsigned long long* q, unsigned* qn, uint32_t qcap,
                                                TeamCtl* c, uint32_t* qerr, unsigned lane) {
  if (__ballot_sync(kFullMask, push) == 0u) return;
  uint32_t nu = push ? ((deg + (1u << cshift) - 1u) >> cshift) : 0u;
  uint32_t incl = warp_incl_scan(nu, lane);
  uint32_t tot = __shfl_sync(kFullMask, incl, 31);
  if (tot == 0u) return;
  uint32_t base = 0;
  if (lane == 31) base = atomicAdd(qn, tot);
  base = __shfl_sync(kFullMask, base, 31);
  if ((unsigned long long)base + tot > qcap) {
    if (lane == 0) set_err(c, qerr, kErrInternal);
    return;
  }
  for (uint32_t j0 = 0; j0 < tot; j0 += 32u) {
    uint32_t j = j0 + lane;
    int k = warp_owner(incl, j < tot ? j : tot - 1u);
    uint32_t xk = __shfl_sync(kFullMask, x, k);
    uint32_t ik = __shfl_sync(kFullMask, incl, k);
    uint32_t nk = __shfl_sync(kFullMask, nu, k);
    if (j < tot) q[base + j] = (unsigned long long)xk | ((unsigned long long)(j - (ik - nk)) << 32);
  }
}

// ---------------------------------------------------------------------------
// Staged append.  Every warp appends into a private buffer of kStageUnits
// units in shared memory and copies it to the queue with one atomic when it
// fills; at the end of a round the CTA copies all leftovers with one atomic.
// One counter serves every warp of the grid, and same-address atomics
// serialise in L2, so an atomic per push would cap a round's throughput.
constexpr uint32_t kStageUnits = 64;

// A vertex of more than kHubUnits units goes to a list of the CTA, and the
// whole CTA writes the listed units at the end of the round: a round of a few
// edges can queue tens of thousands of units (at scale 20 the source's first
// 3,000 edges queue 84,000), which one warp would write alone.
constexpr uint32_t kHubUnits = 32, kStageHubs = 128;

struct StageHubs {  // in shared memory
  uint32_t n;                            // vertices listed (may pass kStageHubs: those took the other way)
  uint32_t x[kStageHubs], units[kStageHubs], off[kStageHubs];
};

constexpr int kStageThreads = 512;  // of every kernel that stages pushes
struct StageMem {  // a kernel's shared memory for staged pushes
  unsigned long long units[(kStageThreads / 32) * kStageUnits];
  StageHubs hubs;
  uint32_t best[2][kBestSnaps];  // the relaxation's, here so that its instances share it
  uint32_t changed;              // improvements of a pull round
};

struct PushStage {
  unsigned long long* buf;  // this warp's slots in shared memory
  uint32_t fill;            // warp-uniform
  uint32_t out;             // units this warp copied to the queue in this round (warp-uniform)
  StageHubs* hubs;
  // `fresh`: the first stage of the kernel on this memory (a CTA barrier comes
  // before its first push); else everything staged before has been flushed
  __device__ __forceinline__ PushStage(StageMem* m, bool fresh)
      : buf(m->units + (threadIdx.x >> 5) * kStageUnits), fill(0u), out(0u), hubs(&m->hubs) {
    if (fresh && threadIdx.x == 0) m->hubs.n = 0u;
  }
};

__device__ __forceinline__ void stage_flush_warp(PushStage& st, unsigned long long* q, unsigned* qn,
                                                 uint32_t qcap, TeamCtl* c, uint32_t* qerr, unsigned lane) {
  if (st.fill == 0u) return;
  uint32_t base = 0;
  if (lane == 0) base = atomicAdd(qn, st.fill);
  base = __shfl_sync(kFullMask, base, 0);
  __syncwarp();
  if ((unsigned long long)base + st.fill > qcap) {
    if (lane == 0) set_err(c, qerr, kErrInternal);
  } else {
    for (uint32_t j = lane; j < st.fill; j += 32u) q[base + j] = st.buf[j];
  }
  __syncwarp();
  st.out += st.fill;
  st.fill = 0;
}

// Same contract as warp_push_units, through the warp's stage.
__device__ __forceinline__ void stage_push_units(bool push, uint32_t x, uint32_t deg, uint32_t cshift,
                                                 PushStage& st, unsigned long long* q, unsigned* qn,
                                                 uint32_t qcap, TeamCtl* c, uint32_t* qerr, unsigned lane) {
  if (__ballot_sync(kFullMask, push) == 0u) return;
  uint32_t nu = push ? ((deg + (1u << cshift) - 1u) >> cshift) : 0u;
  if (nu > kHubUnits) {
    const uint32_t h = atomicAdd(&st.hubs->n, 1u);
    if (h < kStageHubs) {
      st.hubs->x[h] = x;
      st.hubs->units[h] = nu;
      nu = 0u;
    }
  }
  const uint32_t incl = warp_incl_scan(nu, lane);
  const uint32_t tot = __shfl_sync(kFullMask, incl, 31);
  if (tot == 0u) return;
  unsigned long long* dst;
  if (tot > kStageUnits) {  // more than the stage holds: straight to the queue
    uint32_t base = 0;
    if (lane == 31) base = atomicAdd(qn, tot);
    base = __shfl_sync(kFullMask, base, 31);
    if ((unsigned long long)base + tot > qcap) {
      if (lane == 0) set_err(c, qerr, kErrInternal);
      return;
    }
    dst = q + base;
    st.out += tot;
  } else {
    if (st.fill + tot > kStageUnits) stage_flush_warp(st, q, qn, qcap, c, qerr, lane);
    dst = st.buf + st.fill;
    st.fill += tot;
  }
  for (uint32_t j0 = 0; j0 < tot; j0 += 32u) {
    const uint32_t j = j0 + lane;
    const int k = warp_owner(incl, j < tot ? j : tot - 1u);
    const uint32_t xk = __shfl_sync(kFullMask, x, k);
    const uint32_t ik = __shfl_sync(kFullMask, incl, k);
    const uint32_t nk = __shfl_sync(kFullMask, nu, k);
    if (j < tot) dst[j] = (unsigned long long)xk | ((unsigned long long)(j - (ik - nk)) << 32);
  }
  __syncwarp();
}

// End of a round: every warp's leftovers go to the queue with one atomic per
// CTA.  Every thread of the CTA must call it; a CTA barrier follows (the
// team's) before the stages are used again.  Returns, in thread 0, the units
// the CTA queued since the last flush.
__device__ __forceinline__ uint32_t stage_flush_cta(PushStage& st, unsigned long long* q, unsigned* qn,
                                                uint32_t qcap, TeamCtl* c, uint32_t* qerr, unsigned lane) {
  __shared__ uint32_t s_off[33], s_out[32], s_hubs;
  const unsigned wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (lane == 0) {
    s_off[wid] = st.fill;
    s_out[wid] = st.out;
  }
  uint32_t queued = 0;
  __syncthreads();
  if (wid == 0) {
    const uint32_t f = lane < nw ? s_off[lane] : 0u;
    const uint32_t incl = warp_incl_scan(f, lane);
    uint32_t tot = __shfl_sync(kFullMask, incl, 31);
    if (lane < nw) s_off[lane] = incl - f;
    const uint32_t nh = min(st.hubs->n, kStageHubs);
    for (uint32_t h0 = 0; h0 < nh; h0 += 32u) {
      const uint32_t u = h0 + lane < nh ? st.hubs->units[h0 + lane] : 0u;
      const uint32_t hi = warp_incl_scan(u, lane);
      if (h0 + lane < nh) st.hubs->off[h0 + lane] = tot + hi - u;
      tot += __shfl_sync(kFullMask, hi, 31);
    }
    queued = tot + __reduce_add_sync(kFullMask, lane < nw ? s_out[lane] : 0u);
    if (lane == 0) {
      uint32_t base = 0;
      if (tot) {
        base = atomicAdd(qn, tot);
        if ((unsigned long long)base + tot > qcap) {
          set_err(c, qerr, kErrInternal);
          base = 0xFFFFFFFFu;
        }
      }
      s_off[32] = base;
      s_hubs = nh;
      st.hubs->n = 0u;
    }
  }
  __syncthreads();
  const uint32_t base = s_off[32];
  if (base != 0xFFFFFFFFu) {
    for (uint32_t j = lane; j < st.fill; j += 32u) q[base + s_off[wid] + j] = st.buf[j];
    for (uint32_t h = wid; h < s_hubs; h += nw) {
      const uint32_t x = st.hubs->x[h], nu = st.hubs->units[h];
      unsigned long long* dst = q + base + st.hubs->off[h];
      for (uint32_t j = lane; j < nu; j += 32u) dst[j] = (unsigned long long)x | ((unsigned long long)j << 32);
    }
  }
  st.fill = st.out = 0;
  return queued;
}

// Improvements counted by a pull round: every warp's into the CTA's word,
// which thread 0 takes along to the team barrier.
__device__ __forceinline__ void fold_changes(uint32_t changed, uint32_t* s_changed, unsigned lane) {
  const uint32_t n = __reduce_add_sync(kFullMask, changed);
  if (lane == 0 && n) atomicAdd(s_changed, n);
}
__device__ __forceinline__ uint32_t take_changes(uint32_t* s_changed) {
  uint32_t n = 0;
  if (threadIdx.x == 0) {
    n = *s_changed;
    *s_changed = 0u;
  }
  return n;
}

}  // namespace svv
