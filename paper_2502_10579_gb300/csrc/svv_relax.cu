// svv_relax.cu -- concurrent relaxation of every window snapshot over the
// Q-relevant subgraph (Section 4.2, Algorithm 2), and the output scatter.
//
// Values are kept vertex-major: row r of `val` holds the LP values of unstable
// vertex uv[r], one per snapshot of the slab, so one out-edge of a frontier
// vertex touches one contiguous run of the target's values.  A group of P
// lanes owns one work unit (row, chunk of edges); lane gl of the group holds
// snapshots gl, gl+P, ... (K of them).  The group loads P edges at once, then
// broadcasts them one by one; each lane relaxes its snapshots whose bit is set
// in the edge's mask (edge ownership, Section 4.2).  The frontier is
// snapshot-oblivious: a row is queued once per round if any of its snapshots
// improved.
//
// Round 0 initialises every row to the intersection-graph value (Algorithm 2
// "R_i = R_QRS") and seeds from the addition edges whose sink is unstable
// (Algorithm 2 addition batches; Section 3 Step 4 drops those with a stable
// sink).  The seeding reads the resident list of edges that are not present in
// all snapshots; an edge present in every window snapshot belongs to the
// intersection graph, whose values are already a fixed point on it, so it is
// skipped.  Sources of seed edges hold their intersection-graph value in every
// snapshot at that point.
#include <algorithm>

#include "svv_relax.cuh"

namespace svv {

constexpr int kRelaxThreads = kStageThreads;

template <class Op, int P, int K>
__global__ void __launch_bounds__(kRelaxThreads, 2) relax_kernel(const __grid_constant__ RelaxArgs a) {
  __shared__ StageMem s_stage;
  __shared__ TeamBar s_bar;
  const Team t{a.ctl, a.qerr, gridDim.x, blockIdx.x, a.spin_ns, &s_bar};
  t.begin();
  relax_team<Op, P, K>(a, t, &s_stage);
}

// ---------------------------------------------------------------------------
// Output scatter: out[(s0+i)*V + v] = intersection value if v is stable, else
// the relaxed value of its row.  A CTA writes a tile of kTV vertices x ls
// snapshots.  The rows of the tile's unstable vertices are copied to shared
// memory by 16-byte asynchronous copies, all of them in flight at once; the
// 16-byte granule g of vertex t's row lands at g ^ (t / 4), so that a warp that
// reads 8 groups of four vertices at 4 consecutive snapshots meets every bank
// once.  A thread keeps its four vertices' intersection values in registers
// and writes 16 bytes per snapshot (streaming stores: this query does not read
// the output again); stable vertices touch shared memory nowhere.
// Bound by the output's bytes: at 1M vertices x 64 snapshots (268 MB, 40 us as
// a plain fill) 59 us with 10% of the vertices unstable and 70 us with half of
// them (68 and 98 when every value went through shared memory).  When V is no
// multiple of 4 the rows start at any word, and a thread writes one word at a
// time: aligned groups of four that shift with the row were no faster (37 us
// for 92 MB either way).
constexpr int kTV = 128;
constexpr int kScatterThreads = 256;

__device__ __forceinline__ void copy16_async(uint32_t* smem, const uint32_t* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
               :
               : "r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem)
               : "memory");
}

__global__ void __launch_bounds__(kScatterThreads) scatter_kernel(ScatterArgs a) {
  extern __shared__ __align__(16) uint32_t tile[];  // [kTV][LP], granules swizzled
  __shared__ __align__(16) uint32_t s_row[kTV];
  __shared__ __align__(16) uint32_t s_x[kTV];
  if (*a.qerr != 0u) return;
  const uint32_t lps = __ffs(a.LP) - 1, gmask = (a.LP >> 2) - 1u;
  const bool vec = (a.V & 3u) == 0u && ((uintptr_t)a.out & 15u) == 0u;
  const uint32_t v0 = blockIdx.x * kTV;  // one tile per CTA
  const uint32_t nv = min((uint32_t)kTV, a.V - v0);
  bool mine = false;
  if (threadIdx.x < kTV) {
    const uint32_t t = threadIdx.x;
    const uint32_t r = t < nv ? a.row[v0 + t] : kNone;
    s_row[t] = r;
    s_x[t] = t < nv ? a.rI[v0 + t] : 0u;
    mine = r != kNone;
  }
  if (__syncthreads_or(mine)) {
    // a granule per thread and step: consecutive threads copy one row's
    const uint32_t ng = (a.ls + 3u) >> 2;
    for (uint32_t k = threadIdx.x; k < (uint32_t)kTV << (lps - 2u); k += kScatterThreads) {
      const uint32_t t = k >> (lps - 2u), g = k & gmask, r = s_row[t];
      if (r != kNone && g < ng)
        copy16_async(tile + (t << lps) + ((g ^ ((t >> 2) & gmask)) << 2), a.val + ((size_t)r << lps) + (g << 2));
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
  }
  auto value = [&](uint32_t t, uint32_t i) {
    return tile[(t << lps) + (((i >> 2) ^ ((t >> 2) & gmask)) << 2) + (i & 3u)] ^ a.rflip;
  };
  if (vec && nv == (uint32_t)kTV) {
    // lane = (group of four vertices, snapshot): 8 groups x 4 snapshots a
    // warp, 4 warps across the tile, so a store covers 4 rows of 128 bytes
    const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
    const uint32_t q = (wid & 3u) * 8u + (lane & 7u), i0 = (wid >> 2) * 4u + (lane >> 3);
    const uint4 r = *reinterpret_cast<const uint4*>(s_row + 4u * q), x = *reinterpret_cast<const uint4*>(s_x + 4u * q);
    uint4* o = reinterpret_cast<uint4*>(a.out + (size_t)(a.s0 + i0) * a.V + v0) + q;
    const size_t step = (size_t)(kScatterThreads / 32) * a.V / 4u;  // 8 snapshots on, in 16-byte words
    const bool stable = (r.x & r.y & r.z & r.w) == kNone;
    for (uint32_t i = i0; i < a.ls; i += kScatterThreads / 32u, o += step) {
      uint4 w = x;
      if (!stable) {
        if (r.x != kNone) w.x = value(4u * q, i);
        if (r.y != kNone) w.y = value(4u * q + 1u, i);
        if (r.z != kNone) w.z = value(4u * q + 2u, i);
        if (r.w != kNone) w.w = value(4u * q + 3u, i);
      }
      __stcs(o, w);
    }
  } else {
    const uint32_t t = threadIdx.x & (kTV - 1u), r = s_row[t], x = s_x[t];
    if (t < nv)
      for (uint32_t i = threadIdx.x / kTV; i < a.ls; i += kScatterThreads / kTV)
        __stcs(a.out + (size_t)(a.s0 + i) * a.V + v0 + t, r == kNone ? x : value(t, i));
  }
}

// Compact output: copy slab columns [s0, s0+ls) of the U relaxed rows into the
// caller's U x wl array.
__global__ void __launch_bounds__(256) compact_kernel(CompactArgs a) {
  if (*a.qerr != 0u) return;
  const uint32_t U = a.counts[0];
  if ((unsigned long long)U * a.wl > a.rows_cap) {
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicCAS(a.qerr, 0u, 2u);  // 2 = SVV_ENOMEM
    return;
  }
  const uint32_t lps = __ffs(a.LP) - 1;
  const unsigned long long n = (unsigned long long)U * a.ls;
  for (unsigned long long k = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; k < n;
       k += (unsigned long long)gridDim.x * blockDim.x) {
    const uint32_t r = (uint32_t)(k / a.ls), i = (uint32_t)(k % a.ls);
    a.rows_out[(size_t)r * a.wl + a.s0 + i] = a.val[((size_t)r << lps) + i];
  }
}

// The result of a query from a source with no out-edge, written at the
// output's bandwidth: 16-byte streaming stores when V is a multiple of 4.
//
// A thread keeps its columns and goes down the rows: no division per store, and
// the value never changes.  With fewer columns than threads, as many rows are
// written side by side as the threads cover; one thread going down every row of
// a column took 90 us for 1,000 vertices x 1,000 snapshots (30 now, the call's latency).
template <class T, class Value, class Store>
__device__ __forceinline__ void fill_rows(T* out, size_t cols, uint32_t L, Value value, Store store) {
  const size_t nthreads = (size_t)gridDim.x * blockDim.x;
  const size_t tid = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const size_t side = nthreads > cols ? nthreads / cols : 1u;  // rows side by side
  const size_t r0 = tid / cols;
  if (r0 >= side || r0 >= L) return;
  const size_t step = side * cols;
  const uint32_t rows = (uint32_t)((L - 1u - r0) / side + 1u);
  for (size_t k = tid - r0 * cols; k < cols; k += nthreads) {
    const T x = value(k);
    T* p = out + r0 * cols + k;
    for (uint32_t n = rows; n != 0u; --n, p += step) store(p, x);
  }
}

__global__ void __launch_bounds__(256) isolated_kernel(IsolatedArgs a) {
  const size_t nthreads = (size_t)gridDim.x * blockDim.x;
  const size_t tid = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (size_t v = tid; v < a.V; v += nthreads) {
    const uint32_t x = v == a.source ? a.src_val : a.ident;
    a.rI[v] = x;
    a.rU[v] = x;
    a.row[v] = kNone;
  }
  if (!a.out) return;
  auto at = [&](uint32_t v) { return v == a.source ? a.src_val : a.ident; };
  if ((a.V & 3u) == 0u && ((uintptr_t)a.out & 15u) == 0u) {
    fill_rows(
        reinterpret_cast<uint4*>(a.out), a.V >> 2, a.L,
        [&](size_t k) {
          const uint32_t v = (uint32_t)k * 4u;
          return make_uint4(at(v), at(v + 1u), at(v + 2u), at(v + 3u));
        },
        [](uint4* p, uint4 x) { __stcs(p, x); });
  } else {
    fill_rows(
        a.out, a.V, a.L, [&](size_t v) { return at((uint32_t)v); }, [](uint32_t* p, uint32_t x) { *p = x; });
  }
}

cudaError_t launch_isolated(const IsolatedArgs& a, cudaStream_t s) {
  isolated_kernel<<<std::max<uint32_t>(1, a.sms) * 8u, 256, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_compact(const CompactArgs& a, cudaStream_t s) {
  compact_kernel<<<1216, 256, 0, s>>>(a);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
template <class Op, int P, int K>
static cudaError_t launch_r(const RelaxArgs& a, LaunchCfg cfg, cudaStream_t s) {
  RelaxArgs copy = a;
  void* args[] = {&copy};
  return cudaLaunchCooperativeKernel((const void*)relax_kernel<Op, P, K>, dim3(cfg.blocks),
                                     dim3(cfg.threads), args, 0, s);
}

template <class Op>
static cudaError_t launch_pk(uint32_t P, uint32_t K, const RelaxArgs& a, LaunchCfg cfg, cudaStream_t s) {
  switch (P * 100 + K) {
    case 801: return launch_r<Op, 8, 1>(a, cfg, s);
    case 802: return launch_r<Op, 8, 2>(a, cfg, s);
    case 804: return launch_r<Op, 8, 4>(a, cfg, s);
    case 808: return launch_r<Op, 8, 8>(a, cfg, s);
    case 1601: return launch_r<Op, 16, 1>(a, cfg, s);
    case 1602: return launch_r<Op, 16, 2>(a, cfg, s);
    case 1604: return launch_r<Op, 16, 4>(a, cfg, s);
    case 1608: return launch_r<Op, 16, 8>(a, cfg, s);
    case 3201: return launch_r<Op, 32, 1>(a, cfg, s);
    case 3202: return launch_r<Op, 32, 2>(a, cfg, s);
    case 3204: return launch_r<Op, 32, 4>(a, cfg, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_relax(int type, uint32_t P, uint32_t K, const RelaxArgs& a, LaunchCfg cfg,
                         cudaStream_t s) {
  switch (type) {
    case 0: return launch_pk<OpSSSP>(P, K, a, cfg, s);
    case 1: return launch_pk<OpSSWP>(P, K, a, cfg, s);
    case 3: return launch_pk<OpSSNP>(P, K, a, cfg, s);
    case kTypeMixed: return launch_pk<OpMixed>(P, K, a, cfg, s);
    default: return launch_pk<OpBFS>(P, K, a, cfg, s);
  }
}

cudaError_t launch_scatter(const ScatterArgs& a, cudaStream_t s) {
  const uint32_t blocks = (a.V + kTV - 1) / kTV;  // one tile per CTA
  const size_t smem = (size_t)a.LP * kTV * sizeof(uint32_t);  // up to 64 KB for 128 snapshots
  if (smem > 40 * 1024) {  // with the static row map, past what needs no opt-in
    cudaError_t e = cudaFuncSetAttribute((const void*)scatter_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
  }
  scatter_kernel<<<blocks, kScatterThreads, smem, s>>>(a);
  return cudaGetLastError();
}

template <class Op>
static int occ_op(int threads) {
  const void* ks[] = {(const void*)relax_kernel<Op, 8, 1>,  (const void*)relax_kernel<Op, 8, 2>,
                      (const void*)relax_kernel<Op, 8, 4>,  (const void*)relax_kernel<Op, 8, 8>,
                      (const void*)relax_kernel<Op, 16, 1>, (const void*)relax_kernel<Op, 16, 2>,
                      (const void*)relax_kernel<Op, 16, 4>, (const void*)relax_kernel<Op, 16, 8>,
                      (const void*)relax_kernel<Op, 32, 1>, (const void*)relax_kernel<Op, 32, 2>,
                      (const void*)relax_kernel<Op, 32, 4>};
  int best = 1 << 30;
  for (const void* k : ks) {
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, threads, 0) != cudaSuccess) return 0;
    best = n < best ? n : best;
  }
  return best;
}

int occupancy_relax(int threads) {
  int a = occ_op<OpSSSP>(threads), b = occ_op<OpSSWP>(threads), c = occ_op<OpBFS>(threads);
  int d = occ_op<OpSSNP>(threads), e = occ_op<OpMixed>(threads);
  int m = a < b ? a : b;
  m = m < c ? m : c;
  m = m < d ? m : d;
  return m < e ? m : e;
}

}  // namespace svv
