// svv_layout.cu -- the transposed graph of the pull rounds, built on the
// device from the resident forward graph when a graph is loaded.
//
// A pull round takes, for every vertex, the best candidate over its in-edges.
// The in-edges are laid out so that a lane owns a target and keeps its best
// candidate in a register: targets are sorted by in-degree, 32 of them form a
// slice, and step k of a slice holds the k-th in-edge of each of its targets
// side by side (32 x 8 bytes, one coalesced load).  Sorting makes the targets
// of a slice equally long, so the padding over the whole graph is at most
// 32 x kHubDegree slots plus 31 per hub.  A target with more than kHubDegree
// in-edges gets a slice of its own with its in-edges over all 32 lanes; the
// lanes' candidates are folded once per item.  Slices are cut into items of
// at most 16 steps (kItemSteps), which the warps of a pull round take in turn.
//
// A target's in-edges are sorted by weight, so that a lane can stop at the
// first edge that no source could make better than what it has (svv_pull.cuh).
// The items are ordered by their place in the slice -- every slice's first 16
// steps, then every slice's next 16 -- so that the later items of a long slice
// mostly find their targets already improved by its first ones, and stop at
// once.  Padding slots are self-loops of the largest weight: they improve no
// value in any of the four relaxations and sort last.
#include <algorithm>

#include "svv_ctx.h"

namespace svv {

namespace {

constexpr uint32_t kHubDegree = 512;
constexpr uint32_t kBins = kHubDegree + 1;  // bin 0: hubs; bin 1 + kHubDegree - d: in-degree d
constexpr uint32_t kRankBlock = 256, kRankVerts = 1024;

constexpr uint32_t kMaxSegs = kHubDegree / kItemSteps;  // items of the longest slice that is not a hub's
constexpr uint32_t kSortBlocks = 192, kSortThreads = 1024;  // of both halves; counters: 256 per block

enum : int { kMetaHubs = 0, kMetaOrd = 1, kMetaRows = 2, kMetaItems = 3, kMetaMaxW = 4, kMeta = 5 };

struct Degrees {
  const uint32_t* all;
  const uint32_t* less;  // subtracted when not null
  __device__ __forceinline__ uint32_t operator()(uint32_t v) const { return all[v] - (less ? less[v] : 0u); }
};

// One half of the layout under construction: the edges present in every
// snapshot (part 0) or the partial ones (part 1).  A launch covers both, by
// blockIdx.y: a small graph's load is a chain of launches of a few microseconds.
struct Half {
  Degrees deg;
  uint32_t n, nhub, ns, nitems;  // edges, hub slices, slices, items
  uint32_t sb;                   // blocks of a sort pass
  uint32_t *hist, *off, *segoff;
  unsigned long long* meta;
  uint32_t *width, *sbase, *sitem, *start, *tgt, *counts;
  uint2 *tpos, *items;
  uint2* buf[2];  // the list being sorted: scratch, and the layout's own slots, which are filled afterwards
  uint64_t* mask;
};
struct Halves {
  Half h[2];
};

__device__ __forceinline__ uint32_t bin_of(uint32_t d) { return d > kHubDegree ? 0u : 1u + kHubDegree - d; }

// exclusive prefix of x over a block of 1,024 threads, and the block's total
__device__ __forceinline__ uint32_t block_scan(uint32_t x, uint32_t& total) {
  __shared__ uint32_t s_w[32];
  const unsigned lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
  uint32_t incl = x;
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t a = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= (unsigned)o) incl += a;
  }
  if (lane == 31) s_w[wid] = incl;
  __syncthreads();
  uint32_t base = 0;
  total = 0;
  for (unsigned k = 0; k < 32u; ++k) {
    if (k < wid) base += s_w[k];
    total += s_w[k];
  }
  __syncthreads();
  return base + incl - x;
}

__global__ void __launch_bounds__(256) degree_kernel(DevGraph g, uint32_t* all, uint32_t* part) {
  const uint2* cw = blockIdx.y ? g.nfcw : g.cw;
  const uint32_t n = blockIdx.y ? g.NF : g.E;
  uint32_t* deg = blockIdx.y ? part : all;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x)
    atomicAdd(deg + cw[e].x, 1u);
}

__global__ void __launch_bounds__(256) hist_kernel(const __grid_constant__ Halves hs, uint32_t V) {
  const Half& h = hs.h[blockIdx.y];
  __shared__ uint32_t s[kBins];
  for (uint32_t b = threadIdx.x; b < kBins; b += blockDim.x) s[b] = 0u;
  __syncthreads();
  for (size_t v = blockIdx.x * (size_t)blockDim.x + threadIdx.x; v < V; v += (size_t)gridDim.x * blockDim.x) {
    const uint32_t d = h.deg((uint32_t)v);
    if (d) atomicAdd(s + bin_of(d), 1u);
  }
  __syncthreads();
  for (uint32_t b = threadIdx.x; b < kBins; b += blockDim.x)
    if (s[b]) atomicAdd(h.hist + b, s[b]);
}

// one CTA a half: bin offsets (hubs counted apart from the sorted targets)
__global__ void __launch_bounds__(1024) binscan_kernel(const __grid_constant__ Halves hs) {
  static_assert(kBins <= 1024u, "a thread per bin");
  const Half& h = hs.h[blockIdx.y];
  const uint32_t b = threadIdx.x;
  uint32_t total;
  const uint32_t at = block_scan(b && b < kBins ? h.hist[b] : 0u, total);
  if (b < kBins) h.off[b] = at;
  if (b == 0) {
    h.meta[kMetaHubs] = h.hist[0];
    h.meta[kMetaOrd] = total;
  }
}

// slice and lane of every target (lane 32: a hub's own slice), the targets of
// every slice, and the slice's number of steps
__global__ void __launch_bounds__(kRankBlock) rank_kernel(const __grid_constant__ Halves hs, uint32_t V) {
  const Half& h = hs.h[blockIdx.y];
  __shared__ uint32_t s_cnt[kBins], s_base[kBins];
  const uint32_t v0 = blockIdx.x * kRankVerts;
  for (uint32_t b = threadIdx.x; b < kBins; b += blockDim.x) s_cnt[b] = 0u;
  __syncthreads();
  uint32_t d[kRankVerts / kRankBlock], r[kRankVerts / kRankBlock];
#pragma unroll
  for (uint32_t j = 0; j < kRankVerts / kRankBlock; ++j) {
    const size_t v = (size_t)v0 + j * kRankBlock + threadIdx.x;
    d[j] = v < V ? h.deg((uint32_t)v) : 0u;
    r[j] = d[j] ? atomicAdd(s_cnt + bin_of(d[j]), 1u) : 0u;
  }
  __syncthreads();
  for (uint32_t b = threadIdx.x; b < kBins; b += blockDim.x)
    if (s_cnt[b]) s_base[b] = atomicAdd(h.off + b, s_cnt[b]);
  __syncthreads();
#pragma unroll
  for (uint32_t j = 0; j < kRankVerts / kRankBlock; ++j) {
    if (!d[j]) continue;
    const uint32_t v = v0 + j * kRankBlock + threadIdx.x;
    const uint32_t b = bin_of(d[j]), k = s_base[b] + r[j];
    if (b == 0) {
      h.tpos[v] = make_uint2(k, 32u);
      for (uint32_t l = 0; l < 32u; ++l) h.tgt[(size_t)k * 32u + l] = v;
      h.width[k] = d[j] / 32u + (d[j] % 32u != 0u);
    } else {
      const uint32_t slice = h.nhub + (k >> 5);
      h.tpos[v] = make_uint2(slice, k & 31u);
      h.tgt[(size_t)slice * 32u + (k & 31u)] = v;
      atomicMax(h.width + slice, d[j]);
    }
  }
}

// one CTA a half: exclusive scan of the slices' steps; the items of hub slices come
// first, slice by slice, then the others by their place in the slice: segoff[j]
// is where the items that start at step j * kItemSteps begin
__global__ void __launch_bounds__(1024) slicescan_kernel(const __grid_constant__ Halves hs) {
  const Half& h = hs.h[blockIdx.y];
  const uint32_t n = h.ns, nhub = h.nhub;
  __shared__ uint32_t s_w[32], s_i[32], s_seg[kMaxSegs];
  const unsigned lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
  if (threadIdx.x < kMaxSegs) s_seg[threadIdx.x] = 0u;
  uint32_t cw = 0, ci = 0;  // totals so far, the same in every thread
  for (uint32_t s0 = 0; s0 < n; s0 += 1024u) {
    __syncthreads();
    const uint32_t s = s0 + threadIdx.x;
    const uint32_t w = s < n ? h.width[s] : 0u, it = s < nhub ? (w + kItemSteps - 1u) / kItemSteps : 0u;
    if (s >= nhub)
      for (uint32_t j = 0; j * kItemSteps < w; ++j) atomicAdd(s_seg + j, 1u);
    uint32_t iw = w, ii = it;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t a = __shfl_up_sync(0xFFFFFFFFu, iw, o), b = __shfl_up_sync(0xFFFFFFFFu, ii, o);
      if (lane >= (unsigned)o) iw += a, ii += b;
    }
    if (lane == 31) s_w[wid] = iw, s_i[wid] = ii;
    __syncthreads();
    uint32_t bw = cw, bi = ci;
    for (unsigned k = 0; k < 32u; ++k) {
      if (k < wid) bw += s_w[k], bi += s_i[k];
      cw += s_w[k], ci += s_i[k];
    }
    if (s < n) {
      h.sbase[s] = bw + iw - w;
      h.sitem[s] = bi + ii - it;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    h.meta[kMetaRows] = cw;
    for (uint32_t j = 0; j < kMaxSegs; ++j) {
      h.segoff[j] = ci;
      ci += s_seg[j];
    }
    h.meta[kMetaItems] = ci;
  }
}

__global__ void __launch_bounds__(256) items_kernel(const __grid_constant__ Halves hs) {
  const Half& h = hs.h[blockIdx.y];
  const uint32_t s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= h.ns) return;
  const uint32_t w = h.width[s], b = h.sbase[s];
  for (uint32_t k = 0, j = 0; k < w; k += kItemSteps, ++j)
    h.items[s < h.nhub ? h.sitem[s] + j : h.segoff[j] + (s - h.nhub)] =
        make_uint2(b + k, (s << 4) | (min(w - k, kItemSteps) - 1u));
}

// every slot starts as its target's self-loop (0 where a slice has no target)
__global__ void __launch_bounds__(256) pad_kernel(const __grid_constant__ Halves hs) {
  const Half& h = hs.h[blockIdx.y];
  const unsigned lane = threadIdx.x & 31u;
  const size_t nw = (size_t)gridDim.x * (blockDim.x >> 5);
  for (size_t i = (blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5; i < h.nitems; i += nw) {
    const uint2 d = h.items[i];
    const uint32_t t = h.tgt[(size_t)(d.y >> 4) * 32u + lane];
    for (uint32_t k = 0; k <= (d.y & 15u); ++k)
      h.buf[1][(size_t)(d.x + k) * 32u + lane] = make_uint2(t == kNone ? 0u : t, 0xFFFFFFFFu);
  }
}

// row of edge e: rp[row] <= e < rp[row + 1]
__device__ __forceinline__ uint32_t row_of(const DevGraph& g, uint32_t e) {
  uint32_t lo = 0, hi = g.V;
  while (hi - lo > 1u) {
    const uint32_t mid = lo + (hi - lo) / 2u;
    if (g.rp[mid] <= e) lo = mid;
    else hi = mid;
  }
  return lo;
}

// the list to sort, {weight, edge}: the edges present in every snapshot
// (part 0: edge = index in the forward rows) or the partial ones (index in
// their own list); and the largest weight
__global__ void __launch_bounds__(256) list_kernel(DevGraph g, const __grid_constant__ Halves hs) {
  const Half& h = hs.h[blockIdx.y];
  const uint32_t n = blockIdx.y ? g.NF : g.E;
  uint2* list = h.buf[0];
  uint32_t top = 0;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
    if (blockIdx.y) {
      const uint32_t w = g.nfcw[e].y;
      list[e] = make_uint2(w, (uint32_t)e);
      top = max(top, w);
    } else {
      const uint4 rd = g.rowd[row_of(g, (uint32_t)e)];
      if (e >= rd.z) continue;
      const uint32_t w = g.cw[e].y;
      list[e - rd.w] = make_uint2(w, (uint32_t)e);
      top = max(top, w);
    }
  }
  top = __reduce_max_sync(0xFFFFFFFFu, top);
  if ((threadIdx.x & 31u) == 0 && top) atomicMax(h.meta + kMetaMaxW, (unsigned long long)top);
}

// the targets as keys, from buffer `from` to buffer `to` (or in place)
__global__ void __launch_bounds__(256) rekey_kernel(DevGraph g, const __grid_constant__ Halves hs, int from, int to) {
  const Half& h = hs.h[blockIdx.y];
  const uint2* cw = blockIdx.y ? g.nfcw : g.cw;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < h.n; i += (size_t)gridDim.x * blockDim.x) {
    const uint32_t e = h.buf[from][i].y;
    h.buf[to][i] = make_uint2(cw[e].x, e);
  }
}

// One pass of a stable radix sort by the 8 key bits at `shift`, from buffer
// `from` to the other: digit counts per block (blocks take consecutive ranges),
// their exclusive scan in digit order, and the ordered move.
__device__ __forceinline__ void sort_range(const Half& h, uint32_t& lo, uint32_t& hi) {
  const uint32_t n = h.n, per = n / h.sb + (n % h.sb != 0u);  // n may be close to 2^32
  lo = (uint32_t)min((unsigned long long)n, (unsigned long long)per * blockIdx.x);
  hi = (uint32_t)min((unsigned long long)n, (unsigned long long)per * blockIdx.x + per);
}

__global__ void __launch_bounds__(kSortThreads) sort_count_kernel(const __grid_constant__ Halves hs, int from,
                                                                  uint32_t shift) {
  const Half& h = hs.h[blockIdx.y];
  if (blockIdx.x >= h.sb) return;
  const uint2* in = h.buf[from];
  __shared__ uint32_t s[256];
  if (threadIdx.x < 256u) s[threadIdx.x] = 0u;
  __syncthreads();
  uint32_t lo, hi;
  sort_range(h, lo, hi);
  for (size_t i = lo + threadIdx.x; i < hi; i += kSortThreads) atomicAdd(s + ((in[i].x >> shift) & 255u), 1u);
  __syncthreads();
  if (threadIdx.x < 256u) h.counts[threadIdx.x * h.sb + blockIdx.x] = s[threadIdx.x];
}

__global__ void __launch_bounds__(1024) sort_scan_kernel(const __grid_constant__ Halves hs) {
  const Half& h = hs.h[blockIdx.y];
  uint32_t base = 0;
  for (uint32_t i0 = 0; i0 < 256u * h.sb; i0 += 1024u) {
    const uint32_t i = i0 + threadIdx.x, n = 256u * h.sb;
    uint32_t total;
    const uint32_t at = block_scan(i < n ? h.counts[i] : 0u, total);
    if (i < n) h.counts[i] = base + at;
    base += total;
  }
}

__global__ void __launch_bounds__(kSortThreads) sort_move_kernel(const __grid_constant__ Halves hs, int from,
                                                                 uint32_t shift) {
  const Half& h = hs.h[blockIdx.y];
  if (blockIdx.x >= h.sb) return;
  const uint2* in = h.buf[from];
  uint2* out = h.buf[from ^ 1];
  __shared__ uint32_t s_base[256], s_cnt[kSortThreads / 32][256];
  const unsigned lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
  if (threadIdx.x < 256u) s_base[threadIdx.x] = h.counts[threadIdx.x * h.sb + blockIdx.x];
  uint32_t lo, hi;
  sort_range(h, lo, hi);
  for (size_t i0 = lo; i0 < hi; i0 += kSortThreads) {
    for (uint32_t k = lane; k < 256u; k += 32u) s_cnt[wid][k] = 0u;
    __syncwarp();
    const size_t i = i0 + threadIdx.x;
    const bool in_range = i < hi;
    const uint2 x = in_range ? in[i] : make_uint2(0u, 0u);
    const uint32_t digit = (x.x >> shift) & 255u;
    const unsigned peers = __match_any_sync(0xFFFFFFFFu, in_range ? digit : 256u);
    const unsigned before = __popc(peers & ((1u << lane) - 1u));
    if (in_range && before == 0u) s_cnt[wid][digit] = __popc(peers);
    __syncthreads();
    if (threadIdx.x < 256u) {
      uint32_t run = s_base[threadIdx.x];
      for (unsigned w = 0; w < kSortThreads / 32; ++w) {
        const uint32_t c = s_cnt[w][threadIdx.x];
        s_cnt[w][threadIdx.x] = run;
        run += c;
      }
      s_base[threadIdx.x] = run;
    }
    __syncthreads();
    if (in_range) out[s_cnt[wid][digit] + before] = x;
    __syncthreads();
  }
}

// where each target's edges begin in the sorted list
__global__ void __launch_bounds__(256) start_kernel(const __grid_constant__ Halves hs) {
  const Half& h = hs.h[blockIdx.y];
  const uint2* list = h.buf[0];
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < h.n; i += (size_t)gridDim.x * blockDim.x) {
    const uint32_t x = list[i].x;
    if (i == 0 || list[i - 1].x != x) h.start[x] = (uint32_t)i;
  }
}

__global__ void __launch_bounds__(256) fill_kernel(DevGraph g, const __grid_constant__ Halves hs) {
  const Half& h = hs.h[blockIdx.y];
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < h.n; i += (size_t)gridDim.x * blockDim.x) {
    const uint2 x = h.buf[0][i];  // {target, edge}
    const uint2 tp = h.tpos[x.x];
    const uint32_t k = (uint32_t)i - h.start[x.x], b = h.sbase[tp.x];
    const size_t slot = tp.y == 32u ? (size_t)b * 32u + k : (size_t)(b + k) * 32u + tp.y;
    if (blockIdx.y) {
      h.buf[1][slot] = make_uint2(g.nfsrc[x.y], g.nfcw[x.y].y);
      for (uint32_t j = 0; j < g.W; ++j) h.mask[slot * g.W + j] = g.nfmask[(size_t)x.y * g.W + j];
    } else {
      h.buf[1][slot] = make_uint2(row_of(g, x.y), g.cw[x.y].y);
    }
  }
}

unsigned blocks_for(uint64_t n, unsigned per) {
  return (unsigned)std::max<uint64_t>(1, std::min<uint64_t>((n + per - 1) / per, 152u * 16u));
}

}  // namespace

__global__ void __launch_bounds__(256) rowd_kernel(const uint32_t* rp, const uint32_t* nfp, uint32_t V, uint4* rowd) {
  for (size_t v = blockIdx.x * (size_t)blockDim.x + threadIdx.x; v < V; v += (size_t)gridDim.x * blockDim.x)
    rowd[v] = make_uint4(rp[v], rp[v + 1], rp[v + 1] - (nfp[v + 1] - nfp[v]), nfp[v]);
}

// row descriptors from the row offsets and the (host) prefix counts of partial
// edges, queued on the legacy stream
svv_status build_rowd(svv_ctx* c, const uint32_t* nfp, uint4* rowd) {
  const uint32_t V = c->g.V;
  uint32_t* tmp = reinterpret_cast<uint32_t*>(c->q0);  // more than 2V words
  cudaError_t e = cudaMemcpy(tmp, nfp, ((size_t)V + 1) * 4, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    rowd_kernel<<<blocks_for(V, 1024), 256>>>(c->g.rp, tmp, V, rowd);
    e = cudaGetLastError();
  }
  return e == cudaSuccess ? SVV_OK : cuda_fail(c, e, "building the row descriptors");
}

// Build both halves of the transposed graph (edges present in every snapshot;
// partial edges with their masks).  Runs on the legacy stream with the query
// scratch as working memory (svv_load owns the device at that point); only
// the layout itself is allocated.  Two copies to the host give the sizes; one
// launch per step for both halves, since a small graph's load is bound by the
// chain of launches (16 vertices, 64 edges: svv_load 0.57 -> 0.33 ms; 4,096 and
// 32,768: 0.84 -> 0.60, few allocations included).
svv_status build_pull(svv_ctx* c) {
  const DevGraph& g = c->g;
  const uint32_t V = g.V;
  cudaError_t e = cudaSuccess;
  auto step = [&](cudaError_t r) {
    if (e == cudaSuccess) e = r;
  };
  auto fill_words = [&](void* p, int byte, size_t n) { step(cudaMemsetAsync(p, byte, n * 4, 0)); };
  uint32_t *deg = c->stamp, *deg_p = c->rI;
  uint32_t *w0 = reinterpret_cast<uint32_t*>(c->q0), *w1 = reinterpret_cast<uint32_t*>(c->q1);  // more than 2V words each
  uint2* pos = reinterpret_cast<uint2*>(c->qrow);                                               // 2V
  unsigned long long* meta = reinterpret_cast<unsigned long long*>(c->part);
  uint32_t* counters = c->part + 2 * 2 * kMeta;
  static_assert(2 * (2 * kMeta + 2 * kBins + kMaxSegs) == kLayoutWords, "part_words");
  static_assert(sizeof(TeamCtl) * kNumCtl >= 256 * kSortBlocks * sizeof(uint32_t), "sort counters");
  Halves hs{};
  Half &f = hs.h[0], &p = hs.h[1];
  f.n = g.E - g.NF;
  p.n = g.NF;
  f.deg = Degrees{deg, deg_p};
  p.deg = Degrees{deg_p, nullptr};
  f.width = c->row, f.sbase = c->uv, f.sitem = w0, f.start = c->rU, f.tpos = pos;
  p.width = w0 + V, p.sbase = w1, p.sitem = w1 + V, p.start = c->procv, p.tpos = pos + V;
  f.buf[0] = c->qcw;
  p.buf[0] = c->qcw + f.n;
  for (int i = 0; i < 2; ++i) {
    Half& h = hs.h[i];
    h.meta = meta + i * kMeta;
    h.hist = counters + i * (2 * kBins + kMaxSegs);
    h.off = h.hist + kBins;
    h.segoff = h.off + kBins;
    // at least 1,024 edges a block, and the counters shared by the halves' sizes
    h.sb = h.n ? std::max<uint32_t>(1, std::min<uint32_t>(ceil_div(h.n, kSortThreads),
                                                          (uint32_t)((kSortBlocks - 1ull) * h.n / g.E)))
               : 0u;
  }
  f.counts = reinterpret_cast<uint32_t*>(c->ctl);  // cleared by every query
  p.counts = f.counts + 256 * f.sb;
  unsigned long long m[2][kMeta] = {};
  auto sizes = [&]() {
    step(cudaGetLastError());
    if (e == cudaSuccess) step(cudaMemcpy(m, meta, sizeof(m), cudaMemcpyDeviceToHost));
    return e;
  };
  auto both = [](unsigned x) { return dim3(x, 2); };
  fill_words(deg, 0, V);
  fill_words(deg_p, 0, V);
  fill_words(c->part, 0, kLayoutWords);
  degree_kernel<<<both(blocks_for(g.E, 1024)), 256>>>(g, deg, deg_p);
  hist_kernel<<<both(blocks_for(V, 1024)), 256>>>(hs, V);
  binscan_kernel<<<both(1), 1024>>>(hs);
  if (sizes() != cudaSuccess) return cuda_fail(c, e, "building the transposed graph");
  for (int i = 0; i < 2; ++i) {
    hs.h[i].nhub = (uint32_t)m[i][kMetaHubs];
    hs.h[i].ns = hs.h[i].nhub + ceil_div(m[i][kMetaOrd], 32);
  }
  svv_status st;
  uint32_t* d_tgt;
  const uint64_t ntgt = ((uint64_t)f.ns + p.ns) * 32;
  if ((st = alloc_n(c, c->graph_bufs, ntgt, &d_tgt))) return st;
  f.tgt = d_tgt;
  p.tgt = d_tgt + (uint64_t)f.ns * 32;
  fill_words(d_tgt, 0xFF, ntgt);
  fill_words(f.width, 0, f.ns);
  fill_words(p.width, 0, p.ns);
  rank_kernel<<<both(ceil_div(V, kRankVerts)), kRankBlock>>>(hs, V);
  slicescan_kernel<<<both(1), 1024>>>(hs);
  list_kernel<<<both(blocks_for(g.E, 1024)), 256>>>(g, hs);
  if (sizes() != cudaSuccess) return cuda_fail(c, e, "building the transposed graph");
  uint64_t slots[2];
  Arrays out;
  for (int i = 0; i < 2; ++i) {
    hs.h[i].nitems = (uint32_t)m[i][kMetaItems];
    slots[i] = m[i][kMetaRows] * 32;
    out.add(hs.h[i].nitems, &hs.h[i].items).add(slots[i], &hs.h[i].buf[1]);
  }
  if ((st = out.add(slots[1] * g.W, &p.mask).alloc(c, c->graph_bufs))) return st;
  if (g.E) {
    // by weight, then by target (stable): 8 bits a pass, between the scratch
    // list and the layout's slots, which are filled afterwards
    const unsigned sb = std::max(f.sb, p.sb);
    int at = 0;  // the buffer that holds the list
    auto sort_by = [&](uint64_t top) {
      for (uint32_t shift = 0; shift < 32u && (top >> shift) != 0; shift += 8u, at ^= 1) {
        sort_count_kernel<<<both(sb), kSortThreads>>>(hs, at, shift);
        sort_scan_kernel<<<both(1), 1024>>>(hs);
        sort_move_kernel<<<both(sb), kSortThreads>>>(hs, at, shift);
      }
    };
    sort_by(std::max(m[0][kMetaMaxW], m[1][kMetaMaxW]));
    int left = 0;  // passes by target: the last one has to end in the scratch list
    for (uint32_t shift = 0; shift < 32u && ((V - 1u) >> shift) != 0; shift += 8u) ++left;
    rekey_kernel<<<both(blocks_for(g.E, 1024)), 256>>>(g, hs, at, left & 1);
    at = left & 1;
    sort_by(V - 1u);
    items_kernel<<<both(ceil_div(std::max(f.ns, p.ns), 256)), 256>>>(hs);
    pad_kernel<<<both(blocks_for(std::max(f.nitems, p.nitems), 8)), 256>>>(hs);
    fill_words(p.mask, 0, slots[1] * g.W * 2);
    start_kernel<<<both(blocks_for(g.E, 1024)), 256>>>(hs);
    fill_kernel<<<both(blocks_for(g.E, 256)), 256>>>(g, hs);
  }
  step(cudaGetLastError());
  if (e != cudaSuccess) return cuda_fail(c, e, "building the transposed graph");
  for (int i = 0; i < 2; ++i) {
    const Half& h = hs.h[i];
    (i ? c->g.pp : c->g.pf) = PullGraph{h.items, h.tgt, h.buf[1], h.nitems, h.nhub, slots[i]};
  }
  c->g.ppmask = p.mask;
  c->g.pull = 1;
  return SVV_OK;
}

}  // namespace svv
