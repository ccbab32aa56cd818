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
constexpr uint32_t kSortBlocks = 128, kSortThreads = 1024;  // counters: 256 per block

enum : int { kMetaHubs = 0, kMetaOrd = 1, kMetaRows = 2, kMetaItems = 3, kMetaMaxW = 4, kMeta = 5 };

struct Degrees {
  const uint32_t* all;
  const uint32_t* less;  // subtracted when not null
  __device__ __forceinline__ uint32_t operator()(uint32_t v) const { return all[v] - (less ? less[v] : 0u); }
};

__device__ __forceinline__ uint32_t bin_of(uint32_t d) { return d > kHubDegree ? 0u : 1u + kHubDegree - d; }

__global__ void __launch_bounds__(256) degree_kernel(const uint2* cw, uint32_t n, uint32_t* deg) {
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x)
    atomicAdd(deg + cw[e].x, 1u);
}

__global__ void __launch_bounds__(256) hist_kernel(Degrees deg, uint32_t V, uint32_t* hist) {
  __shared__ uint32_t s[kBins];
  for (uint32_t b = threadIdx.x; b < kBins; b += blockDim.x) s[b] = 0u;
  __syncthreads();
  for (size_t v = blockIdx.x * (size_t)blockDim.x + threadIdx.x; v < V; v += (size_t)gridDim.x * blockDim.x) {
    const uint32_t d = deg((uint32_t)v);
    if (d) atomicAdd(s + bin_of(d), 1u);
  }
  __syncthreads();
  for (uint32_t b = threadIdx.x; b < kBins; b += blockDim.x)
    if (s[b]) atomicAdd(hist + b, s[b]);
}

// one thread: bin offsets (hubs counted apart from the sorted targets)
__global__ void binscan_kernel(const uint32_t* hist, uint32_t* off, unsigned long long* meta) {
  uint32_t sum = 0;
  off[0] = 0u;
  for (uint32_t b = 1; b < kBins; ++b) {
    off[b] = sum;
    sum += hist[b];
  }
  meta[kMetaHubs] = hist[0];
  meta[kMetaOrd] = sum;
}

// slice and lane of every target (lane 32: a hub's own slice), the targets of
// every slice, and the slice's number of steps
__global__ void __launch_bounds__(kRankBlock) rank_kernel(Degrees deg, uint32_t V, uint32_t nhub, uint32_t* off,
                                                          uint2* tpos, uint32_t* tgt, uint32_t* width) {
  __shared__ uint32_t s_cnt[kBins], s_base[kBins];
  const uint32_t v0 = blockIdx.x * kRankVerts;
  for (uint32_t b = threadIdx.x; b < kBins; b += blockDim.x) s_cnt[b] = 0u;
  __syncthreads();
  uint32_t d[kRankVerts / kRankBlock], r[kRankVerts / kRankBlock];
#pragma unroll
  for (uint32_t j = 0; j < kRankVerts / kRankBlock; ++j) {
    const size_t v = (size_t)v0 + j * kRankBlock + threadIdx.x;
    d[j] = v < V ? deg((uint32_t)v) : 0u;
    r[j] = d[j] ? atomicAdd(s_cnt + bin_of(d[j]), 1u) : 0u;
  }
  __syncthreads();
  for (uint32_t b = threadIdx.x; b < kBins; b += blockDim.x)
    if (s_cnt[b]) s_base[b] = atomicAdd(off + b, s_cnt[b]);
  __syncthreads();
#pragma unroll
  for (uint32_t j = 0; j < kRankVerts / kRankBlock; ++j) {
    if (!d[j]) continue;
    const uint32_t v = v0 + j * kRankBlock + threadIdx.x;
    const uint32_t b = bin_of(d[j]), k = s_base[b] + r[j];
    if (b == 0) {
      tpos[v] = make_uint2(k, 32u);
      for (uint32_t l = 0; l < 32u; ++l) tgt[(size_t)k * 32u + l] = v;
      width[k] = d[j] / 32u + (d[j] % 32u != 0u);
    } else {
      const uint32_t slice = nhub + (k >> 5);
      tpos[v] = make_uint2(slice, k & 31u);
      tgt[(size_t)slice * 32u + (k & 31u)] = v;
      atomicMax(width + slice, d[j]);
    }
  }
}

// one CTA: exclusive scan of the slices' steps; the items of hub slices come
// first, slice by slice, then the others by their place in the slice: segoff[j]
// is where the items that start at step j * kItemSteps begin
__global__ void __launch_bounds__(1024) slicescan_kernel(const uint32_t* width, uint32_t n, uint32_t nhub,
                                                         uint32_t* sbase, uint32_t* sitem, uint32_t* segoff,
                                                         unsigned long long* meta) {
  __shared__ uint32_t s_w[32], s_i[32], s_seg[kMaxSegs];
  const unsigned lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
  if (threadIdx.x < kMaxSegs) s_seg[threadIdx.x] = 0u;
  uint32_t cw = 0, ci = 0;  // totals so far, the same in every thread
  for (uint32_t s0 = 0; s0 < n; s0 += 1024u) {
    __syncthreads();
    const uint32_t s = s0 + threadIdx.x;
    const uint32_t w = s < n ? width[s] : 0u, it = s < nhub ? (w + kItemSteps - 1u) / kItemSteps : 0u;
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
      sbase[s] = bw + iw - w;
      sitem[s] = bi + ii - it;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    meta[kMetaRows] = cw;
    for (uint32_t j = 0; j < kMaxSegs; ++j) {
      segoff[j] = ci;
      ci += s_seg[j];
    }
    meta[kMetaItems] = ci;
  }
}

__global__ void __launch_bounds__(256) items_kernel(const uint32_t* width, uint32_t n, uint32_t nhub,
                                                    const uint32_t* sbase, const uint32_t* sitem,
                                                    const uint32_t* segoff, uint2* items) {
  const uint32_t s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  const uint32_t w = width[s], b = sbase[s];
  for (uint32_t k = 0, j = 0; k < w; k += kItemSteps, ++j)
    items[s < nhub ? sitem[s] + j : segoff[j] + (s - nhub)] =
        make_uint2(b + k, (s << 4) | (min(w - k, kItemSteps) - 1u));
}

// every slot starts as its target's self-loop (0 where a slice has no target)
__global__ void __launch_bounds__(256) pad_kernel(const uint2* items, uint32_t nitems, const uint32_t* tgt, uint2* cw) {
  const unsigned lane = threadIdx.x & 31u;
  const size_t nw = (size_t)gridDim.x * (blockDim.x >> 5);
  for (size_t i = (blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5; i < nitems; i += nw) {
    const uint2 d = items[i];
    const uint32_t t = tgt[(size_t)(d.y >> 4) * 32u + lane];
    for (uint32_t k = 0; k <= (d.y & 15u); ++k)
      cw[(size_t)(d.x + k) * 32u + lane] = make_uint2(t == kNone ? 0u : t, 0xFFFFFFFFu);
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
// (part == 0: edge = index in the forward rows) or the partial ones (index in
// their own list); and the largest weight
__global__ void __launch_bounds__(256) list_kernel(DevGraph g, int part, uint2* list, unsigned long long* meta) {
  const uint32_t n = part ? g.NF : g.E;
  uint32_t top = 0;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
    if (part) {
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
  if ((threadIdx.x & 31u) == 0 && top) atomicMax(meta + kMetaMaxW, (unsigned long long)top);
}

__global__ void __launch_bounds__(256) rekey_kernel(DevGraph g, int part, uint2* list, uint32_t n) {
  const uint2* cw = part ? g.nfcw : g.cw;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    list[i].x = cw[list[i].y].x;
}

// One pass of a stable radix sort by the 8 key bits at `shift`: digit counts
// per block (blocks take consecutive ranges), their exclusive scan in digit
// order, and the ordered move.
__device__ __forceinline__ void sort_range(uint32_t n, uint32_t& lo, uint32_t& hi) {
  const uint32_t per = n / gridDim.x + (n % gridDim.x != 0u);  // n may be close to 2^32
  lo = (uint32_t)min((unsigned long long)n, (unsigned long long)per * blockIdx.x);
  hi = (uint32_t)min((unsigned long long)n, (unsigned long long)per * blockIdx.x + per);
}

__global__ void __launch_bounds__(kSortThreads) sort_count_kernel(const uint2* in, uint32_t n, uint32_t shift,
                                                                  uint32_t* counts) {
  __shared__ uint32_t s[256];
  if (threadIdx.x < 256u) s[threadIdx.x] = 0u;
  __syncthreads();
  uint32_t lo, hi;
  sort_range(n, lo, hi);
  for (size_t i = lo + threadIdx.x; i < hi; i += kSortThreads) atomicAdd(s + ((in[i].x >> shift) & 255u), 1u);
  __syncthreads();
  if (threadIdx.x < 256u) counts[threadIdx.x * gridDim.x + blockIdx.x] = s[threadIdx.x];
}

__global__ void __launch_bounds__(1024) sort_scan_kernel(uint32_t* counts, uint32_t n) {
  __shared__ uint32_t s_w[32];
  const unsigned lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
  uint32_t total = 0;
  for (uint32_t i0 = 0; i0 < n; i0 += 1024u) {
    __syncthreads();
    const uint32_t i = i0 + threadIdx.x, c = i < n ? counts[i] : 0u;
    uint32_t inc = c;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t a = __shfl_up_sync(0xFFFFFFFFu, inc, o);
      if (lane >= (unsigned)o) inc += a;
    }
    if (lane == 31) s_w[wid] = inc;
    __syncthreads();
    uint32_t base = total;
    for (unsigned k = 0; k < 32u; ++k) {
      if (k < wid) base += s_w[k];
      total += s_w[k];
    }
    if (i < n) counts[i] = base + inc - c;
  }
}

__global__ void __launch_bounds__(kSortThreads) sort_move_kernel(const uint2* in, uint2* out, uint32_t n, uint32_t shift,
                                                                 const uint32_t* offsets) {
  __shared__ uint32_t s_base[256], s_cnt[kSortThreads / 32][256];
  const unsigned lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
  if (threadIdx.x < 256u) s_base[threadIdx.x] = offsets[threadIdx.x * gridDim.x + blockIdx.x];
  uint32_t lo, hi;
  sort_range(n, lo, hi);
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
__global__ void __launch_bounds__(256) start_kernel(const uint2* list, uint32_t n, uint32_t* start) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const uint32_t x = list[i].x;
    if (i == 0 || list[i - 1].x != x) start[x] = (uint32_t)i;
  }
}

__global__ void __launch_bounds__(256) fill_kernel(DevGraph g, int part, const uint2* list, uint32_t n,
                                                   const uint32_t* start, const uint2* tpos, const uint32_t* sbase,
                                                   uint2* out, uint64_t* mask) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const uint2 x = list[i];  // {target, edge}
    const uint2 tp = tpos[x.x];
    const uint32_t k = (uint32_t)i - start[x.x], b = sbase[tp.x];
    const size_t slot = tp.y == 32u ? (size_t)b * 32u + k : (size_t)(b + k) * 32u + tp.y;
    if (part) {
      out[slot] = make_uint2(g.nfsrc[x.y], g.nfcw[x.y].y);
      for (uint32_t j = 0; j < g.W; ++j) mask[slot * g.W + j] = g.nfmask[(size_t)x.y * g.W + j];
    } else {
      out[slot] = make_uint2(row_of(g, x.y), g.cw[x.y].y);
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

// row descriptors from the row offsets and the (host) prefix counts of partial edges
svv_status build_rowd(svv_ctx* c, const uint32_t* nfp, uint4* rowd) {
  const uint32_t V = c->g.V;
  uint32_t* tmp = reinterpret_cast<uint32_t*>(c->q0);  // more than 2V words
  cudaError_t e = cudaMemcpy(tmp, nfp, ((size_t)V + 1) * 4, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    rowd_kernel<<<blocks_for(V, 1024), 256>>>(c->g.rp, tmp, V, rowd);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(0);
  return e == cudaSuccess ? SVV_OK : cuda_fail(c, e, "building the row descriptors");
}

// Build both halves of the transposed graph (edges present in every snapshot;
// partial edges with their masks).  Runs on the legacy stream with the query
// scratch as working memory (svv_load owns the device at that point); only
// the layout itself is allocated.
svv_status build_pull(svv_ctx* c) {
  const DevGraph& g = c->g;
  const uint32_t V = g.V;
  cudaError_t e = cudaSuccess;
  uint32_t *deg = c->stamp, *deg_p = c->rI, *start = c->rU, *width = c->row, *sbase = c->uv;
  uint32_t* sitem = reinterpret_cast<uint32_t*>(c->q0);
  uint2* tpos = reinterpret_cast<uint2*>(c->qrow);
  unsigned long long* meta = reinterpret_cast<unsigned long long*>(c->part);
  uint32_t *hist = c->part + 2 * kMeta, *off = hist + kBins;
  uint32_t* segoff = off + kBins;
  static_assert(2 * kMeta + 2 * kBins + kMaxSegs == kLayoutWords, "part_words");
  uint32_t* counts = reinterpret_cast<uint32_t*>(c->ctl);  // cleared by every query
  static_assert(sizeof(TeamCtl) * kNumCtl >= 256 * kSortBlocks * sizeof(uint32_t), "sort counters");
  auto step = [&](cudaError_t r) {
    if (e == cudaSuccess) e = r;
  };
  auto fill_words = [&](void* p, int byte, size_t n) { step(cudaMemsetAsync(p, byte, n * 4, 0)); };
  fill_words(deg, 0, V);
  fill_words(deg_p, 0, V);
  if (g.E) degree_kernel<<<blocks_for(g.E, 1024), 256>>>(g.cw, g.E, deg);
  if (g.NF) degree_kernel<<<blocks_for(g.NF, 1024), 256>>>(g.nfcw, g.NF, deg_p);
  for (int part = 0; part < 2; ++part) {
    const Degrees d{part ? deg_p : deg, part ? nullptr : deg_p};
    const uint32_t n = part ? g.NF : g.E - g.NF;
    PullGraph& p = part ? c->g.pp : c->g.pf;
    unsigned long long m[kMeta] = {};
    fill_words(c->part, 0, 2 * kMeta + 2 * kBins + kMaxSegs);
    hist_kernel<<<blocks_for(V, 1024), 256>>>(d, V, hist);
    binscan_kernel<<<1, 1>>>(hist, off, meta);
    step(cudaGetLastError());
    step(cudaMemcpy(m, meta, 2 * sizeof(m[0]), cudaMemcpyDeviceToHost));
    if (e != cudaSuccess) return cuda_fail(c, e, "building the transposed graph");
    const uint32_t nhub = (uint32_t)m[kMetaHubs], ns = nhub + ceil_div(m[kMetaOrd], 32);
    uint32_t* d_tgt;
    svv_status st = alloc_n(c, c->graph_bufs, (uint64_t)ns * 32, &d_tgt);
    if (st) return st;
    fill_words(d_tgt, 0xFF, (size_t)ns * 32);
    fill_words(width, 0, std::max<uint32_t>(ns, 1));
    rank_kernel<<<ceil_div(V, kRankVerts), kRankBlock>>>(d, V, nhub, off, tpos, d_tgt, width);
    slicescan_kernel<<<1, 1024>>>(width, ns, nhub, sbase, sitem, segoff, meta);
    if (n) list_kernel<<<blocks_for(part ? g.NF : g.E, 1024), 256>>>(g, part, c->qcw, meta);
    step(cudaGetLastError());
    step(cudaMemcpy(m, meta, sizeof(m), cudaMemcpyDeviceToHost));
    if (e != cudaSuccess) return cuda_fail(c, e, "building the transposed graph");
    const uint32_t nitems = (uint32_t)m[kMetaItems];
    const uint64_t slots = m[kMetaRows] * 32;
    uint2 *d_items, *d_cw;
    uint64_t* d_mask = nullptr;
    if ((st = alloc_n(c, c->graph_bufs, nitems, &d_items)) || (st = alloc_n(c, c->graph_bufs, slots, &d_cw))) return st;
    if (part && (st = alloc_n(c, c->graph_bufs, slots * g.W, &d_mask))) return st;
    if (n) {
      // by weight, then by target (stable): 8 bits a pass, between the scratch
      // edge list and the layout's own array, which is filled afterwards
      uint2 *cur = c->qcw, *other = d_cw;
      const unsigned sb = std::max<uint32_t>(1, std::min<uint32_t>(kSortBlocks, ceil_div(n, 4096)));
      auto sort_by = [&](uint64_t top) {
        for (uint32_t shift = 0; shift < 32u && (top >> shift) != 0; shift += 8u) {
          sort_count_kernel<<<sb, kSortThreads>>>(cur, n, shift, counts);
          sort_scan_kernel<<<1, 1024>>>(counts, 256u * sb);
          sort_move_kernel<<<sb, kSortThreads>>>(cur, other, n, shift, counts);
          std::swap(cur, other);
        }
      };
      sort_by(m[kMetaMaxW]);
      rekey_kernel<<<blocks_for(n, 1024), 256>>>(g, part, cur, n);
      sort_by(V - 1u);
      if (cur != c->qcw) step(cudaMemcpyAsync(c->qcw, cur, (size_t)n * sizeof(uint2), cudaMemcpyDeviceToDevice, 0));
      items_kernel<<<ceil_div(ns, 256), 256>>>(width, ns, nhub, sbase, sitem, segoff, d_items);
      pad_kernel<<<blocks_for(nitems, 8), 256>>>(d_items, nitems, d_tgt, d_cw);
      if (part) step(cudaMemsetAsync(d_mask, 0, slots * g.W * 8, 0));
      start_kernel<<<blocks_for(n, 1024), 256>>>(c->qcw, n, start);
      fill_kernel<<<blocks_for(n, 256), 256>>>(g, part, c->qcw, n, start, tpos, sbase, d_cw, d_mask);
    }
    step(cudaGetLastError());
    p.items = d_items;
    p.tgt = d_tgt;
    p.cw = d_cw;
    p.nitems = nitems;
    p.nhub = nhub;
    p.slots = slots;
    if (part) c->g.ppmask = d_mask;
  }
  step(cudaStreamSynchronize(0));
  if (e != cudaSuccess) return cuda_fail(c, e, "building the transposed graph");
  c->g.pull = 1;
  return SVV_OK;
}

}  // namespace svv
