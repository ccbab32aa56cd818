// svv_build.cpp -- host builder of the versioned union graph (Section 4.1):
// one edge per live edge instance, grouped by source, with a presence mask of
// ceil(S/64) words per edge (bit i = live in snapshot i).
//
// Every pass runs on several host threads.  A thread owns a range of sources:
// it reads the whole log and takes the instances of its range in log order, so
// rows keep instance order without locks, histograms or extra memory; reading
// the log once per thread costs less than one thread's scattered writes (4.2M
// instances: 60 ms on one thread).  The ranges of the writing pass hold equal
// numbers of edges, since low vertex ids carry most of an RMAT graph.
#include <cstdint>
#include <new>
#include <vector>

#include "../../include/svv.h"
#include "svv_threads.h"

// svv_build_versioned_csr, but for memory that runs out (std::bad_alloc)
static svv_status build_versioned_csr(uint32_t V, uint32_t S, uint64_t n_inst, const uint32_t* src,
                                      const uint32_t* dst, const uint32_t* w, const uint32_t* t_add,
                                      const uint32_t* t_del, uint64_t* row_ptr, uint32_t* col,
                                      uint32_t* weight, uint64_t* mask, uint64_t* E_out) {
  if (V == 0 || S == 0 || !row_ptr || !E_out) return SVV_EINVAL;
  if (n_inst && (!src || !dst || !w || !t_add || !t_del || !col || !weight || !mask)) return SVV_EINVAL;
  const uint32_t W = (S + 63) / 64;
  const unsigned nt = svv::host_threads(n_inst);
  std::vector<char> bad(nt, 0);
  svv::parallel(nt, [&](unsigned t) {
    for (uint64_t k = svv::part(n_inst, nt, t), hi = svv::part(n_inst, nt, t + 1); k < hi; ++k)
      if (src[k] >= V || dst[k] >= V || t_add[k] > S || t_del[k] > S) {
        bad[t] = 1;
        return;
      }
  });
  for (char b : bad)
    if (b) return SVV_EINVAL;
  // counts: row v's in row_ptr[v + 1]
  row_ptr[0] = 0;
  svv::parallel(nt, [&](unsigned t) {
    const uint64_t lo = svv::part(V, nt, t), hi = svv::part(V, nt, t + 1);
    for (uint64_t v = lo; v < hi; ++v) row_ptr[v + 1] = 0;
    for (uint64_t k = 0; k < n_inst; ++k)
      if (src[k] - lo < hi - lo && t_add[k] < t_del[k]) row_ptr[src[k] + 1]++;
  });
  for (uint32_t v = 0; v < V; ++v) row_ptr[v + 1] += row_ptr[v];
  std::vector<uint64_t> fill(row_ptr, row_ptr + V);
  svv::parallel(nt, [&](unsigned t) {
    const uint64_t lo = svv::row_at(row_ptr, V, nt, t), hi = svv::row_at(row_ptr, V, nt, t + 1);
    if (lo == hi) return;
    for (uint64_t k = 0; k < n_inst; ++k) {
      if (src[k] - lo >= hi - lo || t_add[k] >= t_del[k]) continue;
      const uint64_t p = fill[src[k]]++;
      col[p] = dst[k];
      weight[p] = w[k];
      uint64_t* m = mask + p * W;
      for (uint32_t j = 0; j < W; ++j) {
        // bits [t_add, t_del) restricted to word j
        const uint32_t b = t_add[k] > 64 * j ? t_add[k] : 64 * j;
        const uint32_t e = t_del[k] < 64 * j + 64 ? t_del[k] : 64 * j + 64;
        uint64_t x = 0;
        if (b < e) {
          const uint32_t n = e - b;
          x = (n == 64 ? ~0ull : ((1ull << n) - 1ull)) << (b - 64 * j);
        }
        m[j] = x;
      }
    }
  });
  *E_out = row_ptr[V];
  return SVV_OK;
}

extern "C" svv_status svv_build_versioned_csr(uint32_t V, uint32_t S, uint64_t n_inst, const uint32_t* src,
                                              const uint32_t* dst, const uint32_t* w, const uint32_t* t_add,
                                              const uint32_t* t_del, uint64_t* row_ptr, uint32_t* col,
                                              uint32_t* weight, uint64_t* mask, uint64_t* E_out) {
  try {
    return build_versioned_csr(V, S, n_inst, src, dst, w, t_add, t_del, row_ptr, col, weight, mask, E_out);
  } catch (const std::bad_alloc&) {
    return SVV_ENOMEM;
  }
}
