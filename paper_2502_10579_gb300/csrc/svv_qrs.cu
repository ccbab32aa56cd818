// svv_qrs.cu -- stable-vertex compaction and Q-relevant subgraph extraction.
//
// Section 3 Step 2 (Theorem 2): v is stable iff its intersection-graph and
// union-graph values agree; Algorithm 1 collects those into `found`.
// Section 3 Steps 3-4 and Algorithm 1 RemoveIncomingEdges /
// RemoveDeltaAdditionBatches: the in-edges of stable vertices, and the
// additions whose sink is stable, are dropped.  As Section 6.2 does, the
// subgraph is built "in reverse": only in-edges of unstable vertices are
// gathered.  Stable sources keep no rows: their value is final, so their edges
// into unstable vertices only matter once, in the seeding pass of the
// relaxation (which reads the addition edges directly).  The kept edges are
// those whose source and target are both unstable and that are present in at
// least one window snapshot; per row, edges present in every window snapshot
// come first (Section 4.1).  The rest, with masks rebased so that bit i is
// snapshot win_begin+i, fill the row's room from its end.
//
// One cooperative launch, three phases separated by the team barrier:
//   P1 per-CTA counts of unstable vertices, their work units and out-edges;
//   P2 rows in vertex order (CTA offsets from P1), row -> vertex map, units,
//      and each row's place in the edge arrays, with room for all its out-edges;
//   P3 fill: the kept edges of every unit next to those its row already holds.
// The edges are walked once.  Counting the kept edges first, to pack the rows,
// walked them twice, at one CTA per SM (114 registers): 121 us instead of 79 at
// scale 20 with 111K unstable vertices, 458 instead of 311 with 533K.  Two CTAs
// per SM at 64 registers; three (40, with spills) took 85 and 353 us.  Bound by
// the walk's chain of dependent loads (unit, row, target, row map) and its
// returning atomics.
#include "svv_qrs.cuh"

namespace svv {

constexpr int kQrsThreads = 512;

__global__ void __launch_bounds__(kQrsThreads, 2) qrs_kernel(QrsArgs a) {
  __shared__ TeamBar s_bar;
  const Team t{a.ctl, a.qerr, gridDim.x, blockIdx.x, a.spin_ns, &s_bar};
  t.begin();
  qrs_team(a, t);
}

cudaError_t launch_qrs(const QrsArgs& a, LaunchCfg cfg, cudaStream_t s) {
  QrsArgs copy = a;
  void* args[] = {&copy};
  return cudaLaunchCooperativeKernel((const void*)qrs_kernel, dim3(cfg.blocks), dim3(cfg.threads),
                                     args, 0, s);
}

int occupancy_qrs(int threads) {
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, (const void*)qrs_kernel, threads, 0) !=
      cudaSuccess)
    return 0;
  return n;
}

}  // namespace svv
