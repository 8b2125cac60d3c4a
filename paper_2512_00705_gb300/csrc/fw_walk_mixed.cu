// fw_walk_mixed.cu -- launches over tables of several jobs.
//
// A table of up to 64 jobs is split by algorithm.  The jobs of one
// algorithm form one walker queue (one concatenated index space) walked by
// one persistent launch of the walk kernel compiled for that algorithm, so
// jobs of very different sizes and lengths still share the GPU.  A single
// kernel that reads the algorithm per job, or that switches between
// algorithm-specialised loops, keeps every algorithm's state live and spills:
// its node2vec steps measured twice as slow as the specialised kernel's.
// The per-algorithm launches run one after another on the caller's stream,
// or side by side on helper streams when the caller provides them (the batch
// plans do, inside their CUDA graph), so that one launch's last walkers share
// the GPU with the next launch's first ones.
#include "fw_internal.h"
#include "fw_walk.cuh"

namespace fw {
const WalkLaunches& table_weighted();
const WalkLaunches& table_node2vec();
const WalkLaunches& table_metapath();
const WalkLaunches& table_pagerank2();

const WalkLaunches& table_launches(int algo) {
  switch (algo) {
    case ALGO_WEIGHTED: return table_weighted();
    case ALGO_NODE2VEC: return table_node2vec();
    case ALGO_METAPATH: return table_metapath();
    default: return table_pagerank2();
  }
}

cudaError_t prime_walk_mixed_occupancy() {
  cudaError_t e = cudaSuccess;
  for (int a = 0; a < kAlgos && e == cudaSuccess; ++a) e = table_launches(a).prime();
  return e;
}

cudaError_t launch_walk_mixed(const fw_graph* g, const Job* jobs, int njobs, bool count, int beside,
                              unsigned long long* qctr, cudaStream_t stream, const cudaStream_t* side, cudaEvent_t* ev) {
  if (njobs < 1 || njobs > kMaxJobs) return cudaErrorInvalidValue;
  Job grp[kMaxJobs];
  int present[kAlgos], np = 0;
  long long totals[kAlgos];
  int firsts[kAlgos], counts[kAlgos];
  int m = 0;
  for (int a = 0; a < kAlgos; ++a) {
    firsts[a] = m;
    totals[a] = 0;
    for (int i = 0; i < njobs; ++i) {
      if (jobs[i].algo != a) continue;
      grp[m] = jobs[i];
      grp[m].gbase = totals[a];  // index space of the algorithm's queue
      totals[a] += jobs[i].num_walkers;
      ++m;
    }
    counts[a] = m - firsts[a];
    if (totals[a] > 0) present[np++] = a;
  }
  if (m != njobs) return cudaErrorInvalidValue;  // an algorithm outside 0..kAlgos-1
  const bool fork = side && ev && np > 1;
  cudaError_t e = cudaSuccess;
  if (fork) {  // helper stream i waits for the work queued before the launch on `stream`
    e = cudaEventRecord(ev[0], stream);
    for (int i = 1; i < np && e == cudaSuccess; ++i) e = cudaStreamWaitEvent(side[i - 1], ev[0], 0);
  }
  for (int i = 0; i < np && e == cudaSuccess; ++i) {
    const int a = present[i];
    cudaStream_t st = (fork && i > 0) ? side[i - 1] : stream;
    // the branches of one call are shaped as if alone: the longest decides when it ends (see fw_shape.h)
    e = table_launches(a).launch(g, grp + firsts[a], counts[a], totals[a], count, beside, qctr + a, st);
  }
  if (fork) {  // `stream` waits for the helper streams
    for (int i = 1; i < np && e == cudaSuccess; ++i) {
      e = cudaEventRecord(ev[i], side[i - 1]);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(stream, ev[i], 0);
    }
  }
  return e;
}

}  // namespace fw
