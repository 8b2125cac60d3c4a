// fw_kernels.cu -- single-job launches, the node statistics and the
// quantization and offset checks (per-row preprocessing: fw_preprocess.cu).
//
// A single job is one persistent launch of the walk kernel (fw_walk.cuh)
// compiled for its algorithm, so the other algorithms' code folds away;
// tables of several jobs go to fw_walk_mixed.cu.
#include <cstring>

#include "fw_internal.h"
#include "fw_rows.h"
#include "fw_walk.cuh"

namespace fw {


const WalkLaunches& single_weighted();
const WalkLaunches& single_node2vec();
const WalkLaunches& single_metapath();
const WalkLaunches& single_pagerank2();

const WalkLaunches& single_launches(int algo) {
  switch (algo) {
    case ALGO_WEIGHTED: return single_weighted();
    case ALGO_NODE2VEC: return single_node2vec();
    case ALGO_METAPATH: return single_metapath();
    default: return single_pagerank2();
  }
}

cudaError_t prime_walk_occupancy() {
  cudaError_t e = cudaSuccess;
  for (int a = 0; a < kAlgos && e == cudaSuccess; ++a) e = single_launches(a).prime();
  if (e == cudaSuccess) e = prime_walk_mixed_occupancy();
  return e;
}

cudaError_t single_needs_queue(const fw_graph* g, const Job& job, long long total, bool count, int beside, bool* need) {
  return single_launches(job.algo).needs_queue(g, &job, 1, total, count, beside, need);
}

cudaError_t launch_walk(const fw_graph* g, const Job* jobs, int njobs, long long total, bool count, int beside,
                        unsigned long long* qctr, cudaStream_t stream) {
  if (njobs == 1) return single_launches(jobs[0].algo).launch(g, jobs, 1, total, count, beside, qctr, stream);
  return launch_walk_mixed(g, jobs, njobs, count, beside, qctr, stream);
}

// ---------------------------------------------------------------- preprocessing
// h_MAX[v] and h_SUM[v]: one warp per node, lanes stride over the row
// (coalesced), then a shuffle-tree max and sum (Sec. 4.2 preprocess()).
// Lists the rows too long for one warp in the kernels that follow.  (0.27 ms
// on R-MAT s20; eight rows' offsets at a time with up to 32 loads in flight
// took 0.32.)
__global__ void node_stats_kernel(const int32_t* __restrict__ off, const float* __restrict__ h, int32_t n,
                                  float* __restrict__ hmax, float* __restrict__ hsum, int4* __restrict__ nrec,
                                  int* __restrict__ maxdeg, RowLists rows, double* __restrict__ mass) {
  const int lane = threadIdx.x & 31;
  const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  int localmax = 0;
  double envelope = 0.0, weight = 0.0, squares = 0.0;  // over the warp's rows: (4 n0 + 2 n1 + n2) / 4 * h_MAX, h_SUM, d^2
  for (long long v = warp; v < n; v += nwarps) {
    const int32_t s = off[v], e = off[v + 1];
    float m = 0.0f, sum = 0.0f;
    if (h) {
      for_entries(s, e - s, lane, 32, [&](int32_t i) {
        const float x = h[i];
        m = fmaxf(m, x);
        sum += x;
      });
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        m = fmaxf(m, __shfl_xor_sync(kFull, m, o));
        sum += __shfl_xor_sync(kFull, sum, o);
      }
    } else {
      m = (e > s) ? 1.0f : 0.0f;
      sum = (float)(e - s);
    }
    // entries of weight classes 0 (h > h_MAX / 2) and 1 (h_MAX / 4 < h <= h_MAX / 2);
    // without weights every entry is in class 0
    int n0 = e - s, n1 = 0;
    if (h) {
      const float half = 0.5f * m, quarter = 0.25f * m;
      n0 = 0;
      for_entries(s, e - s, lane, 32, [&](int32_t i) {
        const float x = h[i];
        n0 += (x > half) ? 1 : 0;
        n1 += (x > quarter && !(x > half)) ? 1 : 0;
      });
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        n0 += __shfl_xor_sync(kFull, n0, o);
        n1 += __shfl_xor_sync(kFull, n1, o);
      }
    }
    if (lane == 0) {
      hmax[v] = m;
      hsum[v] = sum;
      nrec[2 * v] = make_int4(s, e - s, __float_as_int(m), __float_as_int(sum));
      nrec[2 * v + 1] = make_int4(n0, n1, 0, 0);
      if (e - s > kBlockRow) rows.big[atomicAdd(rows.counts + 1, 1)] = (int32_t)v;
      else if (e - s > kWarpRow) rows.mid[atomicAdd(rows.counts, 1)] = (int32_t)v;
    }
    localmax = max(localmax, e - s);
    envelope += 0.25 * (double)(e - s + 3ll * n0 + n1) * (double)m;
    weight += (double)sum;
    squares += (double)(e - s) * (double)(e - s);
  }
  if (lane == 0 && localmax > 0) atomicMax(maxdeg, localmax);
  __shared__ double part[3][8];
  if (lane == 0) {
    part[0][threadIdx.x >> 5] = envelope;
    part[1][threadIdx.x >> 5] = weight;
    part[2][threadIdx.x >> 5] = squares;
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    double x = 0.0;
    for (int w = 0; w < 8; ++w) x += part[threadIdx.x][w];
    atomicAdd(mass + threadIdx.x, x);
  }
}

cudaError_t launch_node_stats(const int32_t* off, const float* h, int32_t n, float* hmax, float* hsum, int4* nrec,
                              int* maxdeg, const RowLists& rows, double* mass, int num_sms, cudaStream_t stream) {
  if (n == 0) return cudaSuccess;
  const long long want = ((long long)n * 32 + 255) / 256;
  const int grid = (int)(want < (long long)num_sms * 8 ? want : (long long)num_sms * 8);
  node_stats_kernel<<<grid, 256, 0, stream>>>(off, h, n, hmax, hsum, nrec, maxdeg, rows, mass);
  g_launches.fetch_add(1);
  return cudaGetLastError();
}

// Loads the statistics kernel (lazy module loading would otherwise do it
// inside the first timed launch).
cudaError_t prime_node_stats() {
  cudaFuncAttributes a;
  return cudaFuncGetAttributes(&a, node_stats_kernel);
}

// 8-bit weights with one scale per node: s_v = h_MAX[v] / 255 (FP32
// division; h_MAX of the FP32 weights), code = rint(h / s_v) (ties to even)
// clamped to [1, 255] (h > 0 stays > 0), and the FP32 copy rewritten as
// code * s_v, from which every derived structure is then rebuilt.  One warp
// per row; *maxbits receives the largest s_v (as bits: the scales are >= 0).
__global__ void quantize_rows_kernel(const int32_t* __restrict__ off, float* __restrict__ h,
                                     const float* __restrict__ hmax, int32_t n, uint8_t* __restrict__ codes,
                                     float* __restrict__ scales, unsigned* __restrict__ maxbits) {
  const int lane = threadIdx.x & 31;
  const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  unsigned m = 0;
  for (long long v = warp; v < n; v += nwarps) {
    const float sv = __fdiv_rn(hmax[v], 255.0f);
    if (lane == 0) scales[v] = sv;
    m = max(m, __float_as_uint(sv));
    for_entries(off[v], off[v + 1] - off[v], lane, 32, [&](int32_t i) {
      const float c = fminf(255.0f, fmaxf(1.0f, rintf(__fdiv_rn(h[i], sv))));
      codes[i] = (uint8_t)c;
      h[i] = __fmul_rn(c, sv);
    });
  }
  if (lane == 0 && m) atomicMax(maxbits, m);
}

cudaError_t launch_quantize(const int32_t* off, float* h, const float* hmax, int32_t n, uint8_t* codes,
                            float* scales, float* max_scale, unsigned* maxbits, int num_sms, cudaStream_t stream) {
  cudaError_t err = cudaMemsetAsync(maxbits, 0, sizeof(unsigned), stream);
  if (err != cudaSuccess) return err;
  if (n > 0) {
    quantize_rows_kernel<<<num_sms * 8, 256, 0, stream>>>(off, h, hmax, n, codes, scales, maxbits);
    g_launches.fetch_add(1);
    err = cudaGetLastError();
    if (err != cudaSuccess) return err;
  }
  unsigned bits = 0;
  err = cudaMemcpyAsync(&bits, maxbits, sizeof(unsigned), cudaMemcpyDeviceToHost, stream);
  if (err == cudaSuccess) err = cudaStreamSynchronize(stream);
  if (err != cudaSuccess) return err;
  std::memcpy(max_scale, &bits, sizeof(float));
  return cudaSuccess;
}

// CSR validation of device-resident input: bit 1 = offsets (the rows: see
// check_rows_kernel).
__global__ void check_offsets_kernel(const int32_t* __restrict__ off, int32_t n, int64_t e, unsigned* err) {
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v <= n; v += (long long)gridDim.x * blockDim.x) {
    const int32_t o = off[v];
    bool bad = (v == 0 && o != 0) || (v == n && (int64_t)o != e) || (v < n && off[v + 1] < o) || o < 0;
    if (bad) atomicOr(err, 1u);
  }
}

cudaError_t launch_check_offsets(const int32_t* off, int32_t n, int64_t e, unsigned* err, int num_sms,
                                 cudaStream_t stream) {
  const long long want = ((long long)n + 1 + 255) / 256;
  const int grid = (int)(want < (long long)num_sms * 8 ? want : (long long)num_sms * 8);
  check_offsets_kernel<<<grid > 0 ? grid : 1, 256, 0, stream>>>(off, n, e, err);
  g_launches.fetch_add(1);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- plan test hook
__global__ void step_plan_kernel(DevGraph g, Job J, const int32_t* __restrict__ v, const int32_t* __restrict__ vp,
                                 int32_t count, float* __restrict__ bound, float* __restrict__ sum_hat,
                                 int32_t* __restrict__ mode) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const int32_t x = v[i], y = vp[i];
  if (x < 0 || x >= g.n || y < -1 || y >= g.n) {
    mode[i] = -1;
    return;
  }
  float hm, hs, B, S, w1 = 1.0f, w2 = 1.0f;
  const int32_t d = g.off[x + 1] - g.off[x];
  if (J.weighted) {
    hm = g.hmax[x];
    hs = g.hsum[x];
  } else {
    hm = 1.0f;
    hs = (float)d;
  }
  if (J.algo == ALGO_PAGERANK2 && y >= 0) {
    const int32_t dp = g.off[y + 1] - g.off[y];
    if (d < 1 || dp < 1) {
      mode[i] = -1;
      return;
    }
    pagerank2_weights(J, d, dp, w1, w2);
  }
  mode[i] = plan_choice(J, hm, hs, y >= 0, w1, w2, B, S);
  bound[i] = B;
  sum_hat[i] = S;
}

cudaError_t launch_step_plan(const fw_graph* g, const Job& job, const int32_t* v, const int32_t* vp, int32_t count,
                             float* bound, float* sum_hat, int32_t* mode, cudaStream_t stream) {
  if (count <= 0) return cudaSuccess;
  step_plan_kernel<<<(count + 255) / 256, 256, 0, stream>>>(dev_graph(g), job, v, vp, count, bound, sum_hat, mode);
  g_launches.fetch_add(1);
  return cudaGetLastError();
}

}  // namespace fw
