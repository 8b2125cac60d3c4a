// fw_walk.cuh -- the walk kernel: its loop, the kernel template, its variants
// and their launcher, instantiated for single jobs (fw_walk_single_*.cu) and
// for tables of up to 64 jobs of one algorithm (fw_walk_table_*.cu).
//
// One warp runs the loop over one walker queue [Sec. 5.3]:
//   * query fetch   lanes without a walker take the next global walker
//                   indices with one warp-aggregated atomicAdd on the queue
//                   counter (launches with a lane for every walker take them
//                   by place instead, see LaunchShape); a table of jobs is one concatenated index space
//                   (job j owns [gbase_j, gbase_j + W_j)).
//   * plan          [Sec. 3.3, Sec. 4.1]: per walker-step the bound B and the
//                   sum estimate give the eRJS / eRVS choice (or a forced mode).
//   * eRJS          [Sec. 3.3, Sec. 5.2]: one walker per lane; a fixed number
//                   of trials per round, then the warp checks by ballot which
//                   lanes need a reservoir step (chosen eRVS, or trial cap hit).
//   * eRVS / exact  [Sec. 3.2, Sec. 5.2]: steps of degree <= a small threshold
//                   run on their own lane; larger ones are handed to the whole
//                   warp one at a time (shuffle of the walker's state), and
//                   the result goes back to the owning lane; hub rows
//                   (d >= kHubMinDeg) are cut into chunks that every warp of
//                   the block scans (CTA-level parallel jumps, see hub steps).
//   * update        [Sec. 4.2, update()]: prev <- cur, cur <- next, row write.
// All loops are bounded (trial cap, degree, walk length, hub wait limit); no
// warp waits on another.
#pragma once

#include <algorithm>

#include "fw_internal.h"
#include "fw_shape.h"

namespace fw {

constexpr int kBlock = 256;
// Resident blocks of 256 threads per SM, by kernel variant: 64 registers per
// thread at 4, 80 at 3, 48 at 5, 40 at 6, 32 at 7.  More warps hide the gathers'
// latency until the spills cost more.  GB300, ms: node2vec s22 p = 1/4, q = 4
// 40.0 / 33.9 / 37.5 with 3 / 4 / 5, its trials-together variant (Pareto 1,
// s20) 50.6 / 42.4 / 41.0; weighted s22 8.57 / 7.21 / 7.04 and 7.43 with 6
// (5: the dense variant, see kDenseRecords), for few walkers 0.061 with 4,
// 0.069 with 5; second-order PageRank s20 4.35
// / 4.49 / 4.8, its trials-together variant on Pareto 1 24.7 / 22.6 with 3 /
// 4; metapath 1.55 / 1.33 / 1.65; the eRVS-only variant (node2vec s18) 10.5 /
// 9.5 / 9.1 / 8.42 / 8.40 with 4 / 5 / 6 / 7 / 8, exact-only (weighted s18)
// 2.92 / 2.87 / 3.14 / 3.80 with 4 / 5 / 6 / 7.
// samplers a kernel variant holds (kWhole: all, short eRVS rows scanned at once, see kLaneRvs; kDense: all)
enum : int { kAny = 0, kOnlyRvs = 1, kOnlyExact = 2, kWhole = 3, kDense = 4 };
template <int ALG, bool SPREAD, bool SHARE, bool COOP, int ONLY>
constexpr int kMinBlocks = ONLY == kOnlyRvs                           ? 7
                           : ONLY == kOnlyExact                       ? 5
                           : SHARE                                    ? 4
                           : ALG == ALGO_NODE2VEC && COOP             ? 5
                           : ONLY == kDense                           ? 5
                           : ALG == ALGO_PAGERANK2 && (SPREAD || !COOP) ? 3
                                                                      : 4;
constexpr int kThreadExactMaxDeg = 16; // exact steps with d <= this run on one lane

// Row writes are staged per lane in shared memory, one aligned group of
// kStageSlots entries at a time, and written out when the group (or the
// row) is complete: scattered 4-byte stores would each cost a DRAM write.
// Slot s of lane t lives at obuf[s * kBlock + t] (no bank conflicts).
constexpr int kStageSlots = 8;  // 32-byte groups
static_assert(kStageSlots % 4 == 0 && (kStageSlots & (kStageSlots - 1)) == 0, "whole int4s, power of two");
__device__ __forceinline__ int32_t stage_slot(const int32_t* a) {
  return (int32_t)((reinterpret_cast<uintptr_t>(a) >> 2) & (uintptr_t)(kStageSlots - 1));
}

// write the staged slots [first, last] of the group holding `a` (a = address of slot `last`)
__device__ __forceinline__ void stage_flush(const int32_t* obuf, int tid, int32_t* a, int32_t first, int32_t last) {
  int32_t* base = a - last;
  if (first == 0 && last == kStageSlots - 1) {
#pragma unroll
    for (int q = 0; q < kStageSlots / 4; ++q)
      reinterpret_cast<int4*>(base)[q] = make_int4(obuf[(4 * q) * kBlock + tid], obuf[(4 * q + 1) * kBlock + tid],
                                                   obuf[(4 * q + 2) * kBlock + tid], obuf[(4 * q + 3) * kBlock + tid]);
  } else {
    for (int32_t k = first; k <= last; ++k) base[k] = obuf[k * kBlock + tid];
  }
}

// stage row[p] = val; `final` marks the last entry the lane will write in this row.  The row's first group may begin
// before the row.
__device__ __forceinline__ void stage_put(int32_t* obuf, int tid, int32_t* row, int32_t p, int32_t val, bool final) {
  int32_t* a = row + p;
  const int32_t slot = stage_slot(a);
  obuf[slot * kBlock + tid] = val;
  if (slot == kStageSlots - 1 || final) stage_flush(obuf, tid, a, max(slot - p, 0), slot);
}

// row[from, to) = -1 after a dead end: finish the staged group, then whole groups, then the tail
__device__ __forceinline__ void stage_fill_minus_one(int32_t* obuf, int tid, int32_t* row, int32_t from, int32_t to) {
  int32_t p = from;
  while (p < to && (p == from || stage_slot(row + p) != 0)) {
    stage_put(obuf, tid, row, p, -1, p + 1 == to);
    ++p;
  }
  for (; p + kStageSlots <= to; p += kStageSlots) {
    int4* q = reinterpret_cast<int4*>(row + p);
#pragma unroll
    for (int k = 0; k < kStageSlots / 4; ++k) q[k] = make_int4(-1, -1, -1, -1);
  }
  for (; p < to; ++p) row[p] = -1;
}

template <int NJ>
struct JobTableN {
  Job jobs[NJ];
};

// ---------------------------------------------------------------- hub steps
// An eRVS step of degree >= kHubMinDeg is shared by the warps of the block
// (the parallel jump process of Sec. 3.2 at CTA level).  The warp that owns
// the step keys the row's first kHubPhase1 positions (phase 1, the draws of
// the warp scan), and their maximum key K_g becomes the reference from which
// every other position is reached by jumps.  Those positions are cut into
// chunks of kHubChunk; inside a chunk, lane l scans lo + l, lo + l + 32, ...
// and starts with its own jump threshold, drawn from counter (walker, hop,
// 5, lo + l); crossings draw as in the warp scan.  A chunk's keys therefore
// depend on its positions and K_g alone, so the result is the same whether
// the owning warp scans every chunk itself or the block shares them, and
// whatever warp scans which chunk when.
//
// Sharing: the owning warp posts the step to a free slot of the block's task
// table in shared memory (else it scans the chunks alone).  A warp that
// looks (see the walk loop: warps with a waiting lane, and warps whose queue
// ran dry) claims the next chunk of an open task, scans it and enters the
// chunk's best (key, position) by one 64-bit atomicMax on the pair packed in
// key order (equal keys: the larger position, as in warp_argmax), then
// counts the chunk done.  The owning lane takes the result once every chunk
// is done; its warp keeps walking its other lanes and claims chunks itself,
// so no warp waits on another and a task completes even when no other warp
// helps.  Busy warps do not look: with every lane walking, sharing would
// move work between warps without shortening the launch, and the check
// itself costs time on every iteration.
constexpr int32_t kHubMinDeg = 32768;            // eRVS steps of at least this degree are shared
constexpr int32_t kHubPhase1Keys = 32;           // phase-1 keys per lane
constexpr int32_t kHubPhase1 = 32 * kHubPhase1Keys;  // positions keyed in phase 1
constexpr int32_t kHubChunk = 8192;              // positions per chunk (256 per lane)
constexpr int kHubTasks = 4;                     // open hub steps per block
constexpr int32_t kHubMaxChunks = 1 << 19;       // the 20-bit chunk counter never wraps
constexpr uint32_t kHubWaitLimit = 1u << 24;     // loop iterations a lane waits for its step at most
// slot word: state (2 bits) | generation (10 bits) | next unclaimed chunk (20 bits)
constexpr uint32_t kHubFree = 0u, kHubReserved = 1u, kHubOpen = 2u;
constexpr uint32_t kHubGenMask = 0x3ff00000u, kHubNextMask = 0x000fffffu;

struct HubTask {
  uint32_t word;
  int32_t nchunks;
  int32_t done;              // chunks scanned
  int32_t job;
  unsigned long long best;   // packed (ordered key, position) of the best key so far; 0: none
  float ref;                 // K_g: the phase-1 maximum key
  int32_t grp;               // grouped metapath: c.s, c.d are the label segment
  StepCtx c;
};

struct HubBlock {  // shared memory, per block
  HubTask task[kHubTasks];
  int32_t open;    // tasks with chunks left to claim
  int32_t live;    // warps of the block still walking (the others linger to help)
};
constexpr uint32_t kLingerLimit = 1u << 22;  // idle checks of a lingering warp at most

// float key -> unsigned in the same order (no NaN keys arise)
__device__ __forceinline__ uint32_t key_order(float k) {
  const uint32_t u = __float_as_uint(k);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ unsigned long long key_pack(float k, int32_t pos) {
  return (k == -CUDART_INF_F) ? 0ull : (((unsigned long long)key_order(k) << 32) | (uint32_t)pos);
}

__device__ __forceinline__ int32_t hub_chunks(int32_t d) { return (d - kHubPhase1 + kHubChunk - 1) / kHubChunk; }

// Phase 1 of a hub step (the whole warp): keys of positions lane + 32 j,
// j < kHubPhase1Keys, four per Philox block as in rvs_scan.  A chunk lane crosses K_g about ln(1 + n / kHubPhase1)
// times over its n positions, every crossing a divergent key draw, so the
// reference is taken over more positions than a warp scan's phase 1.
// Leaves the lane's best in bestK / best.
template <bool COUNT, int ALG, bool GRP>
__device__ __forceinline__ void hub_phase1(const DevGraph& g, const Job& J, const StepCtx& c, int lane,
                                           LaneCounters& lc, float& bestK, int32_t& best) {
  uint32_t probes = 0;
  bestK = -CUDART_INF_F;
  best = -1;
  int32_t keys = 0;
  uint4 x4 = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll 1
  for (int32_t j = 0; j < kHubPhase1Keys; ++j) {
    const int32_t k = lane + 32 * j;
    const float wt = scan_weight<ALG, GRP>(g, J, c, c.s + k, probes);
    if ((j & 3) == 0) x4 = philox(make_uint4(c.wid, (uint32_t)c.step, 6u, (uint32_t)k), J.key0, J.key1);
    const uint32_t r = (j & 3) == 0 ? x4.x : ((j & 3) == 1 ? x4.y : ((j & 3) == 2 ? x4.z : x4.w));
    if (wt > 0.0f) {
      const float K = logf(u01_open(r)) / wt;
      ++keys;
      if (K >= bestK) {
        bestK = K;
        best = k;
      }
    }
  }
  if (COUNT) rvs_count<ALG, GRP>(J, kHubPhase1Keys, keys, probes, lc);
}

// Chunk [lo, hi) of a hub step (the whole warp): jumps from K_g = ref with
// per-lane thresholds from counter stream 5 (without jumps: every key, as in
// the warp scan).  Leaves the lane's best in bestK / best.
template <bool COUNT, int ALG, bool GRP>
__device__ __forceinline__ void hub_chunk_scan(const DevGraph& g, const Job& J, const StepCtx& c, int32_t lo,
                                               int32_t hi, float ref, bool jump, int lane, LaneCounters& lc,
                                               float& bestK, int32_t& best) {
  uint32_t probes = 0;
  int32_t scanned = 0, keys = 0;
  bestK = -CUDART_INF_F;
  best = -1;
  float r = ref, rem = 0.0f;  // K_g = -inf: the first positive item crosses
  if (jump && r != -CUDART_INF_F) {
    const uint4 x0 = philox(make_uint4(c.wid, (uint32_t)c.step, 5u, (uint32_t)(lo + lane)), J.key0, J.key1);
    rem = (r < 0.0f) ? logf(u01_open(x0.x)) / r : CUDART_INF_F;
  }
  for (int32_t k = lo + lane; k < hi; k += 32) {
    const float wt = scan_weight<ALG, GRP>(g, J, c, c.s + k, probes);
    ++scanned;
    if (!(wt > 0.0f)) continue;
    if (!jump) {
      const uint4 x = philox(make_uint4(c.wid, (uint32_t)c.step, 2u, (uint32_t)k), J.key0, J.key1);
      const float K = logf(u01_open(x.x)) / wt;
      ++keys;
      if (K >= bestK) {
        bestK = K;
        best = k;
      }
    } else {
      rem -= wt;
      if (rem <= 0.0f) {
        const uint4 x = philox(make_uint4(c.wid, (uint32_t)c.step, 2u, (uint32_t)k), J.key0, J.key1);
        // key conditioned on beating r: u' ~ U(exp(r*wt), 1), K = ln(u') / wt
        const float K = log1pf(expm1f(r * wt) * u01_open(x.y)) / wt;
        ++keys;
        bestK = K;
        best = k;
        r = K;
        rem = (r < 0.0f) ? logf(u01_open(x.z)) / r : CUDART_INF_F;
      }
    }
  }
  if (COUNT) rvs_count<ALG, GRP>(J, scanned, keys, probes, lc);
}

// Post a hub step (one lane); -1: every slot taken.
__device__ __forceinline__ int hub_post(HubBlock* hb, const StepCtx& c, int32_t job, bool grp, float ref,
                                        unsigned long long best) {
  for (int i = 0; i < kHubTasks; ++i) {
    HubTask& t = hb->task[i];
    const uint32_t w = *reinterpret_cast<volatile uint32_t*>(&t.word);
    if ((w >> 30) != kHubFree) continue;
    if (atomicCAS(&t.word, w, (kHubReserved << 30) | (w & kHubGenMask)) != w) continue;
    t.c = c;
    t.job = job;
    t.grp = grp ? 1 : 0;
    t.ref = ref;
    t.nchunks = hub_chunks(c.d);
    t.done = 0;
    t.best = best;
    __threadfence_block();  // the fields before the slot opens
    const uint32_t gen = ((w >> 20) + 1u) & 0x3ffu;
    atomicExch(&t.word, (kHubOpen << 30) | (gen << 20));
    atomicAdd(&hb->open, 1);
    return i;
  }
  return -1;
}

// Claim the next unclaimed chunk of the open task in `slot` (one lane);
// false: none left.  The compare-and-swap against the word read fails if
// the slot was claimed, closed or reopened meanwhile, so a successful claim
// also vouches for the chunk count read before it.  Taking a task's last
// chunk closes it for the lingering warps' check.
__device__ __forceinline__ bool hub_claim_slot(HubBlock* hb, int slot, int32_t& chunk) {
  HubTask& t = hb->task[slot];
  uint32_t w = *reinterpret_cast<volatile uint32_t*>(&t.word);
  for (int tries = 0; tries < 64 && (w >> 30) == kHubOpen; ++tries) {
    const int32_t nc = *reinterpret_cast<volatile int32_t*>(&t.nchunks);
    const int32_t nx = (int32_t)(w & kHubNextMask);
    if (nx >= nc) return false;
    const uint32_t old = atomicCAS(&t.word, w, w + 1u);
    if (old == w) {
      if (nx + 1 == nc) atomicSub(&hb->open, 1);
      chunk = nx;
      return true;
    }
    w = old;
  }
  return false;
}

// Scan claimed chunk `chunk` of the task in `slot` (the whole warp,
// converged), enter its best and count it done.
template <bool COUNT, int ALG>
__device__ __forceinline__ void hub_scan_claimed(const DevGraph& g, const Job* sj, HubBlock* hb, int slot,
                                                 int32_t chunk, LaneCounters& lc) {
  const int lane = threadIdx.x & 31;
  HubTask& t = hb->task[slot];  // fixed until this chunk is counted done
  StepCtx hc;
  const volatile int32_t* src = reinterpret_cast<const volatile int32_t*>(&t.c);
  int32_t* dst = reinterpret_cast<int32_t*>(&hc);
#pragma unroll
  for (int q = 0; q < (int)(sizeof(StepCtx) / 4); ++q) dst[q] = src[q];
  const Job& J = sj[*reinterpret_cast<volatile int32_t*>(&t.job)];
  const float ref = *reinterpret_cast<volatile float*>(&t.ref);
  const int32_t lo = kHubPhase1 + chunk * kHubChunk, hi = min(hc.d, lo + kHubChunk);
  const bool jump = !(J.flags & FW_FLAG_RVS_NOJUMP);
  float bk;
  int32_t bi;
  if (ALG == ALGO_METAPATH && *reinterpret_cast<volatile int32_t*>(&t.grp) != 0)
    hub_chunk_scan<COUNT, ALG, true>(g, J, hc, lo, hi, ref, jump, lane, lc, bk, bi);
  else
    hub_chunk_scan<COUNT, ALG, false>(g, J, hc, lo, hi, ref, jump, lane, lc, bk, bi);
  warp_argmax(bk, bi);
  if (lane == 0) {
    if (bk != -CUDART_INF_F) atomicMax(&t.best, key_pack(bk, bi));
    __threadfence_block();  // the result before the chunk counts as done
    atomicAdd(&t.done, 1);
  }
  __syncwarp();
}

// A lingering warp (converged, no walker left): claim and scan one chunk of
// any open task of the block.  Returns whether a chunk was scanned.
template <bool COUNT, int ALG>
__device__ __forceinline__ bool hub_help(const DevGraph& g, const Job* sj, HubBlock* hb, LaneCounters& lc) {
  const int lane = threadIdx.x & 31;
  if (__shfl_sync(kFull, *reinterpret_cast<volatile int32_t*>(&hb->open), 0) <= 0) return false;
  int32_t chunk = 0;
  int slot = -1;
  if (lane == 0) {
    for (int i = 0; i < kHubTasks && slot < 0; ++i)
      if (hub_claim_slot(hb, i, chunk)) slot = i;
  }
  slot = __shfl_sync(kFull, slot, 0);
  if (slot < 0) return false;
  chunk = __shfl_sync(kFull, chunk, 0);
  __syncwarp();
  hub_scan_claimed<COUNT, ALG>(g, sj, hb, slot, chunk, lc);
  return true;
}

// A hub step (the whole warp, converged; cw, JW: the step and its job, jb
// its index, grp: grouped metapath).  Phase 1; then, when a warp of the
// block lingers to help, the step is posted and this warp claims and scans
// chunks alongside the helpers until none is left, waits for the chunks the
// helpers hold (they wait on nothing) and frees the slot; otherwise it scans
// every chunk alone (always, without SHARE).  Returns the position (-1: all
// weights zero, or the join wait ran out, which also sets DEVERR_HUB).
template <bool COUNT, int ALG, bool SHARE>
__device__ __forceinline__ int32_t hub_step(const DevGraph& g, const Job* sj, const Job& JW, const StepCtx& cw,
                                            int32_t jb, bool grp, HubBlock* hb, unsigned* err, LaneCounters& lc) {
  const int lane = threadIdx.x & 31;
  float bk;
  int32_t bi;
  if (ALG == ALGO_METAPATH && grp) hub_phase1<COUNT, ALG, true>(g, JW, cw, lane, lc, bk, bi);
  else hub_phase1<COUNT, ALG, false>(g, JW, cw, lane, lc, bk, bi);
  const float ref = warp_max(bk);
  warp_argmax(bk, bi);
  int slot = -1;
  if (SHARE && lane == 0 && *reinterpret_cast<volatile int32_t*>(&hb->live) < (int32_t)(blockDim.x >> 5))
    slot = hub_post(hb, cw, jb, grp, ref, key_pack(bk, bi));
  if (SHARE) slot = __shfl_sync(kFull, slot, 0);
  if (SHARE && slot >= 0) {
    HubTask& t = hb->task[slot];
    while (true) {
      int32_t chunk = 0;
      bool got = false;
      if (lane == 0) got = hub_claim_slot(hb, slot, chunk);
      if (!__shfl_sync(kFull, (int)got, 0)) break;
      chunk = __shfl_sync(kFull, chunk, 0);
      __syncwarp();
      hub_scan_claimed<COUNT, ALG>(g, sj, hb, slot, chunk, lc);
    }
    // join: the helpers finish the chunks they claimed
    bool ok = false;
    if (lane == 0) {
      const int32_t nc = t.nchunks;
      for (uint32_t it = 0; it < kHubWaitLimit; ++it) {
        if (*reinterpret_cast<volatile int32_t*>(&t.done) >= nc) {
          ok = true;
          break;
        }
        __nanosleep(64);
      }
    }
    ok = __shfl_sync(kFull, (int)ok, 0) != 0;
    if (!ok) {
      if (lane == 0) atomicOr(err, DEVERR_HUB);  // the slot stays taken
      return -1;
    }
    __threadfence_block();
    const unsigned long long r = *reinterpret_cast<volatile unsigned long long*>(&t.best);
    __syncwarp();
    if (lane == 0) {
      const uint32_t wd = *reinterpret_cast<volatile uint32_t*>(&t.word);
      atomicExch(&t.word, wd & kHubGenMask);  // free, keeping the generation
    }
    return r ? (int32_t)(uint32_t)r : -1;
  }
  const bool jump = !(JW.flags & FW_FLAG_RVS_NOJUMP);
  const int32_t nch = hub_chunks(cw.d);
  for (int32_t q = 0; q < nch; ++q) {
    const int32_t lo = kHubPhase1 + q * kHubChunk, hi = min(cw.d, lo + kHubChunk);
    float ck;
    int32_t ci;
    if (ALG == ALGO_METAPATH && grp) hub_chunk_scan<COUNT, ALG, true>(g, JW, cw, lo, hi, ref, jump, lane, lc, ck, ci);
    else hub_chunk_scan<COUNT, ALG, false>(g, JW, cw, lo, hi, ref, jump, lane, lc, ck, ci);
    warp_argmax(ck, ci);
    if (ck > bk || (ck == bk && ci > bi)) {
      bk = ck;
      bi = ci;
    }
  }
  return (bk == -CUDART_INF_F) ? -1 : bi;
}

// Trials together: failed trials after which a step's next ones are made by
// the whole warp.  The code costs the loop registers, so it is a kernel
// variant, used on graphs whose mean envelope mass per unit of weight, the
// trials of a first-order hop, is at least kTogetherEnvelope.  Second-order
// PageRank, whose steps without a split fail most trials, uses it from
// kTogetherPagerank, and for few walkers always.
// GB300, R-MAT s18 x 10 hops, 20,000 / 400,000 walkers, a lane's own trials
// -> together (ms): envelope 1.4 (U(0,1] weights) node2vec p = 2, q = 1/2
// 0.10 / 0.53 -> 0.13 / 0.78, PageRank 0.46 / 2.19 -> 0.26 / 2.03; 3.6
// (lognormal) node2vec 0.24 / 0.99 -> 0.26 / 2.09, weighted 0.11 / 0.55 ->
// 0.11 / 0.62, PageRank 1.93 / 5.22 -> 0.47 / 3.26; 6.5 (Pareto 2) node2vec
// 1.07 / 4.58 -> 0.35 / 2.77, weighted 0.91 / 2.37 -> 0.13 / 0.80; 246
// (Pareto 1) node2vec 7.9 / 29.6 -> 2.8 / 19.6, weighted 7.1 / 13.5 -> 0.9 /
// 5.0, metapath 0.41 / 1.42 -> 0.13 / 0.73.  From 8 / 16 / 32 trials: Pareto
// 1 node2vec 19.6 / 21.4 / 23.3, PageRank on U(0,1] 2.16 / 2.03 / 1.92 and on
// Pareto 1 21.3 / 22.6 / 24.7; PageRank on s20, U(0,1], 262,144 walkers x 40
// hops 4.9 -> 5.3.
template <int ALG>
constexpr int32_t kTogetherFrom = ALG == ALGO_PAGERANK2 ? 16 : 8;
constexpr double kTogetherEnvelope = 5.0, kTogetherPagerank = 2.5;
// It pays where a launch ends with its longest steps; where all walkers' hops
// outweigh them, the lanes' own trials are the faster ones.  The more so the
// lower the envelope E: launches of up to kTogetherHops * E hops in all (and
// metapath, whose steps see a label's share of a row, kTogetherHopsLeast).
// GB300, speed against the earlier kernel, together / a lane's own: Pareto 2
// (E = 5 to 8 on s16 / s18 / s20) node2vec p = 2, q = 1/2 2.0 M hops 1.14 /
// 2.47 / 1.36 and 1.10 / 0.93 / 0.96, 3.6 M 0.84 / 1.21 / 1.00 and 1.31 / 1.31
// / 1.25, 12 M 0.80 / 0.88 / 0.79 and 1.47 / 1.14 / 1.11, 45 M 0.76 / 0.71 /
// 0.62 and 1.61 / 1.34 / 1.30; weighted 12 M 1.32 / 1.68 / 1.20 and 1.02 /
// 0.97 / 1.00, 45 M 0.83 / 0.98 / 0.91 and 0.99 / 0.99 / 1.01; metapath 2.0 M
// 1.12 / 1.92 / 1.46 and 1.02 / 0.98 / 0.98, 12 M 0.88 / 1.04 / 0.95 and 1.05
// / 1.01 / 1.01.  Pareto 1 (E = 75 and more): node2vec 45 M 1.04 / 1.14 / 1.15
// and 1.12 / 1.08 / 1.04, weighted 45 M 1.13 / 1.45 / 1.69 and 0.97 / 0.98 /
// 0.97, metapath 12 M 0.85 / 1.29 / 1.96 and 1.00 / 0.99 / 0.97.
template <int ALG>
constexpr double kTogetherHops = ALG == ALGO_WEIGHTED ? 2.5e6 : ALG == ALGO_NODE2VEC ? 0.4e6 : 0.09e6;
constexpr double kTogetherHopsLeast = 2.5e6;

// The walk loop of one warp over one queue: take walkers, plan, sample and
// write rows until the queue is exhausted and the warp holds no walker.
// `sj` (shared memory; a single job: kernel parameters) is the queue's job table: its jobs' walkers form the
// index space [0, total), job j owning [sj[j].gbase, sj[j].gbase + W_j).
// ALG fixes the algorithm of every job at compile time.  SPREAD: the launch
// is given its first walkers by place, `wpw` per warp; SHARE: hub steps may be
// shared with the block's idle warps (see hub steps); COOP: long eRJS steps
// try 32 proposals at once (see trials together); ONLY: every job is forced
// eRVS, or every job exact, and the other samplers' code is left out.
template <int NJ, bool COUNT, int ALG, bool SPREAD, bool SHARE, bool COOP, int ONLY>
__device__ __forceinline__ void walk_loop(const DevGraph& g, const Job* sj, int njobs, long long total, int wpw,
                                          unsigned long long* __restrict__ qctr, unsigned* __restrict__ err,
                                          int32_t* obuf, HubBlock* hb, LaneCounters& lc) {
  static_assert(ALG >= 0 && ALG < kAlgos, "the walk loop is compiled for one algorithm");
  // Short eRVS rows in step with the trials (see rjs_trials): node2vec only.
  // There a row's positions each wait for a membership test, and a warp paid
  // for them whenever one of its lanes had such a step: GB300, one walker per
  // node x 80 hops, whole rows at once -> one position per trial: s20 p = 4,
  // q = 1/4 7.60 -> 6.71 ms, s22 p = 1/4, q = 4 49.5 -> 44.9 ms; with warp
  // rows of up to 32 entries as well, each of which held all 32 lanes, 6.28
  // and 39.3 ms.  First-order
  // rows are one or two sectors of h that stay in L1 (weighted s22 7.46 ms at
  // once, 7.64 in step; metapath 1.32 and 1.40 ms); so are launches with few
  // lanes per warp (5,003 walkers 379 and 538 us); second-order PageRank
  // seldom has such rows and loses the registers (8.46 and 8.80 ms).
  constexpr bool kLaneRvs = !SPREAD && ALG == ALGO_NODE2VEC && ONLY != kWhole;
  constexpr bool kTrials = ONLY != kOnlyRvs && ONLY != kOnlyExact, kRvs = ONLY != kOnlyExact;
  constexpr bool kExact = ONLY == kOnlyExact || (kTrials && (COUNT || NJ > 1));  // single exact jobs: kOnlyExact
  const int lane = threadIdx.x & 31;
  const int tid = threadIdx.x;

  // Walker state that lives across iterations; every word of it is a register
  // the trials lack (64 per thread with 4 blocks per SM; what does not fit is
  // spilled in the loop), so values that are never needed together share one
  // (with the job in constant operands: spill loads of the node2vec kernel
  // 236 -> 112 bytes; GB300, s22 p = 1/4, q = 4 39.3 -> 33.9 ms, s20 p = 4, q =
  // 1/4 6.27 -> 5.33 ms, of which the job 5 %):
  // between a hop and its plan the next node's record sits in c.s, c.d, c.n0,
  // c.n1, B (h_MAX) and beta (h_SUM).  c.v current node, c.vp previous node
  // (-1: none), c.step hop, c.s / c.d row of c.v, c.ps / c.pe row of c.vp
  // (metapath in the label-grouped view: the required label's segment of the
  // grouped arrays; metapath has no use for the row of v').
  StepCtx c;
  c.v = c.vp = c.s = c.d = c.ps = c.pe = c.step = 0;
  c.wid = 0;
  c.w1 = c.w2 = 1.0f;
  c.n0 = -1;
  c.n1 = 0;
  c.hsc = 0.0f;
  int32_t job = 0, widx = -1;
  int32_t plan = PLAN_NONE, trials = 0;
  float B = 0.0f;
  // eRJS with the return edge split off: probability of the return component,
  // position of v' in N(v) (-1: unknown) and h(v, v'); before the plan h_ret is h of the edge taken (-1: unknown)
  bool split = false;
  float beta = 0.0f, h_ret = -1.0f;
  // node2vec with 1/q < 1 and d(v') < d(v): two envelopes; beta2 = (E3 + E2) / E
  bool csplit = false;
  float beta2 = 0.0f;
  bool grp = false;  // metapath in the label-grouped view
  int32_t pos_ret = -1;
  bool exhausted = false;  // warp-uniform
  bool first = SPREAD;     // warp-uniform

  while (true) {
    // ------------------------------------------------------------ fetch
    const bool need = widx < 0 && (!SPREAD || lane < wpw);
    const unsigned nm = __ballot_sync(kFull, need);
    if (nm != 0u && !exhausted) {
      const int leader = __ffs(nm) - 1;
      const unsigned cntw = __popc(nm);
      unsigned long long base = 0;
      if (SPREAD && first) {  // warp 0 of every block first, then warp 1, ...
        base = (unsigned)((threadIdx.x >> 5) * gridDim.x + blockIdx.x) * (unsigned)wpw;
        first = false;
        if (qctr == nullptr) exhausted = true;
      } else {
        if (lane == leader) base = atomicAdd(qctr, (unsigned long long)cntw);
        base = __shfl_sync(kFull, base, leader);
        if (SPREAD) base += (unsigned)(gridDim.x * (blockDim.x >> 5)) * (unsigned long long)wpw;
      }
      if (base + cntw >= (unsigned long long)total) exhausted = true;
      if (need) {
        const long long gi = (long long)base + __popc(nm & ((1u << lane) - 1u));
        if (gi < total) {
          if (NJ > 1) {
            job = 0;
            while (job + 1 < njobs && sj[job + 1].gbase <= gi) ++job;
          }
          const Job& J = sj[job];
          widx = (int32_t)(gi - J.gbase);
          if (J.kind == JOB_WALK) {
            const int32_t st = __ldg(J.starts + widx);
            int32_t* row = J.out + (long long)widx * (J.len + 1);
            if (st < 0 || st >= g.n) {
              atomicOr(err, DEVERR_START);
              stage_fill_minus_one(obuf, tid, row, 0, J.len + 1);
              widx = -1;
            } else {
              stage_put(obuf, tid, row, 0, st, J.len == 0);
              c.v = st;
              c.vp = -1;
              c.step = 0;
              if (J.len == 0) widx = -1;
            }
          } else {
            c.v = J.hv;
            c.vp = J.hprev;
            c.step = J.hstep;
            if (c.vp >= 0) {  // during walks the row of v' is carried along; here it is loaded
              const int4 pr = __ldg(g.nrec + 2ll * c.vp);
              c.ps = pr.x;
              c.pe = pr.x + pr.y;
            }
          }
          c.wid = J.wids && widx >= 0 ? __ldg(J.wids + widx) : J.walker_base + (uint32_t)widx;
          plan = PLAN_NONE;
          h_ret = -1.0f;
        }
      }
    }
    if (!__any_sync(kFull, widx >= 0)) {
      if (exhausted) break;
      continue;
    }

    const Job& J = sj[job];
    int32_t pick = -2, node = -1;  // this iteration's outcome: position drawn (-1: dead end, -2: none yet), its node
    bool sum_common = false;       // second-order PageRank: this plan needs S_C
    // ------------------------------------------------------------ plan
    if (widx >= 0 && (plan == PLAN_NONE || plan == PLAN_READY)) {
      // row start, degree, h_MAX, h_SUM and class counts of v: from the hop's edge record, or one load
      if (plan == PLAN_NONE) {
        int4 nr, nr2;
        ld_record(g.nrec + 2ll * c.v, nr, nr2);
        c.s = nr.x;
        c.d = nr.y;
        c.n0 = nr2.x;
        c.n1 = nr2.y;
        B = __int_as_float(nr.z);
        beta = __int_as_float(nr.w);
        if (COUNT) lc.bytes += 32;
      }
      const float node_hm = B, node_hs = beta, h_in = h_ret;
      const int32_t n0 = c.n0, n1 = c.n1;
      if (g.h8) c.hsc = __ldg(g.h8scale + c.v);  // scale of the codes of v's row
      // weight classes in eRJS wherever the bound is a multiple of h_MAX[v]
      const bool cls = J.classes && !(FW_ALGO(J) == ALGO_METAPATH && J.label_stats);
      if (!cls) c.n0 = -1;
      // eRJS envelope mass in units of the class-0 bound: (4 n0 + 2 n1 + n2) / 4
      const float dsl = cls ? __fmul_rn(0.25f, (float)(c.d + 3 * n0 + n1)) : (float)c.d;
      trials = 0;
      split = false;
      csplit = false;
      grp = false;
      beta = 0.0f;
      if (c.d == 0) {
        pick = -1;
        plan = PLAN_RJS;
      } else {
        int32_t m = J.mode;
        if (ONLY == kOnlyExact || (kExact && m == MODE_EXACT)) {
          if (FW_ALGO(J) == ALGO_PAGERANK2 && c.vp >= 0) pagerank2_weights(J, c.d, c.pe - c.ps, c.w1, c.w2);
          plan = (c.d <= kThreadExactMaxDeg) ? PLAN_EXACT_T : PLAN_EXACT_W;
        } else {
          float hm, hs, S;
          if (J.weighted) {
            hm = node_hm;
            hs = node_hs;
          } else {
            hm = 1.0f;
            hs = (float)c.d;
          }
          int32_t choice;
          if (FW_ALGO(J) == ALGO_METAPATH && J.label_group) {
            // per-label record of v: exact bound and sum over the required label,
            // and where its entries sit in the label-grouped view; none -> dead end
            const uint8_t want = J.schema[c.step % J.schema_len];
            int4 lr = make_int4(0, 0, 0, 0), lr2 = make_int4(0, 0, 0, 0);
            if (want < kLabelStats) {
              ld_record(g.lrec + 2ll * ((long long)c.v * kLabelStats + want), lr, lr2);
              if (COUNT) lc.bytes += 32;
            }
            B = __int_as_float(lr.x);
            S = __int_as_float(lr.y);
            grp = true;
            c.ps = c.s + lr.z;
            c.pe = c.ps + lr.w;
            c.gcls = lr2;
            // expected eRJS trials follow the class envelope: bound B * slots / (16 len)
            const float beff = lr.w > 0 ? __fmul_rn(B, (float)class_slots(lr2, lr.w) / (16.0f * (float)lr.w)) : B;
            choice = (__fmul_rn(J.ratio, beff) < S) ? MODE_RJS : MODE_RVS;
            if (!(S > 0.0f)) pick = -1;
          } else if (FW_ALGO(J) == ALGO_METAPATH && J.label_stats) {
            // metapath with per-label statistics: exact bound and exact sum over
            // the edges whose label the step requires; none -> dead end now
            const uint8_t want = J.schema[c.step % J.schema_len];
            float2 ls = make_float2(0.0f, 0.0f);
            if (want < kLabelStats) {
              ls = __ldg(g.lstat + (long long)c.v * kLabelStats + want);
              if (COUNT) lc.bytes += 8;
            }
            B = ls.x;
            S = ls.y;
            choice = (__fmul_rn(J.ratio, B) < S) ? MODE_RJS : MODE_RVS;
            if (!(S > 0.0f)) pick = -1;
          } else {
            if (FW_ALGO(J) == ALGO_PAGERANK2 && c.vp >= 0) pagerank2_weights(J, c.d, c.pe - c.ps, c.w1, c.w2);
            choice = plan_choice<ALG>(J, hm, hs, c.vp >= 0, c.w1, c.w2, B, S);
            // with weight classes the expected trials scale with the envelope mass dsl * B
            const float frac = dsl / (float)c.d;
            if (cls) choice = (__fmul_rn(J.ratio, __fmul_rn(B, frac)) < S) ? MODE_RJS : MODE_RVS;
            if (FW_ALGO(J) == ALGO_PAGERANK2 && c.vp >= 0 && !(J.flags & FW_FLAG_PLAIN_RJS) &&
                c.pe - c.ps <= kPr2SplitMaxPrev && c.w1 > __fmul_rn(2.0f, c.w2)) {
              // common neighbours split off: eRJS then costs as a first-order walk with bound w2 h_MAX
              split = true;
              B = __fmul_rn(c.w2, hm);
              S = __fmul_rn(c.w2, hs);
              choice = (__fmul_rn(J.ratio, __fmul_rn(B, frac)) < S) ? MODE_RJS : MODE_RVS;
            }
          }
          if (m == MODE_AUTO) {
            m = choice;
          } else if (m == MODE_RANDOM) {  // coin from Philox counter (wid, hop, 4, 0)
            m = (philox(make_uint4(c.wid, (uint32_t)c.step, 4u, 0u), J.key0, J.key1).x >> 31) ? MODE_RJS : MODE_RVS;
          } else if (m == MODE_DEGREE) {
            m = (c.d < kDegreeRuleThreshold) ? MODE_RVS : MODE_RJS;
          }
          plan = (kTrials && m == MODE_RJS) ? PLAN_RJS : (((grp ? c.pe - c.ps : c.d) <= J.lane_max) ? PLAN_RVS_T : PLAN_RVS_W);
          if (ALG == ALGO_PAGERANK2) {
            split = split && plan == PLAN_RJS;
            sum_common = split;
          } else if (kTrials && FW_ALGO(J) == ALGO_NODE2VEC && plan == PLAN_RJS && c.vp >= 0 &&
                     (J.split_return || (J.split_common && (float)(c.pe - c.ps) < dsl))) {
            // the return edge alone sets max(w) = 1/p: propose it separately and
            // bound the other neighbours by max(1, 1/q) * h_MAX[v]; with 1/q < 1 and
            // a row of v' shorter than the envelope of N(v), two envelopes (see rjs_trials)
            split = true;
            csplit = J.split_common && (float)(c.pe - c.ps) < dsl;
            B = csplit ? hm : __fmul_rn(J.whi1, hm);
            pos_ret = -1;
            bool have = false;
            if (g.sym && h_in >= 0.0f && J.kind == JOB_WALK) {
              h_ret = h_in;  // symmetric weights: h(v, v') = h(v', v), the edge just taken
              have = true;
            } else {
              uint32_t pb = 0;
              pos_ret = row_find(g.col, c.s, c.s + c.d, c.vp, g.n, pb);
              if (COUNT) {
                lc.probes += pb;
                lc.bytes += 32ull * pb;
              }
              if (pos_ret >= 0) {
                h_ret = load_h(g, J, pos_ret, c.hsc);
                pos_ret -= c.s;
                have = true;
              }
            }
            if (csplit) {
              const float e3 = have ? __fmul_rn(J.inv_p, h_ret) : 0.0f;
              const float e2 = __fmul_rn(__fmul_rn(__fsub_rn(1.0f, J.inv_q), (float)(c.pe - c.ps)), hm);
              const float e1 = __fmul_rn(__fmul_rn(J.inv_q, dsl), hm);
              const float tot = __fadd_rn(__fadd_rn(e3, e2), e1);
              beta = e3 / tot;
              beta2 = __fadd_rn(e3, e2) / tot;
            } else if (have) {
              const float wret = __fmul_rn(J.inv_p, h_ret);
              beta = wret / (wret + dsl * B);
            }
          }
        }
      }
    }
    // ------------------------------------------------------------ common neighbours
    // Second-order PageRank with a short row of v' (Eq. 2ndpr): the common
    // neighbours C = N(v) and N(v') carry w1 > w2, all others w2.  Looking up
    // every x of N(v') in N(v) finds C; a new plan needs S_C = sum of h(v, x)
    // over x in C (FP32, in N(v') order), a trial that drew the common part
    // the x where that running sum first exceeds its t (the last one if
    // rounding leaves none).  The warp looks up the rows of all its lanes
    // that ask, 32 entries at a time, and hands the hits to their lanes in
    // order.  A lane on its own made up to 64 dependent look-ups, with 4 of
    // 32 lanes active on average (GB300, s20, 262,144 walkers x 40
    // hops: 8.4 -> 5.3 ms).
    Accept acc;
    acc.rec_ok = false;
    acc.h = -1.0f;
    if (kTrials && ALG == ALGO_PAGERANK2) {
      const bool find = plan == PLAN_COMMON;
      const int32_t len = widx >= 0 && pick == -2 && (find || sum_common) ? c.pe - c.ps : 0;
      if (__any_sync(kFull, len > 0)) {
        int32_t incl = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int32_t y = __shfl_up_sync(kFull, incl, o);
          if (lane >= o) incl += y;
        }
        const int32_t items = __shfl_sync(kFull, incl, 31);
        const float t = find ? h_ret : CUDART_INF_F;
        float run = 0.0f;
        bool done = false;
        for (int32_t p0 = 0; p0 < items; p0 += 32) {
          const int32_t p = p0 + lane;
          int own = 0;  // owner of item p: the first lane whose running total exceeds p
#pragma unroll
          for (int o = 16; o > 0; o >>= 1)
            if (__shfl_sync(kFull, incl, own + o - 1) <= p) own += o;
          const int32_t k = p - __shfl_sync(kFull, incl - len, own);
          const int32_t v = __shfl_sync(kFull, c.v, own), s = __shfl_sync(kFull, c.s, own),
                        d = __shfl_sync(kFull, c.d, own), ps = __shfl_sync(kFull, c.ps, own);
          const float hsc = g.h8 ? __shfl_sync(kFull, c.hsc, own) : 0.0f;
          const Job& JW = sj[NJ > 1 ? __shfl_sync(kFull, job, own) : 0];
          int32_t x = -1, pos = -1;
          float h = 0.0f;
          if (p < items) {
            uint32_t pb = 0;
            x = __ldg(g.col + ps + k);
            pos = row_lookup<true>(g, JW, v, s, s + d, x, pb);  // most x are not in N(v): the filter says so from L2
            if (pos >= 0) {
              h = load_h(g, JW, pos, hsc);
              pos -= s;
            }
            if (COUNT) {
              lc.probes += pb;
              lc.bytes += 32ull * pb + 4ull;
            }
          }
          for (unsigned hits = __ballot_sync(kFull, pos >= 0); hits != 0u; hits &= hits - 1u) {
            const int i = __ffs(hits) - 1;
            const int to = __shfl_sync(kFull, own, i);
            const float hx = __shfl_sync(kFull, h, i);
            const int32_t ux = __shfl_sync(kFull, x, i), kx = __shfl_sync(kFull, pos, i);
            if (lane == to && !done) {
              run = __fadd_rn(run, hx);
              done = t < run;
              acc.node = ux;
              acc.k = kx;
              acc.h = hx;
            }
          }
        }
        if (len > 0 && find) {
          pick = acc.k;
          node = acc.node;
          if (COUNT) lc.rjs_steps++;
        } else if (len > 0) {
          h_ret = run;
          acc.h = -1.0f;
          const float dsl = c.n0 >= 0 ? __fmul_rn(0.25f, (float)(c.d + 3 * c.n0 + c.n1)) : (float)c.d;
          const float wc = __fmul_rn(__fsub_rn(c.w1, c.w2), h_ret);
          beta = wc / (wc + dsl * B);
        }
      }
    }
    // ------------------------------------------------------------ eRJS trials and lane eRVS positions
    int32_t ent = -2;  // position drawn by eRVS / exact in the row (grouped metapath: label segment); -1: dead end
    const int32_t lane_rvs = !kLaneRvs ? kLaneNone
                             : plan == PLAN_RVS_T ? kLaneJump
                             : (plan == PLAN_RVS_W && c.d <= kLaneKeyedMax) ? kLaneKeyed : kLaneNone;
    if (kTrials && widx >= 0 && pick == -2 && (plan == PLAN_RJS || lane_rvs != kLaneNone)) {
      const bool rvs = lane_rvs != kLaneNone;
      int32_t nt = J.round, budget = kNoTrialBudget;
      if (!rvs && nt >= J.rjs_cap - trials) {  // every budget is at least rjs_cap
        budget = trial_budget(J, grp ? c.pe - c.ps : c.d);
        nt = min(nt, budget - trials);
      }
      if (rjs_trials<COUNT, ALG, kLaneRvs>(g, J, c, B, split, beta, pos_ret, h_ret, trials, nt, acc, lc, csplit, beta2,
                                           grp, lane_rvs)) {
        if (rvs) {
          ent = pos_ret;
          if (COUNT) lc.rvs_steps++;
        } else if (ALG == ALGO_PAGERANK2 && acc.k == kPickCommon) {
          plan = PLAN_COMMON;
          h_ret = acc.h;
        } else {
          pick = acc.k;
          node = acc.node;
          if (COUNT) lc.rjs_steps++;
        }
      } else {
        trials += nt;
        if (trials >= budget) {
          plan = ((grp ? c.pe - c.ps : c.d) <= J.lane_max) ? PLAN_RVS_T : PLAN_RVS_W;
          trials = 0;
          split = csplit = false;
          if (COUNT) lc.handoffs++;
        }
      }
    }
    // ------------------------------------------------------------ single-lane eRVS / exact
    if (kRvs && !kLaneRvs && widx >= 0 && pick == -2 && plan == PLAN_RVS_T) {
      const bool jump = !(J.flags & FW_FLAG_RVS_NOJUMP);
      if ((FW_ALGO(J) == ALGO_METAPATH) && grp) {
        StepCtx cg = c;
        cg.s = c.ps;
        cg.d = c.pe - c.ps;
        ent = rvs_pick<1, COUNT, ALG, true>(g, J, cg, 0, jump, lc);
      } else {
        ent = rvs_pick<1, COUNT, ALG>(g, J, c, 0, jump, lc);
      }
      if (COUNT) lc.rvs_steps++;
    }
    if (kExact && widx >= 0 && pick == -2 && plan == PLAN_EXACT_T) {
      const float u = u01(philox(make_uint4(c.wid, (uint32_t)c.step, 0u, 0u), J.key0, J.key1).x);
      ent = exact_pick<1, COUNT, ALG>(g, J, c, 0, u, lc);
      if (COUNT) lc.exact_steps++;
    }
    // ------------------------------------------------------------ warp hand-off
    unsigned wm = __ballot_sync(kFull, widx >= 0 && pick == -2 && ent == -2 && lane_rvs == kLaneNone && (plan == PLAN_RVS_W || plan == PLAN_EXACT_W));
    while (wm != 0u) {
      const int src = __ffs(wm) - 1;
      wm &= wm - 1u;
      StepCtx w;
      w.v = __shfl_sync(kFull, c.v, src);
      w.vp = __shfl_sync(kFull, c.vp, src);
      w.s = __shfl_sync(kFull, c.s, src);
      w.d = __shfl_sync(kFull, c.d, src);
      w.ps = __shfl_sync(kFull, c.ps, src);
      w.pe = __shfl_sync(kFull, c.pe, src);
      w.step = __shfl_sync(kFull, c.step, src);
      w.wid = __shfl_sync(kFull, c.wid, src);
      if (ALG == ALGO_PAGERANK2) {
        w.w1 = __shfl_sync(kFull, c.w1, src);
        w.w2 = __shfl_sync(kFull, c.w2, src);
      }
      w.hsc = g.h8 ? __shfl_sync(kFull, c.hsc, src) : 0.0f;
      const int jb = __shfl_sync(kFull, job, src);
      const int pl = __shfl_sync(kFull, plan, src);
      bool wg = false;
      if (ALG == ALGO_METAPATH) wg = __shfl_sync(kFull, (int)grp, src) != 0;
      const Job& JW = sj[jb];
      int32_t k;
      const int32_t hd = (ALG == ALGO_METAPATH && wg) ? w.pe - w.ps : w.d;
      if (!kRvs || (kExact && pl == PLAN_EXACT_W)) {
        const float u = u01(philox(make_uint4(w.wid, (uint32_t)w.step, 0u, 0u), JW.key0, JW.key1).x);
        k = exact_pick<32, COUNT, ALG>(g, JW, w, lane, u, lc);
      } else if (hd >= kHubMinDeg && hub_chunks(hd) <= kHubMaxChunks) {
        StepCtx cw = w;
        if (ALG == ALGO_METAPATH && wg) {
          cw.s = w.ps;
          cw.d = hd;
        }
        k = hub_step<COUNT, ALG, SHARE>(g, sj, JW, cw, jb, wg, hb, err, lc);
      } else if (ALG == ALGO_METAPATH && wg) {
        StepCtx cg = w;
        cg.s = w.ps;
        cg.d = w.pe - w.ps;
        k = rvs_pick<32, COUNT, ALG, true>(g, JW, cg, lane, !(JW.flags & FW_FLAG_RVS_NOJUMP), lc);
      } else {
        k = rvs_pick<32, COUNT, ALG>(g, JW, w, lane, !(JW.flags & FW_FLAG_RVS_NOJUMP), lc);
      }
      if (lane == src) {
        ent = k;
        if (COUNT) {
          if (pl == PLAN_EXACT_W) lc.exact_steps++;
          else lc.rvs_steps++;
        }
      }
    }
    // ------------------------------------------------------------ trials together
    // A step that failed that many trials will most likely fail as many
    // again: the warp makes its next trials 32 at a time (trial t draws from
    // its own counter, so the first accepted one is the one the lane would
    // have come to) until one is accepted or the budget ends.
    if (COOP) {
      unsigned cm = __ballot_sync(kFull, widx >= 0 && pick == -2 && plan == PLAN_RJS && trials >= kTogetherFrom<ALG>);
      while (cm != 0u) {
        const int src = __ffs(cm) - 1;
        cm &= cm - 1u;
        StepCtx w;
        w.v = __shfl_sync(kFull, c.v, src);
        w.vp = __shfl_sync(kFull, c.vp, src);
        w.s = __shfl_sync(kFull, c.s, src);
        w.d = __shfl_sync(kFull, c.d, src);
        w.ps = __shfl_sync(kFull, c.ps, src);
        w.pe = __shfl_sync(kFull, c.pe, src);
        w.step = __shfl_sync(kFull, c.step, src);
        w.wid = __shfl_sync(kFull, c.wid, src);
        w.n0 = __shfl_sync(kFull, c.n0, src);
        w.n1 = __shfl_sync(kFull, c.n1, src);
        w.hsc = g.h8 ? __shfl_sync(kFull, c.hsc, src) : 0.0f;
        if (ALG == ALGO_PAGERANK2) {
          w.w1 = __shfl_sync(kFull, c.w1, src);
          w.w2 = __shfl_sync(kFull, c.w2, src);
        }
        if (ALG == ALGO_METAPATH) {
          w.gcls.x = __shfl_sync(kFull, c.gcls.x, src);
          w.gcls.y = __shfl_sync(kFull, c.gcls.y, src);
          w.gcls.z = __shfl_sync(kFull, c.gcls.z, src);
          w.gcls.w = __shfl_sync(kFull, c.gcls.w, src);
        }
        const Job& JW = sj[NJ > 1 ? __shfl_sync(kFull, job, src) : 0];
        const float wB = __shfl_sync(kFull, B, src), wh = __shfl_sync(kFull, h_ret, src);
        float wbeta = __shfl_sync(kFull, beta, src), wbeta2 = __shfl_sync(kFull, beta2, src);
        int32_t wpos = __shfl_sync(kFull, pos_ret, src);
        const int fl = __shfl_sync(kFull, (split ? 1 : 0) | (csplit ? 2 : 0) | (grp ? 4 : 0), src);
        const int32_t dd = (fl & 4) ? w.pe - w.ps : w.d;
        const int32_t budget = trial_budget(JW, dd);
        int32_t t = __shfl_sync(kFull, trials, src);
        unsigned hit = 0;
        Accept wa;
        wa.rec_ok = false;
        wa.k = -2;
        wa.node = -1;
        wa.h = -1.0f;
        wa.rec = make_int4(0, 0, 0, 0);
        wa.rec_n0 = wa.rec_n1 = 0;
        while (hit == 0u && t < budget) {
          const bool got = lane < budget - t &&
                           rjs_trials<COUNT, ALG, false>(g, JW, w, wB, (fl & 1) != 0, wbeta, wpos, wh, t + lane, 1, wa, lc,
                                                         (fl & 2) != 0, wbeta2, (fl & 4) != 0);
          hit = __ballot_sync(kFull, got);
          t += min(32, budget - t);
        }
        const int win = hit ? __ffs(hit) - 1 : 0;
        wa.k = __shfl_sync(kFull, wa.k, win);
        wa.node = __shfl_sync(kFull, wa.node, win);
        wa.h = __shfl_sync(kFull, wa.h, win);
        wa.rec.x = __shfl_sync(kFull, wa.rec.x, win);
        wa.rec.y = __shfl_sync(kFull, wa.rec.y, win);
        wa.rec.z = __shfl_sync(kFull, wa.rec.z, win);
        wa.rec.w = __shfl_sync(kFull, wa.rec.w, win);
        wa.rec_n0 = __shfl_sync(kFull, wa.rec_n0, win);
        wa.rec_n1 = __shfl_sync(kFull, wa.rec_n1, win);
        wa.rec_ok = __shfl_sync(kFull, (int)wa.rec_ok, win) != 0;
        if (lane == src) {
          if (hit == 0u) {
            plan = dd <= J.lane_max ? PLAN_RVS_T : PLAN_RVS_W;
            trials = 0;
            split = csplit = false;
            if (COUNT) lc.handoffs++;
          } else if (ALG == ALGO_PAGERANK2 && wa.k == kPickCommon) {
            plan = PLAN_COMMON;
            h_ret = wa.h;
          } else {
            acc = wa;
            pick = wa.k;
            node = wa.node;
            if (COUNT) lc.rjs_steps++;
          }
        }
      }
    }
    // ------------------------------------------------------------ entry drawn -> node and its record
    // One 32-byte edge record gives the node, its node record and h of the
    // edge, as an accepted trial does: the column, the node record and the
    // search for v' of the next node2vec plan were up to six more dependent
    // accesses per eRVS hop (GB300, s22 p = 1/4, q = 4: 55.9 -> 49.4 ms).
    if (ent >= 0) {
      const bool in_group = ALG == ALGO_METAPATH && grp;
      int4 a, b;
      ld_record((in_group ? g.gerec + 2ll * (c.ps + ent) : g.erec + 2ll * (c.s + ent)), a, b);
      if (COUNT) lc.bytes += 32;
      pick = in_group ? b.z : ent;
      node = a.x;
      acc.rec = make_int4(a.z, a.w, b.x, b.y);
      acc.rec_n0 = in_group ? 0 : (int32_t)((uint32_t)b.z >> 8);  // grouped metapath plans without weight classes
      acc.rec_n1 = in_group ? 0 : b.w;
      acc.rec_ok = true;
      acc.h = J.weighted ? __int_as_float(a.y) : 1.0f;
    } else if (ent == -1) {
      pick = -1;
    }
    // ------------------------------------------------------------ commit
    if (widx >= 0 && pick != -2) {
      const int32_t end = (J.kind == JOB_WALK) ? J.len : J.hstep + 1;
      if (J.kind == JOB_WALK) {
        int32_t* row = J.out + (long long)widx * (J.len + 1);
        if (pick >= 0) {
          stage_put(obuf, tid, row, c.step + 1, node, c.step + 1 == end);
        } else {
          stage_fill_minus_one(obuf, tid, row, c.step + 1, J.len + 1);
        }
      } else if (pick >= 0) {
        atomicAdd(J.hist + pick, 1ull);
      }
      plan = PLAN_NONE;
      if (pick >= 0) {
        c.vp = c.v;
        c.v = node;
        c.ps = c.s;
        c.pe = c.s + c.d;
        ++c.step;
        h_ret = acc.h;
        if (acc.rec_ok) {
          c.s = acc.rec.x;
          c.d = acc.rec.y;
          c.n0 = acc.rec_n0;
          c.n1 = acc.rec_n1;
          B = __int_as_float(acc.rec.z);
          beta = __int_as_float(acc.rec.w);
          plan = PLAN_READY;
        }
        if (COUNT) {
          lc.hops++;
          lc.bytes += 4;
        }
        if (c.step >= end) widx = -1;
      } else {
        if (COUNT) lc.dead_ends++;
        widx = -1;
      }
    }
  }
}

// A warp with no walker left stops counting among the block's walking warps
// and, while any still walk, scans chunks of their hub steps (sleeping
// between checks).  Lingering is optional help: nothing waits for it, and the
// bound only caps how long a warp stays.
template <bool COUNT, int ALG>
__device__ __forceinline__ void hub_linger(const DevGraph& g, const Job* sj, HubBlock* hb, LaneCounters& lc) {
  if ((threadIdx.x & 31) == 0) atomicSub(&hb->live, 1);
  for (uint32_t it = 0; it < kLingerLimit; ++it) {
    if (hub_help<COUNT, ALG>(g, sj, hb, lc)) continue;
    if (__shfl_sync(kFull, *reinterpret_cast<volatile int32_t*>(&hb->live), 0) <= 0) break;
    __nanosleep(256);
  }
}

// Per-warp sums of the lane counters, added once to the device counters.
__device__ __forceinline__ void flush_counters(const LaneCounters& lc, DevCounters* cnt) {
  const int lane = threadIdx.x & 31;
  const unsigned long long v[11] = {lc.hops,     lc.rjs_steps, lc.rvs_steps, lc.exact_steps,
                                    lc.handoffs, lc.rjs_trials, lc.rvs_items, lc.rvs_keys,
                                    lc.probes,   lc.dead_ends, lc.bytes};
  unsigned long long* dst = reinterpret_cast<unsigned long long*>(cnt);
#pragma unroll
  for (int f = 0; f < 11; ++f) {
    unsigned long long x = v[f];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
    if (lane == 0 && x) atomicAdd(dst + f, x);
  }
}

// Copy a job table into shared memory (all threads of the block).
__device__ __forceinline__ void load_jobs(const Job* src_jobs, int njobs, Job* sj) {
  const int words = njobs * (int)(sizeof(Job) / 4);
  const int* src = reinterpret_cast<const int*>(src_jobs);
  int* dst = reinterpret_cast<int*>(sj);
  for (int i = threadIdx.x; i < words; i += blockDim.x) dst[i] = src[i];
}

// Single-job (or one-algorithm) launch: one walk loop per warp over the
// launch's queue.  SHARE: idle warps linger to
// help the block's hub steps.
template <int NJ, bool COUNT, int ALG, bool SPREAD = false, bool SHARE = false, bool COOP = false, int ONLY = kAny>
__global__ void __launch_bounds__(kBlock, (kMinBlocks<ALG, SPREAD, SHARE, COOP, ONLY>)) walk_kernel(const __grid_constant__ DevGraph g,
                                                      const __grid_constant__ JobTableN<NJ> tab, int njobs, long long total,
                                                      int wpw, unsigned long long* __restrict__ qctr,
                                                      unsigned* __restrict__ err, DevCounters* __restrict__ cnt) {
  __shared__ Job table[NJ > 1 ? NJ : 1];
  __shared__ int32_t obuf[kStageSlots * kBlock];
  __shared__ HubBlock hb;
  // a single job is read where it lies, in the kernel's parameters: constant operands instead of shared-memory loads
  const Job* sj = NJ > 1 ? table : tab.jobs;
  if (NJ > 1) load_jobs(tab.jobs, njobs, table);
  if (SHARE && threadIdx.x < kHubTasks) hb.task[threadIdx.x].word = 0u;
  if (SHARE && threadIdx.x == 0) {
    hb.open = 0;
    hb.live = (int32_t)(blockDim.x >> 5);
  }
  __syncthreads();
  LaneCounters lc;
  lc.zero();
  walk_loop<NJ, COUNT, ALG, SPREAD, SHARE, COOP, ONLY>(g, sj, njobs, total, wpw, qctr, err, obuf, &hb, lc);
  if (SHARE) hub_linger<COUNT, ALG>(g, sj, &hb, lc);
  if (COUNT) flush_counters(lc, cnt);
}

// The kernel variants of one algorithm.  A launch takes its kernel, its
// occupancy and its priming from this one list, so that none of them can be
// first loaded inside a stream capture or a served wave.
enum WalkVariant : int {
  V_COUNTING = 0,     // queued, with the counters
  V_QUEUED,           // full warps that fetch from the queue
  V_QUEUED_TOGETHER,  // the same, with trials together
  V_QUEUED_WHOLE,     // the same, short eRVS rows scanned at once (node2vec; elsewhere V_QUEUED does that)
  V_QUEUED_DENSE,     // the same, 5 blocks per SM (weighted; elsewhere V_QUEUED)
  V_SPREAD,           // walkers given by place
  V_SPREAD_TOGETHER,  // the same, with trials together
  V_SPREAD_SHARE,     // the same, with hub sharing
  V_SPREAD_RVS,       // forced eRVS only
  V_SPREAD_EXACT,     // exact mode only
  kWalkVariants
};

template <int NJ>
using WalkKernel = void (*)(DevGraph, JobTableN<NJ>, int, long long, int, unsigned long long*, unsigned*, DevCounters*);

template <int NJ, int ALG>
inline WalkKernel<NJ> walk_variant(int v) {
  switch (v) {
    case V_COUNTING: return walk_kernel<NJ, true, ALG>;
    case V_QUEUED_TOGETHER: return walk_kernel<NJ, false, ALG, false, false, true>;
    case V_QUEUED_WHOLE: return walk_kernel<NJ, false, ALG, false, false, false, ALG == ALGO_NODE2VEC ? kWhole : kAny>;
    case V_QUEUED_DENSE: return walk_kernel<NJ, false, ALG, false, false, false, ALG == ALGO_WEIGHTED ? kDense : kAny>;
    case V_SPREAD: return walk_kernel<NJ, false, ALG, true>;
    case V_SPREAD_TOGETHER: return walk_kernel<NJ, false, ALG, true, false, true>;
    case V_SPREAD_SHARE: return walk_kernel<NJ, false, ALG, true, true>;
    case V_SPREAD_RVS: return walk_kernel<NJ, false, ALG, true, false, false, kOnlyRvs>;
    case V_SPREAD_EXACT: return walk_kernel<NJ, false, ALG, true, false, false, kOnlyExact>;
    default: return walk_kernel<NJ, false, ALG>;
  }
}

// Resident blocks per SM of a variant; the first call loads its kernel.
template <int NJ, int ALG>
inline cudaError_t walk_blocks_per_sm(int v, int* out) {
  static std::atomic<int> cached[kWalkVariants];
  int b = cached[v].load();
  if (b == 0) {
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, walk_variant<NJ, ALG>(v), kBlock, 0);
    if (e != cudaSuccess) return e;
    b = b > 0 ? b : 1;
    cached[v].store(b);
  }
  *out = b;
  return cudaSuccess;
}

// Hub sharing pays where warps would idle: launches that fill at most 1/8
// of the resident lanes, with eRVS forced (in the cost model's choice hub
// rows go to eRJS almost always) on a graph with hub rows.  The lingering
// code costs the loop about 13 % per step (measured on R-MAT s22), so big
// launches and the cost model's walks use the kernel without it; the rows
// are the same either way.
inline bool hub_share_pays(const fw_graph* g, const Job* jobs, int njobs, long long total, long long lanes) {
  if (g->max_degree < kHubMinDeg || total * 8 > lanes) return false;
  bool rvs = false;
  for (int i = 0; i < njobs; ++i) {
    if (jobs[i].flags & FW_FLAG_NO_HUB_SHARE) return false;
    rvs = rvs || jobs[i].mode == MODE_RVS;
  }
  return rvs;
}

// The shape of one launch.  While every walker can have a lane of its own, and
// no other launches run beside, walkers go to their warps by place, `wpw` to a
// warp (the other lanes stay idle): a warp pays for the longest of its lanes'
// paths in every iteration and scans its lanes' long rows one after another, so
// walkers are spread over the resident warps before they share one, and blocks
// fill before warps do (place_walkers).  No queue counter is needed then.
// Jobs that only scan rows (forced eRVS, exact mode) keep fewer walkers per
// warp (see scan_walkers_per_warp), the rest in the queue: the warp works for
// one walker with a long row at a time anyway, and a warp's lot of 14 made some
// warps run long after the others (65,536 walkers x 20 hops, s18: 12.9 ms with
// wpw 14, 11.8 with 4, 11.2 with 2, 10.9 with 1, 8.2 in the variant that holds
// only eRVS; without exact mode's code the others gain too: metapath s21 1.32
// -> 1.31 ms, second-order PageRank s20 4.36 -> 4.24, 5,003 walkers 351 -> 338
// us).  Other launches: full warps that fetch from the queue.  Measured on
// GB300 (R-MAT s18 / s20, one launch of full warps from a queue -> spread): 37
// walkers x 10 hops 86 -> 28 us, 5,003 x 63 hops 1,152 -> 388 us, 65,536 x 20
// hops of eRVS 22.4 -> 13.5 ms.  A kernel variant of its own, because the same
// choice made inside the queued kernel's fetch cost the whole-graph walks 1 to
// 3 %.
//
// Below this cost ratio, as tuning picks it, eRVS steps are rare and node2vec
// keeps whole scans, as the code of scans in step costs the trials registers:
// in step / whole (ms), s22 p = 1/4, q = 4 at r = 1/4 26.6 / 24.1, 1 27.2 /
// 25.1, 1.5 28.0 / 27.6, 2 28.9 / 30.0, 4 33.7 / 40.8; s20 p = 4, q = 1/4 at
// r = 1/4 4.80 / 4.20, 1 3.67 / 3.63, 1.5 3.90 / 4.05, 2 4.17 / 4.53.
// So do walks with q = 1, whose scans need no membership test, at any ratio:
// 200,000 to 2,000,000 walkers x 4 / 10 / 30 hops, s12 to s21, r = 4, speed
// against the earlier kernel, in step and whole: p = 4 no weights 0.82 / 0.87 /
// 0.90 and 1.13 / 1.11 / 1.08, U(0,1] 1.02 / 1.07 / 1.07 and 1.14 / 1.17 / 1.15;
// p = 1/2 no weights 1.02 / 1.04 / 1.06 and 1.40 / 1.37 / 1.32, 8-bit weights
// 0.99 / 0.98 / 0.98 and 1.17 / 1.17 / 1.15.
constexpr float kRareRatio = 1.5f;
// Queued weighted walks take 5 blocks per SM (48 registers) instead of 4 where
// that hides memory latency: edge records beyond L2, weights whose
// envelope is low (few trials per hop), walks that are not short, and
// fewer turns of the resident lanes.  GB300, speed against the earlier queued
// kernel with 5 / 4 blocks, x 30 hops, 500,000 walkers: U(0,1] s12 1.02 / 1.04,
// s20 1.12 / 1.05, s22 1.11 / 1.05; lognormal s20 1.00 / 1.03, s22 0.97 / 1.00;
// no weights s22 1.02 / 1.03; U(0,1] s20 300,000 walkers (two turns either way)
// 0.98 / 1.05, 800,000 x 5 hops 0.85 / 1.02.  s22, one walker per node x 80
// hops 7.04 / 7.21 ms; served queries on 8 streams 156 / 172 ms.
constexpr long long kDenseRecords = 96ll << 20;  // bytes (s17: 118 MB; L2 holds 129 MB)
constexpr double kDenseEnvelope = 2.0;
constexpr int kShortWalk = 16;  // walks of fewer hops (per walker, on average) are short
struct LaunchShape {
  int variant;  // WalkVariant
  int grid, wpw;
  bool queue;  // needs a zeroed queue counter
};

template <int NJ, int ALG>
inline cudaError_t walk_shape(const fw_graph* g, const Job* jobs, int njobs, long long total, bool count, int beside,
                              LaunchShape* s) {
  static_assert(kBlock == 32 * kShapeWarps, "place_walkers knows the block size");
  bool scans = true, reservoir = true, exact = true, trials = false, whole = true, weighted = true, histogram = true;
  long long hops = 0;
  for (int i = 0; i < njobs; ++i) {
    const bool scan = jobs[i].mode == MODE_RVS || jobs[i].mode == MODE_EXACT;
    scans = scans && scan;
    reservoir = reservoir && jobs[i].mode == MODE_RVS;
    exact = exact && jobs[i].mode == MODE_EXACT;
    trials = trials || (!scan && jobs[i].weighted);
    weighted = weighted && jobs[i].weighted;
    histogram = histogram && jobs[i].kind == JOB_HIST;
    hops += (long long)jobs[i].num_walkers * jobs[i].len;
    whole = whole && (!jobs[i].need_member || jobs[i].mode == MODE_RJS ||
                      (jobs[i].mode == MODE_AUTO && jobs[i].ratio < kRareRatio));
  }
  int bps = 1;
  cudaError_t e = walk_blocks_per_sm<NJ, ALG>(count ? V_COUNTING : V_QUEUED, &bps);
  if (e != cudaSuccess) return e;
  const long long lanes = (long long)g->num_sms * bps * kBlock;
  WalkerPlacement place = {false, 32, 0};
  s->variant = V_COUNTING;
  if (!count) {
    const double most = std::max(kTogetherHops<ALG> * g->envelope, ALG == ALGO_METAPATH ? kTogetherHopsLeast : 0.0);
    const bool together = ALG == ALGO_PAGERANK2 ? !scans && (total <= lanes || g->envelope >= kTogetherPagerank)
                                                : trials && g->envelope >= kTogetherEnvelope &&
                                                      (double)hops <= most;
    s->variant = hub_share_pays(g, jobs, njobs, total, lanes) ? V_SPREAD_SHARE
                 : reservoir                                  ? V_SPREAD_RVS
                 : exact                                      ? V_SPREAD_EXACT
                 : together                                   ? V_SPREAD_TOGETHER
                                                              : V_SPREAD;
    e = walk_blocks_per_sm<NJ, ALG>(s->variant, &bps);
    if (e != cudaSuccess) return e;
    const int fill = !scans && (ALG == ALGO_WEIGHTED || ALG == ALGO_METAPATH) ? kFirstOrderFill : kFillAll;
    const double row = reservoir && ALG == ALGO_METAPATH ? g->mean_row / kLabelStats : g->mean_row;  // eRVS: a label's share
    const bool many = total > (long long)g->num_sms * bps * kBlock;
    place = place_walkers(total, g->num_sms, bps, fill, scans, scan_walkers_per_warp(reservoir, histogram, row, many),
                          NJ > 1, beside);
    if (!place.by_place) {
      s->variant = together ? V_QUEUED_TOGETHER : ALG == ALGO_NODE2VEC && whole ? V_QUEUED_WHOLE : V_QUEUED;
      e = walk_blocks_per_sm<NJ, ALG>(s->variant, &bps);
      if (e != cudaSuccess) return e;
      if (ALG == ALGO_WEIGHTED && s->variant == V_QUEUED && weighted && 32ll * g->e >= kDenseRecords &&
          g->envelope < kDenseEnvelope && hops >= total * kShortWalk) {
        int dense = 1;
        e = walk_blocks_per_sm<NJ, ALG>(V_QUEUED_DENSE, &dense);
        if (e != cudaSuccess) return e;
        auto turns = [&](int b) { return (total + (long long)g->num_sms * b * kBlock - 1) / ((long long)g->num_sms * b * kBlock); };
        if (turns(dense) < turns(bps)) {
          s->variant = V_QUEUED_DENSE;
          bps = dense;
        }
      }
    }
  }
  if (!place.by_place)  // full warps, at most the resident blocks
    place.grid = (int)std::min<long long>((long long)g->num_sms * bps, std::max<long long>(1, (total + kBlock - 1) / kBlock));
  s->wpw = place.wpw;
  s->grid = place.grid;
  s->queue = !place.by_place || (long long)place.grid * kShapeWarps * place.wpw < total;
  return cudaSuccess;
}

// eRJS trials a lane runs per round (0 in the job: this rule; a caller's or
// a tuned rjs_batch as it is).  After a round the lanes that accepted move on
// while the others wait, so a second trial pays where most lanes fail the
// first: measured with 1 / 2 / 3 trials per round on GB300 (s20, ms), U(0,1]
// weights q = 1/4 2.30 / 2.40 / 2.61 and q = 4 5.05 / 4.88 / 5.05, metapath
// 1.52 / 1.43 / 1.47; second-order PageRank 6.09 / 5.24 / 4.97 and 4.82 with 4;
// spread launches, bound by latency, 0.369 / 0.331 / 0.326 and 0.318 with 4
// (5,003 walkers), 57 / 48 / 46 and 45 with 4 (Pareto weights); mean speed of
// 20,000 to 150,000 walkers x 5 hops with 4 / 3 / 2 against 2 from a queue:
// node2vec 1.45 / 1.43 / 1.38, x 30 hops 1.38 / 1.38 / 1.37.  node2vec queues
// with q < 1, 300,000 walkers, 1 / 2 against the earlier two: U(0,1] x 30 hops
// 1.31 / 1.33 and at 160,000 to 1,000,000 1.44 / 1.37, x 5 hops 1.12 / 1.21; no
// weights x 30 1.24 / 1.19, x 5 0.99 / 1.07; lognormal 1.16 / 1.34 and 0.95 /
// 1.16: one for long walks and a low envelope only.  q = 4 without weights x
// 30 hops 1.51 / 1.58: two.  Queues of several jobs mix lanes of q < 1 and q >
// 1 in a warp and keep 2 (64 mixed jobs: 8.54 ms, with 1 for q < 1 8.96); so do
// launches of whole scans (p = 4, q = 1/4, r = 1/4 4.20, with 1 4.28).
constexpr double kOneTrialEnvelope = 2.0;
inline int32_t round_trials(const fw_graph* g, const Job& J, int variant, int njobs) {
  if (J.round > 0) return J.round;
  if (variant >= V_SPREAD || J.algo == ALGO_PAGERANK2) return 4;
  if (njobs == 1 && variant != V_QUEUED_WHOLE && J.algo == ALGO_NODE2VEC && J.inv_q > 1.0f &&
      (!J.weighted || g->envelope < kOneTrialEnvelope) && J.len >= kShortWalk)
    return 1;
  return kRjsBatchDefault;
}

template <int NJ, int ALG>
inline cudaError_t launch_walk_t(const fw_graph* g, const Job* jobs, int njobs, long long total, bool count, int beside,
                                 unsigned long long* qctr, cudaStream_t stream) {
  LaunchShape s;
  cudaError_t e = walk_shape<NJ, ALG>(g, jobs, njobs, total, count, beside, &s);
  if (e != cudaSuccess) return e;
  if (s.queue && !qctr) return cudaErrorInvalidValue;
  if (!s.queue) qctr = nullptr;
  JobTableN<NJ> tab;
  for (int i = 0; i < njobs; ++i) {
    tab.jobs[i] = jobs[i];
    tab.jobs[i].round = round_trials(g, jobs[i], s.variant, njobs);
  }
  walk_variant<NJ, ALG>(s.variant)<<<s.grid, kBlock, 0, stream>>>(dev_graph(g), tab, njobs, total, s.wpw, qctr, g->d_err,
                                                                 g->d_cnt);
  g_launches.fetch_add(1);
  return cudaGetLastError();
}

// Load every variant of one algorithm and cache its occupancy (outside any capture).
template <int NJ, int ALG>
inline cudaError_t prime_walk() {
  cudaError_t e = cudaSuccess;
  int b;
  for (int v = 0; v < kWalkVariants && e == cudaSuccess; ++v) e = walk_blocks_per_sm<NJ, ALG>(v, &b);
  return e;
}

// The launches of one algorithm over a table of at most NJ jobs; each is
// instantiated in a source file of its own (WALK_LAUNCHES), so that they
// compile side by side.
struct WalkLaunches {
  cudaError_t (*launch)(const fw_graph* g, const Job* jobs, int njobs, long long total, bool count, int beside,
                        unsigned long long* qctr, cudaStream_t stream);
  cudaError_t (*needs_queue)(const fw_graph* g, const Job* jobs, int njobs, long long total, bool count, int beside,
                             bool* need);
  cudaError_t (*prime)();
};
const WalkLaunches& single_launches(int algo);  // one job
const WalkLaunches& table_launches(int algo);   // up to kMaxJobs jobs

template <int NJ, int ALG>
inline WalkLaunches make_launches() {
  return {launch_walk_t<NJ, ALG>,
          [](const fw_graph* g, const Job* jobs, int njobs, long long total, bool count, int beside, bool* need) {
            LaunchShape s = {};
            const cudaError_t e = walk_shape<NJ, ALG>(g, jobs, njobs, total, count, beside, &s);
            *need = s.queue;
            return e;
          },
          prime_walk<NJ, ALG>};
}

#define WALK_LAUNCHES(NAME, NJ, ALG)                             \
  namespace fw {                                                 \
  const WalkLaunches& NAME() {                                   \
    static const WalkLaunches launches = make_launches<NJ, ALG>(); \
    return launches;                                             \
  }                                                              \
  }
}  // namespace fw
