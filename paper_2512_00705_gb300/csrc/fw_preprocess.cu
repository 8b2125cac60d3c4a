// fw_preprocess.cu -- per-row preprocessing of a new graph: row validation,
// edge records, label statistics and groups, filters and membership tables,
// weight symmetry (Sec. 4.2 preprocess(), and the layouts of fw_device.cuh).
//
// Row lengths of the graphs this serves span five orders of magnitude, and
// with one warp per row a kernel lasts as long as its hub row's warp (R-MAT
// s20: 27.6 ms of preprocessing, of which the label groups took 14.0 and the
// tables 7.6, on 31 M entries whose records are 3 GB).  Rows are therefore
// scanned by teams of their own size: a warp up to kWarpRow entries, a block
// of 8 warps up to kBlockRow, a block of 32 warps beyond; the longer rows are
// listed by the node statistics' pass: 4.2 ms on the same graph.  Every stable
// order is kept: a team's warps own consecutive segments of the row.
#include "fw_internal.h"
#include "fw_rows.h"

namespace fw {

namespace {

constexpr int kTeamBlock = 256;  // threads of a block of one-warp teams, and of a block team

// A team of NW warps: one warp of the block, or the whole block.
template <int NW>
__device__ __forceinline__ void team_sync() {
  if (NW == 1) __syncwarp();
  else __syncthreads();
}

// Calls f(v, s, d) for every row of the team's size class with at least
// `least` entries; the whole team calls together.
template <int NW, class F>
__device__ __forceinline__ void for_rows(const int32_t* __restrict__ off, int32_t n, const RowLists& rows,
                                         int32_t least, F f) {
  if (NW == 1) {
    // kRowsAtOnce neighbouring rows per turn: their offsets come in one load, where each empty row of an R-MAT
    // graph (two in five) cost a warp the latency of its own
    const int lane = threadIdx.x & 31;
    const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long v0 = warp * kRowsAtOnce; v0 < n; v0 += nwarps * kRowsAtOnce) {
      const long long at = min(v0 + lane, (long long)n);
      const int32_t s = lane <= kRowsAtOnce ? off[at] : 0;
      const int32_t d = __shfl_down_sync(kFull, s, 1) - s;
      unsigned todo = __ballot_sync(kFull, lane < kRowsAtOnce && d >= least && d <= kWarpRow && v0 + lane < n);
      while (todo != 0u) {
        const int j = __ffs(todo) - 1;
        todo &= todo - 1u;
        f((int32_t)(v0 + j), __shfl_sync(kFull, s, j), __shfl_sync(kFull, d, j));
      }
    }
  } else {
    const int32_t* list = NW == 8 ? rows.mid : rows.big;
    const int count = rows.counts[NW == 8 ? 0 : 1];
    for (int i = blockIdx.x; i < count; i += gridDim.x) {
      const int32_t v = list[i], s = off[v];
      f(v, s, off[v + 1] - s);
      __syncthreads();  // the team's shared memory is free for its next row
    }
  }
}

// The team's warp `w` of NW owns positions [lo, hi) of a row of d entries.
template <int NW>
__device__ __forceinline__ void segment(int32_t d, int w, int32_t& lo, int32_t& hi) {
  const int32_t len = (int32_t)(((long long)d + NW * 32 - 1) / (NW * 32)) * 32;
  lo = (int32_t)min((long long)w * len, (long long)d);
  hi = (int32_t)min((long long)lo + len, (long long)d);
}

__device__ __forceinline__ void st_record(int4* p, const int4& a, const int4& b) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(a.x), "r"(a.y), "r"(a.z),
               "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w)
               : "memory");
}

// Launch the three team sizes of a row kernel on `st` (the long rows first).
template <class K1, class K8, class K32>
cudaError_t launch_teams(K1 k1, K8 k8, K32 k32, int num_sms) {
  k32(num_sms);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k8(num_sms * 8);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k1(num_sms * 8);
  g_launches.fetch_add(3);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- edge records
// Edge records (32 bytes per CSR entry): everything one eRJS trial needs and
// everything the next step's plan needs if the trial is accepted.  With
// weights (CLS) also their class-ordered copy: each row stably partitioned
// into weight classes 0 (h > h_MAX / 2), 1 (h_MAX / 4 < h <= h_MAX / 2) and 2.
// Bound by the records' stores (2 x 32 bytes per entry); the two copies come
// from one pass, so the node records are gathered once (s20: 0.38 ms for the
// records and 2.39 ms for their copy before).
template <int NW, bool CLS>
__global__ void __launch_bounds__(NW == 32 ? 1024 : kTeamBlock)
    records_kernel(const int32_t* __restrict__ off, const int32_t* __restrict__ col, const float* __restrict__ h,
                   const uint8_t* __restrict__ lab, const int4* __restrict__ nrec, int32_t n, RowLists rows,
                   int4* __restrict__ erec, int4* __restrict__ cerec) {
  __shared__ int cnt[NW][2];
  const int lane = threadIdx.x & 31, w = NW == 1 ? 0 : threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  for_rows<NW>(off, n, rows, 1, [&](int32_t v, int32_t s, int32_t d) {
    int32_t lo, hi;
    segment<NW>(d, w, lo, hi);
    float half = 0.0f, quarter = 0.0f;
    int run0 = 0, run1 = 0, run2 = 0;  // next place of each class
    if (CLS) {
      const float m = __int_as_float(nrec[2ll * v].z);
      const int4 nc = nrec[2ll * v + 1];
      half = 0.5f * m;
      quarter = 0.25f * m;
      if (NW > 1) {
        int c0 = 0, c1 = 0;
        for_entries(s + lo, hi - lo, lane, 32, [&](int32_t i) {
          const float x = h[i];
          c0 += x > half ? 1 : 0;
          c1 += x > quarter && !(x > half) ? 1 : 0;
        });
        c0 = __reduce_add_sync(kFull, c0);
        c1 = __reduce_add_sync(kFull, c1);
        if (lane == 0) {
          cnt[w][0] = c0;
          cnt[w][1] = c1;
        }
        team_sync<NW>();
        const int p0 = lane < w ? cnt[lane][0] : 0, p1 = lane < w ? cnt[lane][1] : 0;
        run0 = __reduce_add_sync(kFull, p0);
        run1 = __reduce_add_sync(kFull, p1);
        run2 = lo - run0 - run1;
      }
      run1 += nc.x;
      run2 += nc.x + nc.y;
    }
    for (uint32_t b = lo; b < (uint32_t)hi; b += 32) {
      const bool valid = b + lane < (uint32_t)hi;
      const long long i = (long long)s + b + lane;
      float x = 1.0f;
      int4 a = make_int4(0, 0, 0, 0), r = a;
      if (valid) {
        const int32_t u = col[i];
        if (h) x = h[i];
        const int lb = lab ? (int)lab[i] : 0;
        int4 nr, nc;
        ld_record(nrec + 2ll * u, nr, nc);
        // label in the low byte, the target's class-0 count above it (degrees < 2^24)
        a = make_int4(u, __float_as_int(x), nr.x, nr.y);
        r = make_int4(nr.z, nr.w, lb | (int)((unsigned)nc.x << 8), nc.y);
        st_record(erec + 2 * i, a, r);
      }
      if (CLS) {
        const int cls = (x > half) ? 0 : ((x > quarter) ? 1 : 2);
        const unsigned m0 = __ballot_sync(kFull, valid && cls == 0), m1 = __ballot_sync(kFull, valid && cls == 1),
                       m2 = __ballot_sync(kFull, valid && cls == 2);
        if (valid) {
          const int place = cls == 0 ? run0 + __popc(m0 & lt) : (cls == 1 ? run1 + __popc(m1 & lt) : run2 + __popc(m2 & lt));
          st_record(cerec + 2 * ((long long)s + place), a, r);
        }
        run0 += __popc(m0);
        run1 += __popc(m1);
        run2 += __popc(m2);
      }
    }
  });
}

// ---------------------------------------------------------------- label statistics
// Per-label node statistics {max h, sum h} over the edges of each label l <
// kLabelStats (h = 1 without weights); sets *bad if a label >= kLabelStats
// occurs (the statistics are then not used).  Lane l of a warp adds the
// entries l, l + 32, ... in order, whatever the team: a block's warps share
// the labels of a long row, not its entries, so the sums are the same ones.
template <int NW>
__global__ void __launch_bounds__(kTeamBlock)
    label_stats_kernel(const int32_t* __restrict__ off, const float* __restrict__ h, const uint8_t* __restrict__ lab,
                       int32_t n, RowLists rows, float2* __restrict__ out, unsigned* __restrict__ bad) {
  static_assert(kLabelStats == kTeamBlock / 32, "one label per warp of a block team");
  constexpr int kPer = NW == 1 ? kLabelStats : 1;  // labels per warp
  const int lane = threadIdx.x & 31;
  const int first = NW == 1 ? 0 : threadIdx.x >> 5;
  auto row = [&](int32_t v, int32_t s, int32_t d) {
    float mx[kPer], sm[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) mx[k] = sm[k] = 0.0f;
    bool over = false;
    constexpr int kAhead = NW == 1 ? 1 : 8;
    for (uint32_t b = lane; b < (uint32_t)d; b += 32 * kAhead) {
      int l[kAhead];
      float x[kAhead];
#pragma unroll
      for (int q = 0; q < kAhead; ++q) {
        const bool valid = b + 32 * q < (uint32_t)d;
        const long long i = (long long)s + b + 32 * q;
        l[q] = valid ? (int)lab[i] : -1;
        x[q] = valid && h ? h[i] : 1.0f;
      }
#pragma unroll
      for (int q = 0; q < kAhead; ++q) {
        over |= l[q] >= kLabelStats;
#pragma unroll
        for (int k = 0; k < kPer; ++k)
          if (first + k == l[q]) {
            mx[k] = fmaxf(mx[k], x[q]);
            sm[k] += x[q];
          }
      }
    }
    // butterfly over the lanes (16, 8, 4, 2, 1: the order of the plain one); with all labels in the warp, each
    // exchange also halves the labels a lane keeps, so that lanes 4 l .. 4 l + 3 end with label l
    int keep = 0;
    if (NW == 1) {
#pragma unroll
      for (int o = 16, m = kPer / 2; o >= 4; o >>= 1, m >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int k = 0; k < m; ++k) {
          const float sx = up ? mx[k] : mx[k + m], ss = up ? sm[k] : sm[k + m];
          const float kx = up ? mx[k + m] : mx[k], ks = up ? sm[k + m] : sm[k];
          mx[k] = fmaxf(kx, __shfl_xor_sync(kFull, sx, o));
          sm[k] = ks + __shfl_xor_sync(kFull, ss, o);
        }
      }
      keep = lane >> 2;
    }
#pragma unroll
    for (int o = NW == 1 ? 2 : 16; o > 0; o >>= 1) {
      mx[0] = fmaxf(mx[0], __shfl_xor_sync(kFull, mx[0], o));
      sm[0] += __shfl_xor_sync(kFull, sm[0], o);
    }
    if (NW == 1 ? (lane & 3) == 0 : lane == 0)
      out[(long long)v * kLabelStats + first + keep] = make_float2(mx[0], sm[0]);
    if (__any_sync(kFull, over) && lane == 0) atomicOr(bad, 1u);
  };
  if (NW == 1) {
    for_rows<1>(off, n, rows, 0, row);
  } else {
    for_rows<8>(off, n, rows, 0, row);
    RowLists big = rows;  // the longest rows by the same teams
    big.mid = rows.big;
    big.counts = rows.counts + 1;
    for_rows<8>(off, n, big, 0, row);
  }
}

// ---------------------------------------------------------------- label groups
// Label-grouped view (metapath): each row reordered stably by (label, weight
// class) -- labels < kLabelStats; within a label, class c < kWClasses - 1
// holds h in (M / 2^(c+1), M / 2^c] and the last class h <= M /
// 2^(kWClasses-1), M the label's max h -- by a counting pass over the
// kLabelStats * kWClasses buckets, an exclusive prefix over (bucket, warp)
// and a ranked scatter.  It writes grouped edge records (the second half's
// third word is the entry's position in the row, the fourth 0), the grouped
// h, and per label a 32-byte record {max h, sum h (from the label
// statistics), segment start, segment length}, {counts of classes 0 ..
// kWClasses-2}.  The rank among a chunk's entries of the same bucket comes
// from one match over the warp (a ballot per bucket took 40 per chunk).
template <int NW>
__global__ void __launch_bounds__(NW == 32 ? 1024 : kTeamBlock)
    label_group_kernel(const int32_t* __restrict__ off, const int32_t* __restrict__ col, const float* __restrict__ h,
                       const uint8_t* __restrict__ lab, const int4* __restrict__ nrec,
                       const float2* __restrict__ lstat, int32_t n, RowLists rows, int4* __restrict__ lrec,
                       int4* __restrict__ gerec, float* __restrict__ gh) {
  constexpr int kB = kLabelStats * kWClasses;
  static_assert(kB <= 64, "two buckets per lane");
  __shared__ int places[NW == 1 ? kTeamBlock / 32 : NW][kB];  // per warp: counts, then next place of each bucket
  const int lane = threadIdx.x & 31, wb = threadIdx.x >> 5, w = NW == 1 ? 0 : wb;
  const unsigned lt = (1u << lane) - 1u;
  int* mine = places[wb];
  for_rows<NW>(off, n, rows, 0, [&](int32_t v, int32_t s, int32_t d) {
    int32_t lo, hi;
    segment<NW>(d, w, lo, hi);
    const float2 ls = lane < kLabelStats ? lstat[(long long)v * kLabelStats + lane] : make_float2(0.0f, 0.0f);
    // bucket of an entry (kB past the segment's end)
    auto bucket = [&](int l, float x, bool valid) -> int {
      const float m = __shfl_sync(kFull, ls.x, valid ? l : 0);
      int c = 0;
      float t = 0.5f * m;
#pragma unroll
      for (int q = 0; q < kWClasses - 1; ++q) {
        c += x > t ? 0 : 1;
        t *= 0.5f;
      }
      return valid ? l * kWClasses + c : kB;
    };
    for (int q = lane; q < kB; q += 32) mine[q] = 0;
    __syncwarp();
    for (uint32_t b = lo; b < (uint32_t)hi; b += 32) {
      const bool valid = b + lane < (uint32_t)hi;
      const long long i = (long long)s + b + lane;
      const int k = bucket(valid ? (int)lab[i] : 0, valid && h ? h[i] : 1.0f, valid);
      const unsigned same = __match_any_sync(kFull, k);
      if (valid && (same & lt) == 0u) mine[k] += __popc(same);
      __syncwarp();
    }
    team_sync<NW>();
    if (w == 0) {
      // totals of buckets lane and lane + 32, their exclusive prefix, then each warp's first place
      int (*all)[kB] = NW == 1 ? places + wb : places;
      int t0 = 0, t1 = 0;
#pragma unroll 8
      for (int q = 0; q < NW; ++q) {
        t0 += all[q][lane];
        if (lane + 32 < kB) t1 += all[q][lane + 32];
      }
      int i0 = t0, i1 = t1;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, i0, o), z = __shfl_up_sync(kFull, i1, o);
        if (lane >= o) {
          i0 += y;
          i1 += z;
        }
      }
      const int total0 = __shfl_sync(kFull, i0, 31);
      const int p0 = i0 - t0, p1 = total0 + i1 - t1;
      // per-label record: lane l < kLabelStats gathers its kWClasses buckets
      int cnt[kWClasses], start = 0, len = 0;
#pragma unroll
      for (int c = 0; c < kWClasses; ++c) {
        const int q = (lane < kLabelStats ? lane : 0) * kWClasses + c;
        const int a = __shfl_sync(kFull, t0, q & 31), bb = __shfl_sync(kFull, t1, q & 31);
        const int sa = __shfl_sync(kFull, p0, q & 31), sb = __shfl_sync(kFull, p1, q & 31);
        cnt[c] = q < 32 ? a : bb;
        if (c == 0) start = q < 32 ? sa : sb;
        len += cnt[c];
      }
      if (lane < kLabelStats)
        st_record(lrec + 2 * ((long long)v * kLabelStats + lane),
                  make_int4(__float_as_int(ls.x), __float_as_int(ls.y), start, len),
                  make_int4(cnt[0], cnt[1], cnt[2], cnt[3]));
      int r0 = p0, r1 = p1;
      for (int q = 0; q < NW; ++q) {
        const int x0 = all[q][lane];
        all[q][lane] = r0;
        r0 += x0;
        if (lane + 32 < kB) {
          const int x1 = all[q][lane + 32];
          all[q][lane + 32] = r1;
          r1 += x1;
        }
      }
    }
    team_sync<NW>();
    for (uint32_t b = lo; b < (uint32_t)hi; b += 32) {
      const bool valid = b + lane < (uint32_t)hi;
      const long long i = (long long)s + b + lane;
      const float x = valid && h ? h[i] : 1.0f;
      int4 nr = make_int4(0, 0, 0, 0);
      int32_t u = 0;
      if (valid) {
        u = col[i];
        nr = __ldg(nrec + 2ll * u);
      }
      const int k = bucket(valid ? (int)lab[i] : 0, x, valid);
      const unsigned same = __match_any_sync(kFull, k);
      const int rank = __popc(same & lt);
      const int at = valid ? mine[k] + rank : 0;
      __syncwarp();
      if (valid && rank == 0) mine[k] += __popc(same);
      __syncwarp();
      if (valid) {
        const long long o = (long long)s + at;
        st_record(gerec + 2 * o, make_int4(u, __float_as_int(x), nr.x, nr.y), make_int4(nr.z, nr.w, (int)(b + lane), 0));
        gh[o] = x;
      }
    }
    __syncwarp();
  });
}

// ---------------------------------------------------------------- filters and tables
// Bloom filters and membership tables of the rows with at least
// kBloomMinDeg entries (layouts and hashing are those of row_member; the
// table may be nullptr).  An id takes the next slot of its home bucket, or of
// the first bucket after it that is not full; slots fill in order.  The
// team's shared memory holds the buckets' slot counts and the row's filter
// (one shared-memory atomic each per id, where four atomics on the filter
// and on average 2.5 compare-and-swaps on the table went to L2 before); what does not fit, above 100,000 entries the filter and above
// 200,000 the counts too, runs on global memory.
// kTableWords: shared words a team has.
// filter: blocks of 8 words, one per 32 entries and up to 2 more; counts: one per bucket, one per 4 entries and up to 2 more
template <int NW>
constexpr int kTableWords = NW == 1   ? (kWarpRow / 32 + 2) * 8 + kWarpRow / 4 + 2
                            : NW == 8 ? (kBlockRow / 32 + 2) * 8 + kBlockRow / 4 + 2
                                      : 50 * 1024;

template <int NW>
__global__ void __launch_bounds__(NW == 32 ? 1024 : kTeamBlock)
    table_kernel(const int32_t* __restrict__ off, const int32_t* __restrict__ col, int32_t n, RowLists rows,
                 uint32_t* __restrict__ bloom, int32_t* __restrict__ mtab) {
  extern __shared__ uint32_t words[];
  const int t = NW == 1 ? threadIdx.x & 31 : threadIdx.x;
  uint32_t* counts = words + (NW == 1 ? (threadIdx.x >> 5) * kTableWords<NW> : 0);
  for_rows<NW>(off, n, rows, kBloomMinDeg, [&](int32_t v, int32_t s, int32_t d) {
    const int32_t e = s + d;
    const uint32_t fw = bloom_words(s, e);
    const uint32_t tnb = table_buckets(s, e);
    uint32_t* gfilter = bloom + bloom_word0(v, s);
    int32_t* table = mtab ? mtab + 8ll * table_bucket0(v, s) : nullptr;
    const bool count_here = tnb <= (uint32_t)kTableWords<NW>;  // always, for warps and short blocks
    const bool filter_here = fw + tnb <= (uint32_t)kTableWords<NW>;
    uint32_t* bits = filter_here ? counts + tnb : gfilter;  // global filters were cleared before
    for (uint32_t i = t; i < (count_here ? tnb + (filter_here ? fw : 0u) : 0u); i += NW * 32) counts[i] = 0u;
    team_sync<NW>();
    for_entries(s, d, t, NW * 32, [&](int32_t i) {
      const int32_t u = col[i];
      const uint32_t hk = id_hash((uint32_t)u);
      atomicOr(bits + bloom_word(hk, fw), bloom_bits(hk));
      if (!table) return;
      // d < 8 * tnb ids share the row's buckets, so a free slot exists
      uint32_t b = __umulhi(hk, tnb);
      bool placed = false;
      for (uint32_t k = 0; k < tnb && !placed; ++k) {
        if (count_here) {
          const uint32_t slot = atomicAdd(counts + b, 1u);
          placed = slot < 8u;
          if (placed) table[8ll * b + slot] = u;
        } else {
          for (int q = 0; q < 8 && !placed; ++q) placed = atomicCAS(table + 8ll * b + q, -1, u) == -1;
        }
        b = (b + 1 == tnb) ? 0u : b + 1;
      }
    });
    team_sync<NW>();
    if (filter_here) {
      for (uint32_t i = t; i < fw; i += NW * 32) gfilter[i] = bits[i];
      team_sync<NW>();
    }
  });
}

// ---------------------------------------------------------------- symmetry
// Does every entry (v, u) have a mirror (u, v) of the same weight?  Of a pair
// only the entry whose target has the shorter row (equal lengths: the smaller
// id) is looked up there (*flag is set if it has no mirror); those mirrors
// are as many distinct entries of the other kind, so none of them lacks its
// own exactly when both kinds have equal counts (sides[0], sides[1]).  Bound
// by the searches' random accesses, which the short rows keep to a few; teams
// know their row (s20, all three sizes: an entry-parallel search of all
// entries 1.40 ms, teams for those above the diagonal 1.44, by the shorter
// row 1.28).
template <int NW>
__global__ void __launch_bounds__(NW == 32 ? 1024 : kTeamBlock)
    symmetry_kernel(const int32_t* __restrict__ off, const int32_t* __restrict__ col, const float* __restrict__ h,
                    int32_t n, RowLists rows, unsigned* __restrict__ flag, unsigned long long* __restrict__ sides) {
  const int t = NW == 1 ? threadIdx.x & 31 : threadIdx.x;
  unsigned long long taken = 0, left = 0;
  bool missing = false;
  for_rows<NW>(off, n, rows, 1, [&](int32_t v, int32_t s, int32_t d) {
    for_entries(s, d, t, NW * 32, [&](int32_t i) {
      const int32_t u = col[i];
      if (u == v) return;  // its own mirror
      const int32_t us = off[u], ue = off[u + 1];
      if (ue - us > d || (ue - us == d && u > v)) {
        ++left;
        return;
      }
      ++taken;
      uint32_t pb = 0;
      const int32_t j = row_find(col, us, ue, v, n, pb);
      missing |= j < 0 || (h && h[j] != h[i]);
    });
  });
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    taken += __shfl_xor_sync(kFull, taken, o);
    left += __shfl_xor_sync(kFull, left, o);
  }
  missing = __any_sync(kFull, missing);
  if ((threadIdx.x & 31) == 0) {
    if (missing) atomicOr(flag, 1u);
    if (taken) atomicAdd(sides, taken);
    if (left) atomicAdd(sides + 1, left);
  }
}

// ---------------------------------------------------------------- validation
// Columns, row order and weights of device-resident input, one thread per
// entry (the offsets are valid): bit 2 = column range, bit 4 = row order, bit
// 8 = weights.  An entry that does not exceed its predecessor must begin a
// row: only such entries, about one per row, search the offsets.
__global__ void check_rows_kernel(const int32_t* __restrict__ off, const int32_t* __restrict__ col,
                                  const float* __restrict__ h, int32_t n, long long e, unsigned* __restrict__ err) {
  unsigned bits = 0;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < e; i += (long long)gridDim.x * blockDim.x) {
    const int32_t c = col[i];
    if (c < 0 || c >= n) bits |= 2u;
    if (h) {
      const float x = h[i];
      if (!(x > 0.0f) || !isfinite(x)) bits |= 8u;
    }
    if (i > 0 && c <= col[i - 1]) {
      int32_t lo = 0, hi = n;  // first v with off[v] >= i: does a row begin at i?
      while (lo < hi) {
        const int32_t mid = lo + ((hi - lo) >> 1);
        if (__ldg(off + mid) < i) lo = mid + 1;
        else hi = mid;
      }
      if (__ldg(off + lo) != i) bits |= 4u;
    }
  }
  if (bits) atomicOr(err, bits);
}

template <int NW>
cudaError_t table_smem(size_t* bytes) {
  *bytes = sizeof(uint32_t) * (size_t)kTableWords<NW> * (NW == 1 ? kTeamBlock / 32 : 1);
  return cudaFuncSetAttribute(table_kernel<NW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)*bytes);
}

}  // namespace

size_t row_list_words(long long e) { return (size_t)(e / kWarpRow + e / kBlockRow) + 4; }

RowLists row_lists(int32_t* scratch, long long e) {
  RowLists r;
  r.counts = scratch;
  r.mid = scratch + 2;
  r.big = r.mid + e / kWarpRow + 1;
  return r;
}

cudaError_t launch_edge_records(const int32_t* off, const int32_t* col, const float* h, const uint8_t* lab,
                                const int4* nrec, int32_t n, const RowLists& rows, int4* erec, int4* cerec,
                                int num_sms, cudaStream_t st) {
  if (cerec)
    return launch_teams([&](int b) { records_kernel<1, true><<<b, kTeamBlock, 0, st>>>(off, col, h, lab, nrec, n, rows, erec, cerec); },
                        [&](int b) { records_kernel<8, true><<<b, kTeamBlock, 0, st>>>(off, col, h, lab, nrec, n, rows, erec, cerec); },
                        [&](int b) { records_kernel<32, true><<<b, 1024, 0, st>>>(off, col, h, lab, nrec, n, rows, erec, cerec); },
                        num_sms);
  return launch_teams([&](int b) { records_kernel<1, false><<<b, kTeamBlock, 0, st>>>(off, col, h, lab, nrec, n, rows, erec, cerec); },
                      [&](int b) { records_kernel<8, false><<<b, kTeamBlock, 0, st>>>(off, col, h, lab, nrec, n, rows, erec, cerec); },
                      [&](int b) { records_kernel<32, false><<<b, 1024, 0, st>>>(off, col, h, lab, nrec, n, rows, erec, cerec); },
                      num_sms);
}

cudaError_t launch_label_group(const int32_t* off, const int32_t* col, const float* h, const uint8_t* lab,
                               const int4* nrec, const float2* lstat, int32_t n, const RowLists& rows, int4* lrec,
                               int4* gerec, float* gh, int num_sms, cudaStream_t st) {
  return launch_teams(
      [&](int b) { label_group_kernel<1><<<b, kTeamBlock, 0, st>>>(off, col, h, lab, nrec, lstat, n, rows, lrec, gerec, gh); },
      [&](int b) { label_group_kernel<8><<<b, kTeamBlock, 0, st>>>(off, col, h, lab, nrec, lstat, n, rows, lrec, gerec, gh); },
      [&](int b) { label_group_kernel<32><<<b, 1024, 0, st>>>(off, col, h, lab, nrec, lstat, n, rows, lrec, gerec, gh); },
      num_sms);
}

cudaError_t launch_label_stats(const int32_t* off, const float* h, const uint8_t* lab, int32_t n,
                               const RowLists& rows, float2* out, unsigned* bad, int num_sms, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  label_stats_kernel<8><<<num_sms * 8, kTeamBlock, 0, st>>>(off, h, lab, n, rows, out, bad);
  label_stats_kernel<1><<<num_sms * 8, kTeamBlock, 0, st>>>(off, h, lab, n, rows, out, bad);
  g_launches.fetch_add(2);
  return cudaGetLastError();
}

cudaError_t launch_symmetry(const int32_t* off, const int32_t* col, const float* h, int32_t n, const RowLists& rows,
                            unsigned* flag, unsigned long long* sides, int num_sms, cudaStream_t st) {
  return launch_teams(
      [&](int b) { symmetry_kernel<1><<<b, kTeamBlock, 0, st>>>(off, col, h, n, rows, flag, sides); },
      [&](int b) { symmetry_kernel<8><<<b, kTeamBlock, 0, st>>>(off, col, h, n, rows, flag, sides); },
      [&](int b) { symmetry_kernel<32><<<2 * b, 1024, 0, st>>>(off, col, h, n, rows, flag, sides); }, num_sms);
}

size_t bloom_bytes(int32_t n, long long e) { return 32ull * (size_t)((e >> 5) + (long long)n + 1); }
size_t table_bytes(int32_t n, long long e) { return 32ull * (size_t)((e >> 2) + (long long)n + 1); }

cudaError_t launch_bloom(const int32_t* off, const int32_t* col, int32_t n, long long e, const RowLists& rows,
                         uint32_t* bloom, int32_t* mtab, int num_sms, cudaStream_t st) {
  cudaError_t err = cudaMemsetAsync(bloom, 0, bloom_bytes(n, e), st);
  if (err == cudaSuccess && mtab) err = cudaMemsetAsync(mtab, 0xff, table_bytes(n, e), st);
  if (err != cudaSuccess || n == 0) return err;
  size_t m1 = 0, m8 = 0, m32 = 0;
  err = table_smem<1>(&m1);
  if (err == cudaSuccess) err = table_smem<8>(&m8);
  if (err == cudaSuccess) err = table_smem<32>(&m32);
  if (err != cudaSuccess) return err;
  return launch_teams([&](int b) { table_kernel<1><<<b, kTeamBlock, m1, st>>>(off, col, n, rows, bloom, mtab); },
                      [&](int b) { table_kernel<8><<<b, kTeamBlock, m8, st>>>(off, col, n, rows, bloom, mtab); },
                      [&](int b) { table_kernel<32><<<b, 1024, m32, st>>>(off, col, n, rows, bloom, mtab); }, num_sms);
}

cudaError_t launch_check_rows(const int32_t* off, const int32_t* col, const float* h, int32_t n, long long e,
                              unsigned* err, int num_sms, cudaStream_t st) {
  if (n == 0 || e == 0) return cudaSuccess;
  const long long want = (e + 255) / 256;
  const int grid = (int)(want < (long long)num_sms * 16 ? want : (long long)num_sms * 16);
  check_rows_kernel<<<grid, 256, 0, st>>>(off, col, h, n, e, err);
  g_launches.fetch_add(1);
  return cudaGetLastError();
}

cudaError_t prime_preprocess_kernels() {
  cudaFuncAttributes a;
  const void* all[] = {(const void*)records_kernel<1, true>,   (const void*)records_kernel<8, true>,
                       (const void*)records_kernel<32, true>,  (const void*)records_kernel<1, false>,
                       (const void*)records_kernel<8, false>,  (const void*)records_kernel<32, false>,
                       (const void*)label_stats_kernel<1>,     (const void*)label_stats_kernel<8>,
                       (const void*)label_group_kernel<1>,     (const void*)label_group_kernel<8>,
                       (const void*)label_group_kernel<32>,    (const void*)table_kernel<1>,
                       (const void*)table_kernel<8>,           (const void*)table_kernel<32>,
                       (const void*)symmetry_kernel<1>,        (const void*)symmetry_kernel<8>,
                       (const void*)symmetry_kernel<32>};
  for (const void* k : all) {
    const cudaError_t e = cudaFuncGetAttributes(&a, k);
    if (e != cudaSuccess) return e;
  }
  return prime_node_stats();
}

}  // namespace fw
