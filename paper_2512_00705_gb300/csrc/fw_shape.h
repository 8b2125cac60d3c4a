// fw_shape.h -- where the walkers of one launch go: how many share a warp and
// how many blocks are launched (host code without CUDA, tested on the CPU).
#pragma once

#include <algorithm>

namespace fw {

constexpr int kShapeWarps = 8;  // warps per block

// Beside other launches, a launch whose share gives a warp more walkers than
// this takes full warps from the queue.  One job / tables of several, whose
// lanes end at different hops and whose next launches wait behind them.  GB300,
// s22, 8 streams: one job of 3,000 walkers x 40 hops with 16 / 8 / 4: node2vec
// 32 / 32 / 54 us, weighted 19 / 20 / 59, metapath 21 / 22 / 55; batches of 16
// served queries (node2vec, metapath, weighted), 12,000 in all, with 16 / 8 / 4
// / 2 / 1: 255 / 239 / 230 / 225 / 224 ms, of 4 queries 399 / 377 / 356 / 342 /
// 331, which keep less of a lone launch's gain on few streams.
constexpr int kSharedWalkersJob = 16, kSharedWalkersTable = 2;

struct WalkerPlacement {
  bool by_place;  // walkers are given to the warps by place; else they come from the queue, 32 per warp
  int wpw;        // walkers per warp
  int grid;       // blocks
};

// Blocks per SM whose warps a launch fills before its walkers share warps
// further: launches of more than two walkers for each resident warp.
// First-order walks (weighted, metapath) are bound by instruction issue before
// their warps fill every slot.  GB300, R-MAT s12 /
// s16 / s20, U(0,1] and no weights, x 30 hops, mean speed against full warps
// with all resident blocks / 3 / 2 / 1: weighted 5,000 walkers 1.60 / 1.60 /
// 1.59 / 1.56, 20,000 1.23 / 1.28 / 1.34 / 1.31, 60,000 1.00 / 1.12 / 1.18 /
// 1.17, 120,000 1.13 / 1.16 / 1.16 / 1.16 (with every block slower than full
// warps from 40,000 to 60,000, down to 0.91); metapath 20,000 1.28 / 1.32 /
// 1.39 / 1.33, 60,000 1.05 / 1.14 / 1.19 / 1.13.  node2vec 20,000 1.79 with
// all, 1.69 with 2.
constexpr int kFirstOrderFill = 2, kFillAll = 64;

// `total` walkers on `sms` SMs with `bps` resident blocks each of the kernel
// that gives walkers by place, of which it fills `fill` per SM first; `scans`: jobs that only scan rows, at most
// `scan_wpw` walkers per warp, the rest in the queue.  `table`: several jobs.
// `beside`: launches, this one included, that are meant to run at the same
// time.
//
// A launch alone is spread over every resident warp before its walkers share
// one, and over the blocks before their warps: a warp pays for the longest of
// its lanes' paths in every iteration, and idle slots cost nothing.  Beside
// others they do: a block that holds five walkers keeps 256 lanes from the
// next launch.  So a launch takes its share of the blocks only and fills
// them.  GB300, s22 x 40 hops on 8 streams, every launch spread over the GPU
// -> its share of it (us per launch): node2vec 3,000 walkers 60 -> 32, 20,000
// 184 -> 68, 60,000 313 -> 127 (full warps always: 59 / 75 / 169); batches of
// 64 served queries 583 -> 463 ms.
inline WalkerPlacement place_walkers(long long total, int sms, int bps, int fill, bool scans, int scan_wpw, bool table,
                                     int beside) {
  WalkerPlacement p;
  const int blocks = sms * bps;
  if (total <= 2ll * blocks * kShapeWarps) fill = kFillAll;
  const long long share = std::max(1, std::min(sms * fill, blocks / std::max(1, beside)));
  const long long warps = share * kShapeWarps;
  p.wpw = (int)std::min<long long>(32, std::max<long long>(1, (total + warps - 1) / warps));
  if (scans) p.wpw = std::min(p.wpw, scan_wpw);
  const int most = beside <= 1 ? 32 : table ? kSharedWalkersTable : kSharedWalkersJob;
  p.by_place = scans || (total <= (long long)blocks * kShapeWarps * 32 && p.wpw <= most);
  if (!p.by_place) p.wpw = 32;
  const long long per_block = p.by_place && beside <= 1 ? p.wpw : (long long)kShapeWarps * p.wpw;
  p.grid = (int)std::min<long long>(blocks, std::max<long long>(1, (total + per_block - 1) / per_block));
  return p;
}

}  // namespace fw
