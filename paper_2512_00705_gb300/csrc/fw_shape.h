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

// Walkers per warp of jobs that only scan rows, `row` entries long on average.
// The warp scans one long row at a time, so that few walkers per warp leave no
// warp with several hub rows at the end of a launch; short rows are their
// lane's own work, and launches of more walkers than lanes (`many`) last long
// enough to even out.  A histogram's walkers all scan one row.  GB300, R-MAT
// s12 to s18, 5 hops, speed against full warps from a queue with 1 / 4 / 8 /
// 16 / 32 walkers per warp: eRVS, weighted, 1,200,000 walkers, mean row 48
// 0.56 / 0.79 / 0.90 / 1.00 / 1.05, 142 0.77 / 0.94 / 1.02 / 1.05 / 1.06, 745
// 1.20 / 1.30 / 1.31 / 1.29 / 1.26; 60,000 walkers, row 192 1.63 / 1.65 / 1.68
// (no more needed), 745 2.58 / 2.36 / 1.98; metapath (rows of a label's share)
// 1,200,000 walkers, row 48 / 8 0.26 / 0.46 / 0.63 / 0.86 / 1.12.  Exact mode,
// metapath, 1,200,000 walkers, row 48 0.67 / 0.84 / 0.95 / 1.04 / 1.09, 142
// 0.92 / 1.00 / 1.05 / 1.06 / 1.08, 745 1.08 / 1.10 / 1.09 / 1.07 / 1.04;
// 300,000 walkers, row 745 1.27 / 1.24 / 1.19 / 1.15 / 1.00; 60,000 walkers,
// row 48 1.46 / 1.56 / 1.48 / 1.65, 250 2.20 / 1.88 / 1.67.
constexpr double kTinyScan = 100.0, kShortScan = 250.0;
inline int scan_walkers_per_warp(bool reservoir, bool histogram, double row, bool many) {
  if (histogram) return 32;
  if (row < kTinyScan) return reservoir ? 32 : 16;
  if (row < kShortScan) return many || reservoir ? 8 : 1;
  return many ? (reservoir ? 8 : 4) : 1;
}

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
// 185 -> 64, 60,000 315 -> 127 (full warps always: 53 / 72 / 169), weighted 42
// -> 19, 109 -> 30, 155 -> 61 (25 / 31 / 63); batches of 64 served queries 583
// -> 463 ms.  The algorithms of one batch do not count:
// a plan's parallel branches last as long as their longest, which gains more
// from the whole GPU than the others lose (47 plans of 2 to 64 jobs, branches
// sharing / alone: 1.62 / 1.89 times the speed of full warps).
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
