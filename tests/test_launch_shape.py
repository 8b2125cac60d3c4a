"""Launch shapes (csrc/fw_shape.h, csrc/fw_streams.h), compiled with the host
C++ compiler: every walker has a place or a queue, a launch alone is spread
over the GPU, one of several side by side takes its share of the blocks."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2512_00705_gb300", "csrc")

SHAPE = r"""
#include <cstdio>
#include "fw_shape.h"
#define CHECK(c) do { if (!(c)) { std::printf("FAIL line %d: %s (total %lld blocks %d beside %d)\n", __LINE__, #c, total, blocks, beside); return 1; } } while (0)

#define CHECK3(c) do { if (!(c)) { std::printf("FAIL line %d: %s\n", __LINE__, #c); return 1; } } while (0)

int main() {
  for (int sms : {1, 2, 152})
  for (int bps : {1, 3, 4, 7})
    for (int beside : {1, 2, 3, 4, 8, 24, 192})
      for (long long total : {1ll, 2ll, 31ll, 37ll, 300ll, 3000ll, 5003ll, 20000ll, 60000ll, 77824ll, 77825ll, 155647ll, 155648ll, 155649ll, 272384ll, 2000000ll, 1ll << 30})
        for (int k = 0; k < 16; ++k) {
          const int blocks = sms * bps, fill = k >= 8 ? fw::kFirstOrderFill : fw::kFillAll;
          const int scan = (k & 3) == 0 ? 0 : (k & 3) == 1 ? 1 : (k & 3) == 2 ? 8 : 32;
          const bool table = (k & 4) != 0;
          const fw::WalkerPlacement p = fw::place_walkers(total, sms, bps, fill, scan > 0, scan, table, beside);
          const long long lanes = 256ll * blocks, placed = (long long)p.grid * fw::kShapeWarps * p.wpw;
          CHECK(p.wpw >= 1 && p.wpw <= 32 && p.grid >= 1 && p.grid <= blocks);
          CHECK(p.by_place || p.wpw == 32);
          CHECK(!scan || (p.by_place && p.wpw <= scan));
          if (p.by_place && !scan) CHECK(placed >= total);                          // no queue
          if (!scan && beside == 1) CHECK(p.by_place == (total <= lanes));
          const long long filled = 8ll * blocks;
          if (!scan && beside == 1 && total <= filled) CHECK(p.wpw == 1 && p.grid == (total < blocks ? total : blocks));
          if (!scan && beside > 1 && p.by_place) {                                  // its share, filled
            CHECK(p.wpw <= (table ? fw::kSharedWalkersTable : fw::kSharedWalkersJob));
            CHECK((long long)p.grid * beside <= blocks || p.grid == 1);
            CHECK(p.grid <= (total + fw::kShapeWarps * p.wpw - 1) / (fw::kShapeWarps * p.wpw));
          }
          if (!scan && beside > 1 && !p.by_place) CHECK(p.grid == (total + 255) / 256 || p.grid == blocks);
        }
  // scans: full warps for short rows and histograms, few walkers per warp for long rows in small launches
  CHECK3(fw::scan_walkers_per_warp(true, false, 48, true) == 32 && fw::scan_walkers_per_warp(false, false, 48, false) == 16);
  CHECK3(fw::scan_walkers_per_warp(true, true, 5000, true) == 32 && fw::scan_walkers_per_warp(false, true, 5000, false) == 32);
  CHECK3(fw::scan_walkers_per_warp(true, false, 1246, false) == 1 && fw::scan_walkers_per_warp(true, false, 1246, true) == 8);
  CHECK3(fw::scan_walkers_per_warp(true, false, 150, false) == 8 && fw::scan_walkers_per_warp(false, false, 150, false) == 1);
  CHECK3(fw::scan_walkers_per_warp(false, false, 150, true) == 8 && fw::scan_walkers_per_warp(false, false, 1246, true) == 4);
  // first-order: 60,000 walkers alone, 25 to a warp
  CHECK3(fw::place_walkers(60000, 152, 4, fw::kFirstOrderFill, false, 32, false, 1).wpw == 25);
  // 20,000 walkers on 152 SMs x 4 blocks: alone on every block, beside seven others in 79 blocks of full warps
  const fw::WalkerPlacement a = fw::place_walkers(20000, 152, 4, fw::kFillAll, false, 32, false, 1), b = fw::place_walkers(20000, 152, 4, fw::kFillAll, false, 32, false, 8);
  long long total = 20000;
  int blocks = 608, beside = 8;
  CHECK(a.by_place && a.wpw == 5 && a.grid == 608);
  CHECK(!b.by_place && b.grid == 79);
  std::printf("ok\n");
  return 0;
}
"""

STREAMS = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "fw_streams.h"
#define CHECK(c) do { if (!(c)) { std::printf("FAIL line %d: %s\n", __LINE__, #c); return 1; } } while (0)
using R = fw::RecentStreams;

int main() {
  const R::Clock::time_point t0 = R::Clock::now();
  auto at = [&](double ms) { return t0 + std::chrono::duration_cast<R::Clock::duration>(std::chrono::duration<double, std::milli>(ms)); };
  const double w = (double)R::kWindow.count();
  {
    R r;  // one stream, however often
    for (int i = 0; i < 100; ++i) CHECK(r.note(7, at(i * 0.01)) == 1);
    CHECK(r.note(0, at(1.0)) == 2);                 // the default stream is a stream
    CHECK(r.note(7, at(1.1)) == 2);
    CHECK(r.note(7, at(1.0 + 1.5 * w)) == 1);       // the other one has been idle since
  }
  {
    R r;  // eight streams in turn
    for (int i = 0; i < 80; ++i) CHECK(r.note(i % 8, at(i * 0.1)) == (i < 8 ? i + 1 : 8));
  }
  {
    R r;  // a new stream for every call, one call at a time
    for (int i = 0; i < 1000; ++i) CHECK(r.note(1000 + i, at(i * 2.0 * w)) == 1);
    for (int i = 0; i < 1000; ++i) CHECK(r.note(5000 + i, at(2000.0 * w + i * 0.001)) <= R::kMost);
  }
  R r;
  std::vector<std::thread> ts;
  int bad[8] = {};
  for (int t = 0; t < 8; ++t)
    ts.emplace_back([&, t] {
      for (int i = 0; i < 20000; ++i) {
        const int n = r.note((uintptr_t)t);
        if (n < 1 || n > 8) bad[t] = 1;
      }
    });
  for (auto& t : ts) t.join();
  for (int b : bad) CHECK(b == 0);
  std::printf("ok\n");
  return 0;
}
"""


@pytest.mark.parametrize("name", ["shape", "streams"])
def test_host_rules(tmp_path, name):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text({"shape": SHAPE, "streams": STREAMS}[name])
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-pthread", "-I", CSRC, str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout == "ok\n"
