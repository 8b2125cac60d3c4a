"""Steps through the entries of a CSR row (csrc/fw_rows.h), compiled with the
host C++ compiler: rows that end at the last entry a graph can hold, with every
stride the kernels use, visit each of their entries once and nothing else."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2512_00705_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include <vector>
#include "fw_rows.h"
#define CHECK(c) do { if (!(c)) { std::printf("FAIL line %d: %s\n", __LINE__, #c); return 1; } } while (0)

int main() {
  const int64_t most = 2147483647;
  for (int32_t step : {32, 256, 1024})
    for (int32_t d : {1, 31, 32, 33, 255, 256, 257, 1023, 1024, 1025, 4099})
      for (int64_t gap : {0, 1, 31, 32, 1023, 1024, 100000}) {
        const int64_t s = most - gap - d;
        std::vector<int> seen(d, 0);
        bool inside = true;
        for (int32_t t = 0; t < step; ++t)
          fw::for_entries((int32_t)s, d, t, step, [&](int32_t i) {
            if (i < s || i >= s + d) inside = false;
            else ++seen[i - s];
          });
        CHECK(inside);
        for (int n : seen) CHECK(n == 1);
      }
  int64_t count = 0, last = -1;  // one row of all entries
  fw::for_entries(0, (int32_t)most, 1022, 1024, [&](int32_t i) {
    ++count;
    last = i;
  });
  CHECK(count == 2097152 && last == most - 1);
  std::printf("ok\n");
  return 0;
}
"""


def test_rows_at_the_largest_entry(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "rows.cpp", tmp_path / "rows"
    src.write_text(HARNESS)
    subprocess.run([cxx, "-std=c++17", "-O1", "-fsanitize=signed-integer-overflow", "-fno-sanitize-recover=all",
                    "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout == "ok\n"


@pytest.mark.parametrize("name", ["fw_preprocess.cu", "fw_kernels.cu"])
def test_preprocessing_kernels_do_not_step_an_entry_index(name):
    text = open(os.path.join(CSRC, name)).read()
    assert not re.search(r"for \(int32_t \w+ = (s|lo|off\[\w+\]|lane)\b", text)
