"""The searches over row starts at the largest sizes: every probe lies inside
the array and the answer is the last entry at or below the value sought.  The
arrays are virtual (entry i is computed), so that no memory is needed."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_12196_gb300", "csrc")

SOURCE = r"""
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <initializer_list>

#include "search.h"

// entry i of an ascending array with equal runs (empty rows)
static int64_t entry(int64_t i, int64_t run) { return i / run * run; }

int main(int argc, char** argv) {
  const int64_t n = atoll(argv[1]), run = atoll(argv[2]);
  const int threads = 256;
  for (int64_t want : {(int64_t)0, (int64_t)1, n / 3, n / 2, n - 257, n - 2, n - 1}) {
    if (want < 0 || want >= n) continue;
    const int64_t x = entry(want, run);
    const int64_t top = (want / run + 1) * run - 1, last = top < n ? top : n - 1;
    const int64_t got = gm::last_by_probes(n, threads, [&](int64_t lo, int64_t len, int64_t step) {
      int cnt = 0;
      for (int t = 0; t < threads; t++) {
        const int64_t at = t * step;
        if (at >= len) continue;
        if (step < 1 || lo + at < 0 || lo + at >= n) {
          printf("probe %lld of %lld\n", (long long)(lo + at), (long long)n);
          exit(1);
        }
        cnt += entry(lo + at, run) <= x;
      }
      return cnt;
    });
    if (got != last) return printf("probes: %lld, not %lld\n", (long long)got, (long long)last), 1;
    const int32_t b = gm::last_by_bisection<int32_t>(0, (int32_t)n, [&](int32_t i) {
      if (i < 0 || i >= n) {
        printf("bisection at %d of %lld\n", i, (long long)n);
        exit(1);
      }
      return entry(i, run) <= x;
    });
    if (b != last) return printf("bisection: %d, not %lld\n", b, (long long)last), 1;
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("search")
    src, exe = d / "search.cpp", d / "search"
    src.write_text(SOURCE)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return str(exe)


@pytest.mark.parametrize("run", [1, 7, 1 << 21, 1 << 30])
@pytest.mark.parametrize("n", [1, 2, 255, 257, 65537, (1 << 31) - 300, (1 << 31) - 255, (1 << 31) - 1])
def test_every_probe_in_range(program, n, run):
    r = subprocess.run([program, str(n), str(run)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
