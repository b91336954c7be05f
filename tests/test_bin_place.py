"""Placing of the tile bins where a call's entries pass 32 bits (host arithmetic, no GPU): the functions the binning
kernel places tiles with, on synthetic counts.  A bin either lies inside the capacity, apart from every other, or
is left out by readers and writer alike, so that no reader or writer of the bins goes past their end."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include "sge_internal.h"
// argv: capacity, triangles, then (count, tiles) runs; prints bins stored, their entries, whether the total passes
int main(int argc, char** argv) {
  const long long cap = atoll(argv[1]);
  const int nt = atoi(argv[2]);
  unsigned long long total = 0, end = 0, stored = 0;
  for (int a = 3; a + 1 < argc; a += 2) {
    const uint32_t c = (uint32_t)strtoul(argv[a], nullptr, 10);
    for (long long k = atoll(argv[a + 1]); k > 0; --k, total += c) {
      if (c == 0) continue;
      const uint32_t off = sge::bin_start(total, c, cap), cur = sge::bin_cursor(off, nt);
      const uint32_t last = cur + c - 1;             // the last entry's position as the fill forms it: 32 bits
      if (last < cur) return 3;                      // wrapped
      // the fill's test of a position
      auto stores = [&](uint32_t pos) { return (long long)pos < cap && (sge::cursors_above(cap, nt) || off != sge::kNoBin); };
      const bool first_in = stores(cur), last_in = stores(last);
      if ((long long)off + c <= cap) {               // stored, by the readers' test
        if (off != total || off < end || cur != off || !first_in || !last_in) return 4;
        end = (unsigned long long)off + c;
        ++stored;
      } else if (first_in || last_in) {
        return 5;                                    // left out, yet the fill would write into the bins
      }
    }
  }
  printf("%llu %llu %d\n", stored, end, total > (unsigned long long)cap);
  return 0;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    if not shutil.which("g++") or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("bin_place")
    src, exe = str(d / "t.cpp"), str(d / "t")
    open(src, "w").write(SRC)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"), "-I",
                           os.path.join(ROOT, "paper_2404_09758_gb300", "csrc"), "-I", os.path.join(CUDA, "include"),
                           src, "-o", exe])
    return exe


@pytest.mark.parametrize("capacity,nt,runs,want", [
    (1000, 50, [(10, 100)], (100, 1000, 0)),                          # exactly full
    (999, 50, [(10, 100)], (99, 990, 1)),                             # the last tile left out
    (1000, 50, [(0, 5), (7, 2), (0, 3)], (2, 14, 0)),                 # empty tiles
    # 16,400 triangles in every tile of 16 views of 2048^2: 2^32 + 4.2 M entries, whose low 32 bits fit
    (6_000_000, 16_400, [(16_400, 16 * 16_384)], (365, 365 * 16_400, 1)),
    # one CTA's 1,024 counts alone pass 2^32
    (6_000_000, 1 << 22, [(1 << 22, 1024)], (1, 1 << 22, 1)),
    # the largest capacity there is, exceeded by one tile and by many
    ((1 << 32) - 1, 1 << 20, [(1 << 20, 4096)], (4095, 4095 << 20, 1)),
    ((1 << 32) - 1, 1 << 30, [(1 << 30, 9)], (3, 3 << 30, 1)),
    ((1 << 32) - 1, (1 << 31) - 1, [((1 << 31) - 1, 9)], (2, (1 << 32) - 2, 1)),
])
def test_bins_lie_inside_the_capacity_or_are_seen_not_to(harness, capacity, nt, runs, want):
    args = [str(x) for run in runs for x in run]
    r = subprocess.run([harness, str(capacity), str(nt), *args], capture_output=True, text=True)
    assert r.returncode == 0, r.returncode
    assert tuple(int(x) for x in r.stdout.split()) == want
