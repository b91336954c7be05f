"""The batch autotuner's search on made-up times (host logic, no GPU): the default shape is timed first, so the shape
returned is never slower than it, and the cache's key names the kernels the shapes were timed for."""
import os
import shutil
import subprocess

import pytest

import paper_2404_09758_gb300 as sge

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include "sge_internal.h"
// argv: pairs per view, the pairs per item that are fast (-1: none but the first shape timed); prints the shapes timed, then the
// shape returned
int main(int argc, char** argv) {
  const int pairs = atoi(argv[1]), fast = atoi(argv[2]);
  sge_batch_tuning best{};
  float ms = 0.0f;
  int n = 0;
  auto time_of = [&](const sge_batch_tuning& t, float& out) {
    printf("%d,%d,%d ", t.pairs_per_item, t.blocks_per_sm, t.light_bin);
    out = (fast < 0 ? n == 0 : t.pairs_per_item == fast) ? 1.0f + 0.01f * n : 2.0f;
    ++n;
    return 0;
  };
  const int rc = sge::search_batch_shape(pairs, time_of, best, ms);
  printf("%d,%d,%d %g\n", best.pairs_per_item, best.blocks_per_sm, best.light_bin, ms);
  return rc;
}
"""


@pytest.fixture(scope="module")
def search(tmp_path_factory):
    if not shutil.which("g++") or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("shape")
    src, exe = str(d / "t.cpp"), str(d / "t")
    open(src, "w").write(SRC)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"), "-I",
                           os.path.join(ROOT, "paper_2404_09758_gb300", "csrc"), "-I", os.path.join(CUDA, "include"),
                           src, "-o", exe])
    return lambda pairs, fast: subprocess.check_output([exe, str(pairs), str(fast)], text=True).split()


@pytest.mark.parametrize("pairs,default", [(1, "8,0,256"), (3, "8,0,256"), (8, "8,0,256"), (9, "0,0,256"), (64, "0,0,256")])
def test_default_is_timed_first_and_may_be_returned(search, pairs, default):
    out = search(pairs, -1)
    assert out[0] == default and out[-2] == default and float(out[-1]) == 1.0
    assert len(set(out[:-2])) == len(out) - 2  # no shape twice


@pytest.mark.parametrize("pairs,fast", [(16, 16), (64, 2), (64, 8), (5, 4)])
def test_a_faster_shape_is_found(search, pairs, fast):
    out = search(pairs, fast)
    assert out[-2] == f"{fast},0,256" and float(out[-1]) < 2.0


def test_shapes_timed_for_other_kernels_do_not_fit(monkeypatch):
    key = sge.tuning_key("GB300", [(512, 512, 1000)], 8)
    monkeypatch.setattr(sge, "TUNED_KERNELS", "others")
    assert sge.tuning_key("GB300", [(512, 512, 1000)], 8) != key
    assert key != "GB300|8|512x512:T1024"  # the key of caches written before
