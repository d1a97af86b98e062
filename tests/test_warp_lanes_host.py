"""Lanes that take part in the warp reductions of the element kernels (no GPU).

A warp intrinsic with a lane mask waits for exactly the lanes of its mask, so the
mask has to name all threads of the warp: a mask taken from the lanes that are
together by chance (the active mask) may leave some out after a branch, and their
part of the result is lost without a sign.

* no kernel derives a mask from the active lanes;
* the blocks of the FP64 element kernels whose warps reduce (Q >= 4) consist of
  full warps, and the points of a warp belong to one element.
"""
import glob
import os
import shutil
import subprocess

import pytest

from test_layout_host import CSRC, _cuda_include

PROGRAM = r"""
#include <cstdio>
#include "pff_internal.h"
using namespace pff;
int main() {
  int bad = 0;
  for (int Q = 4; Q <= 5; ++Q)
    for (int small = 0; small < 2; ++small) {
      const int q3 = Q * Q * Q, elems = fix_elems(Q, small != 0), threads = fix_threads(Q, elems);
      if (threads % 32) { std::printf("Q=%d: the last warp is not full\n", Q); ++bad; }
      if (threads < q3 * elems) { std::printf("Q=%d: points without a thread\n", Q); ++bad; }
      for (int t = 0; t < q3 * elems; ++t)
        if (t / q3 != t / 32 * 32 / q3) { std::printf("Q=%d warp %d holds two elements\n", Q, t / 32); ++bad; }
    }
  std::printf(bad ? "FAIL\n" : "OK\n");
  return bad ? 1 : 0;
}
"""


def test_no_mask_from_the_active_lanes():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        with open(path) as f:
            assert "__activemask" not in f.read(), path


def test_reduction_lanes(tmp_path):
    cxx, inc = shutil.which("g++"), _cuda_include()
    if cxx is None or inc is None:
        pytest.skip("needs g++ and the CUDA headers")
    src, exe = tmp_path / "lanes.cpp", tmp_path / "lanes"
    src.write_text(PROGRAM)
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, "-I", inc, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip().endswith("OK"), r.stdout[-3000:]
