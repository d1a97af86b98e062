"""Lanes that take part in the warp reductions of the element kernels (no GPU).

A warp intrinsic with a lane mask waits for exactly the lanes of its mask, so the
mask has to name the threads of the block, all of them: a mask taken from the
lanes that are together by chance (the active mask) may leave some out after a
branch, and their part of the result is lost without a sign.

* no kernel derives a mask from the active lanes;
* warp_lanes names the lanes of every warp that hold threads, for the block sizes
  of the FP64 element kernels, and a warp that reduces holds one element only.
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
      const int q3 = Q * Q * Q, threads = q3 * fix_elems(Q, small != 0);
      for (int warp = 0; 32 * warp < threads; ++warp) {
        const unsigned m = warp_lanes(threads, warp);
        if (!(m & 1u)) { std::printf("Q=%d warp %d without lane 0\n", Q, warp); ++bad; }
        for (int lane = 0; lane < 32; ++lane) {
          const int t = 32 * warp + lane;
          if (((m >> lane & 1u) != 0) != (t < threads)) { std::printf("Q=%d thread %d\n", Q, t); ++bad; }
          if (t < threads && t / q3 != 32 * warp / q3) { std::printf("Q=%d warp %d holds two elements\n", Q, warp); ++bad; }
        }
      }
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
