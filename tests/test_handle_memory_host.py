"""Device buffers of an operator across calls that replace or remove its data (no
GPU): the ABI's host code linked against a CUDA runtime that only keeps a list of
the live allocations.

* removing the Dirichlet data keeps the deterministic mode's element values, which
  the next action writes, and frees the mask's buffers;
* every buffer is freed once, by whichever call, and none is left at the end.
"""
import os
import shutil
import subprocess

import pytest

from test_layout_host import CSRC, ROOT, _cuda_include

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <set>
#include "pff_handles.h"

static std::set<void*> live;
static int bad = 0;
#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); ++bad; } } while (0)

extern "C" {
cudaError_t cudaMalloc(void** p, size_t n) { live.insert(*p = std::malloc(n ? n : 1)); return cudaSuccess; }
cudaError_t cudaFree(void* p) {
  if (p && !live.erase(p)) { std::printf("freed twice\n"); ++bad; return cudaSuccess; }
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMemset(void* p, int v, size_t n) { std::memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { std::memset(p, v, n); return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "error"; }
}
namespace pff {
cudaError_t launch_elem_mask(const MeshDev&, const uint8_t*, uint8_t*, cudaStream_t) { return cudaSuccess; }
}

int main() {
  const double row[12] = {0.8, 0.005, 1e3, 0.3};
  const pff_problem pr{1, row, 2, 1e-3, 1e-2, 0.01, 1.0};
  const pff_box box{2, 1, 1, 1.0, 1.0, 1.0};
  pff_ctx* ctx = nullptr;
  pff_basis* basis = nullptr;
  pff_restr* restr = nullptr;
  pff_op* op = nullptr;
  CHECK(pff_create_context(&ctx, &pr) == PFF_OK);
  CHECK(pff_create_basis(ctx, 1, 2, &basis) == PFF_OK);
  CHECK(pff_create_restriction(ctx, &box, 1, nullptr, 12, &restr) == PFF_OK);
  CHECK(pff_create_operator(ctx, basis, restr, &op) == PFF_OK);
  const uint8_t mask[48] = {1};
  const double values[48] = {0.5};
  const size_t before = live.size();
  for (int rep = 0; rep < 2; ++rep) {
    CHECK(pff_set_dirichlet(op, mask, values, nullptr) == PFF_OK);
    CHECK(pff_op_set_deterministic(op, 1) == PFF_OK);
    CHECK(pff_set_dirichlet(op, nullptr, nullptr, nullptr) == PFF_OK);
    CHECK(op->det == 1 && op->evec && live.count(op->evec));  // the next action writes there
    CHECK(live.size() == before + 1);
    CHECK(!op->mask && !op->emask && !op->dvals);
  }
  CHECK(pff_destroy_operator(op) == PFF_OK);
  CHECK(live.empty());
  std::printf(bad ? "FAIL\n" : "OK\n");
  return bad ? 1 : 0;
}
"""


def test_buffers_across_dirichlet_changes(tmp_path):
    cxx, inc = shutil.which("g++"), _cuda_include()
    if cxx is None or inc is None:
        pytest.skip("needs g++ and the CUDA headers")
    src, exe = tmp_path / "memory.cpp", tmp_path / "memory"
    src.write_text(PROGRAM)
    # the launch functions are not called and stay unresolved
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-I", inc,
                        "-Wl,--unresolved-symbols=ignore-all", str(src), os.path.join(CSRC, "pff_abi.cpp"),
                        os.path.join(CSRC, "pff_basis.cpp"), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip().endswith("OK"), r.stdout[-3000:]
