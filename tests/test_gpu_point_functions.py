"""Elementary functions and the eigen-decomposition of the pointwise update
(pff_point.cuh), compiled into a small program and run on the GPU: against extended
precision on both sides of every switch, and through the branches that states of
small strain hardly reach.

Tolerances, u = 2^-53.  Reciprocal: the last Newton step rounds twice, the second
time at 2^-48 of the result: 2 u.  half_log1p, exp_near: two to three roundings of
the leading term inside the series, 1 ulp (2 u) of CUDA's functions outside, halved
or passed on: 3 u.  Eigenpairs: the transform to the FP32 frame rounds each entry
through two sums of three products (6 u), up to three sweeps of three rotations
follow at three roundings each (27 u): 40 u of the largest entry for X V - V w
(times sqrt(9) in the Frobenius norm: 120 u), and 40 u for V^T V - I, per entry.
"""
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2607_21150_gb300 import build  # noqa: E402

U = 2.0 ** -53
PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "pff_point.cuh"
using namespace pff;
// rows of 9 doubles in; out: 3 functions of entry 0 (kind 0), or w, V and the return value of eigh3 (kind 1)
__global__ void k_run(const double* in, double* out, int n, int kind) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double* x = in + 9 * i;
  double* y = out + 13 * i;
  if (kind == 0) {
    y[0] = rcp64(x[0]);
    y[1] = half_log1p(x[0]);
    y[2] = exp_near(x[0]);
    for (int k = 3; k < 13; ++k) y[k] = 0.0;
  } else {
    double X[3][3], V[3][3], w[3];
    for (int r = 0; r < 3; ++r)
      for (int c = 0; c < 3; ++c) X[r][c] = x[3 * r + c];
    y[12] = eigh3(X, V, w);
    for (int r = 0; r < 3; ++r) {
      y[r] = w[r];
      for (int c = 0; c < 3; ++c) y[3 + 3 * r + c] = V[r][c];
    }
  }
}
int main(int argc, char** argv) {
  const int n = std::atoi(argv[1]), kind = std::atoi(argv[2]);
  std::vector<double> h(9 * n), o(13 * n);
  FILE* f = std::fopen(argv[3], "rb");
  if (!f || std::fread(h.data(), 8, h.size(), f) != h.size()) return 2;
  std::fclose(f);
  double *in = nullptr, *out = nullptr;
  if (cudaMalloc(&in, 8 * h.size()) || cudaMalloc(&out, 8 * o.size())) return 3;
  if (cudaMemcpy(in, h.data(), 8 * h.size(), cudaMemcpyHostToDevice)) return 3;
  k_run<<<(n + 127) / 128, 128>>>(in, out, n, kind);
  if (cudaMemcpy(o.data(), out, 8 * o.size(), cudaMemcpyDeviceToHost)) return 4;
  f = std::fopen(argv[4], "wb");
  std::fwrite(o.data(), 8, o.size(), f);
  std::fclose(f);
  return 0;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    d = tmp_path_factory.mktemp("point")
    (d / "p.cu").write_text(PROGRAM)
    cmd = [build.nvcc(), *build.GENCODE, "-O3", "-std=c++17", "-diag-suppress", "128,177", "-I", build.CSRC,
           "-I", os.path.join(build.ROOT, "include"), str(d / "p.cu"), "-o", str(d / "p")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]

    def call(rows, kind):
        rows = np.ascontiguousarray(rows, dtype=np.float64)
        rows.tofile(d / "in")
        r = subprocess.run([str(d / "p"), str(len(rows)), str(kind), str(d / "in"), str(d / "out")], timeout=300)
        assert r.returncode == 0
        return np.fromfile(d / "out").reshape(-1, 13)

    return call


def scalars(run, x):
    rows = np.zeros((len(x), 9))
    rows[:, 0] = x
    return run(rows, 0)


def close_to(x, switch):
    """Values around a switch: the neighbours on both sides and a spread about it."""
    near = switch * (1.0 + np.array([-1e-3, -2.0 ** -52, 0.0, 2.0 ** -52, 1e-3]))
    return np.concatenate([x, near, -near])


def worst(got, want, pick):
    want = np.asarray(want, dtype=np.longdouble)
    return float(np.max(np.abs((got[pick].astype(np.longdouble) - want[pick]) / want[pick])))


def test_reciprocal(run):
    rng = np.random.default_rng(1)
    m = rng.uniform(1.0, 2.0, 20000) * rng.choice([-1.0, 1.0], 20000)
    x = close_to(close_to(m * 2.0 ** rng.integers(-1000, 1000, 20000), 1e-37), 1e37)
    x = np.concatenate([x, m, [1.0, 2.0, 3.0, 1.0 - U, 1.0 + 2 * U]])
    y = scalars(run, x)[:, 0]
    assert worst(y, 1.0 / x.astype(np.longdouble), np.ones(len(x), bool)) <= 2 * U
    y = scalars(run, [0.0, -0.0, np.inf, -np.inf, np.nan, 2.0 ** -1060])[:, 0]
    assert y[0] == np.inf and y[1] == -np.inf and y[2] == 0.0 and y[3] == 0.0 and np.isnan(y[4]) and y[5] == np.inf


def test_half_log1p(run):
    rng = np.random.default_rng(2)
    small = 10.0 ** rng.uniform(-300, -1.3, 20000) * rng.choice([-1.0, 1.0], 20000)
    x = close_to(np.concatenate([small, rng.uniform(-0.0625, 0.0625, 20000), 10.0 ** rng.uniform(-1.3, 300, 5000),
                                 -1.0 + 10.0 ** rng.uniform(-15, -0.1, 5000)]), 0.0625)
    y = scalars(run, x)[:, 1]
    assert worst(y, 0.5 * np.log1p(x.astype(np.longdouble)), x != 0.0) <= 3 * U
    y = scalars(run, [0.0, -1.0, -2.0, np.inf, np.nan])[:, 1]
    assert y[0] == 0.0 and y[1] == -np.inf and np.isnan(y[2]) and y[3] == np.inf and np.isnan(y[4])


def test_exp_near(run):
    rng = np.random.default_rng(3)
    x = close_to(np.concatenate([rng.uniform(-0.0625, 0.0625, 20000), rng.uniform(-700, 700, 20000),
                                 10.0 ** rng.uniform(-300, -1.3, 5000)]), 0.0625)
    y = scalars(run, x)[:, 2]
    assert worst(y, np.exp(x.astype(np.longdouble)), np.ones(len(x), bool)) <= 3 * U
    y = scalars(run, [0.0, np.inf, -np.inf, np.nan, 1000.0])[:, 2]
    assert y[0] == 1.0 and y[1] == np.inf and y[2] == 0.0 and np.isnan(y[3]) and y[4] == np.inf


def frames(rng, n):
    return np.linalg.qr(rng.standard_normal((n, 3, 3)))[0]


def check(run, X):
    X = 0.5 * (X + X.transpose(0, 2, 1))
    o = run(X.reshape(-1, 9), 1)
    w, V = o[:, :3], o[:, 3:12].reshape(-1, 3, 3)
    assert (o[:, 12] == 1.0).all()
    L = np.longdouble
    top = np.abs(X).max((1, 2))
    top = np.where(top > 0.0, top, 1.0)
    Xs, ws, V = (X / top[:, None, None]).astype(L), (w / top[:, None]).astype(L), V.astype(L)
    res = np.einsum("nij,njk->nik", Xs, V) - V * ws[:, None, :]
    orth = np.einsum("nji,njk->nik", V, V) - np.eye(3)
    assert float(np.sqrt((res ** 2).sum((1, 2))).max()) <= 120 * U
    assert float(np.abs(orth).max()) <= 40 * U


@pytest.mark.parametrize("gap", [1.0, 1e-2, 1e-4, 1e-6, 1e-8, 1e-10, 1e-12, 1e-14, 1e-15, 1e-16, 0.0])
@pytest.mark.parametrize("scale", [1.0, 1e-3, 2.0 ** -500, 2.0 ** 400])
def test_eigenpairs(run, gap, scale):
    """Two (or all three) eigenvalues a gap apart: angles of every size are left to the FP64 rotations."""
    rng = np.random.default_rng(int(1 / (gap + 1e-17)) % 2 ** 31)
    n = 4000
    d = rng.uniform(-1, 1, (n, 3))
    d[: n // 2, 1] = d[: n // 2, 0] + gap * rng.uniform(0.5, 1.5, n // 2)
    d[: n // 4, 2] = d[: n // 4, 0] - gap * rng.uniform(0.5, 1.5, n // 4)
    N = frames(rng, n)
    check(run, scale * np.einsum("nij,nj,nkj->nik", N, d, N))


@pytest.mark.parametrize("angle", [1e-2, 1e-3, 1e-4, 1e-8, 1e-9, 1e-10, 1e-17, 1e-19])
def test_nearly_diagonal(run, angle):
    """Off-diagonal entries on both sides of the switches (1e-3, 1e-9 of the diagonal's differences, 1e-18)."""
    rng = np.random.default_rng(5)
    X = np.einsum("ni,ij->nij", rng.uniform(-1, 1, (3000, 3)), np.eye(3))
    off = angle * rng.uniform(0.3, 3.0, (3000, 3)) * rng.choice([-1.0, 0.0, 1.0], (3000, 3))
    for k, (i, j) in enumerate(((0, 1), (0, 2), (1, 2))):
        X[:, i, j] = X[:, j, i] = off[:, k]
    check(run, X)


def test_special_matrices(run):
    one = np.ones((3, 3))
    X = [np.zeros((3, 3)), np.eye(3), one, -one, np.diag([1.0, 1.0, 2.0]), np.diag([1e-200, 1.0, -1.0]),
         np.array([[0, 1, 0], [1, 0, 0], [0, 0, 0.0]]), np.array([[0, 0, 1], [0, 0, 0], [1, 0, 0.0]]),
         np.array([[1, 1, 0], [1, 1, 0], [0, 0, 2.0]]), np.array([[1, 0.5, 0.5], [0.5, 1, 0.5], [0.5, 0.5, 1]])]
    check(run, np.array(X))
    bad = np.array([np.where(np.eye(3) > 0, v, 0.1) for v in (np.nan, np.inf, -np.inf)])
    assert (run(bad.reshape(-1, 9), 1)[:, 12] == 0.0).all()
