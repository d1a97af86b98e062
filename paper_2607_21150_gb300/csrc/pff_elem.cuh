// Element kernels of the matrix-free operator (Sec. 4):
//   y = P^T sum_el E^T [B_I; B_xi]^T W Lambda f_hat(...) [B_I; B_xi] E P x
//
// One thread block handles EB = 256 / Q^2 consecutive elements with Q*Q threads
// per element; thread (i, j) of an element owns the column of quadrature
// points (i, j, 0..Q-1).  The tensor contractions are sum-factorised through
// shared memory one direction at a time; gradients at the Gauss points use
// the collocated derivative D_c (exact because p <= Q - 1).  The pointwise
// linearisation is read from a tiled layout so that every load of a block is
// one contiguous run: in FP64, word w of slice k of block b sits at
//   b * kLinWords * Q^3 * EB + w * Q^3 * EB + k * Q^2 * EB + threadIdx.x;
// the FP32 planes group words 0..63 of a point by four (lin32_word), so that
// one 128-bit load fetches four words.
//
// The action in FP32 arithmetic is here and in pff_elem_pipe.cuh, every FP64
// kernel in pff_elem_fix.cuh.
#pragma once
#include "pff_df.cuh"
#include "pff_internal.h"

namespace pff {

template <typename T> __device__ __forceinline__ T ldg(const T* p) { return __ldg(p); }
// four consecutive words of the FP32 quad layout; p is 16-byte aligned
__device__ __forceinline__ float4 ld_quad(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }

__device__ __forceinline__ double madd(double c, double a, double b) { return fma(a, b, c); }
__device__ __forceinline__ float madd(float c, float a, float b) { return fmaf(a, b, c); }

template <int P, int Q>
__device__ __forceinline__ long long node_of(const MeshDev& m, int e, int a, int b, int c) {
  if (m.offsets) return m.offsets[(long long)e * (P * P * P) + a + P * (b + P * c)];
  int ex = e % m.nx;
  int t = e / m.nx;
  int ey = t % m.ny;
  int ez = t / m.ny;
  return (long long)(m.p * ex + a) + (long long)m.nnx * ((long long)(m.p * ey + b) + (long long)m.nny * (m.p * ez + c));
}

// Shared-memory layout per element of k_elem: the values at the Gauss points
// (4 Q^3), then a ping-pong buffer that extends to the x- and y-derivative outputs
// of all slices (8 Q^3), so that the pointwise stage runs without barriers.
template <int Q> __host__ __device__ constexpr int elem_smem_words() { return 12 * Q * Q * Q; }

struct ElemSmem {
  float* bufA;  // [4][Q^3]
  float* bufB;  // [4][Q^3]
  const float* B;
  const float* Dc;
};

// Gather x into bufA [4][c][b][a] (masked entries zero).
template <int P, int Q>
__device__ __forceinline__ void gather(const ElemArgs<float>& a, float* bufA, int e, bool valid, int ij) {
  constexpr int Q2 = Q * Q, Q3 = Q * Q * Q, P3 = P * P * P;
  const long long nn = a.mesh.nn;
  // the node mask is read only for elements flagged as having masked nodes
  const bool masked = a.mask && valid && (!a.emask || a.emask[e]);
  // every thread's gather loads (values and mask bytes) are independent and
  // issued together: one memory round trip instead of one per node and a
  // second one behind each mask byte
#pragma unroll
  for (int r = 0; r < (P3 + Q2 - 1) / Q2; ++r) {
    const int idx = ij + r * Q2;
    if (idx >= P3) break;
    int aa = idx % P, bb = (idx / P) % P, cc = idx / (P * P);
    long long n = valid ? node_of<P, Q>(a.mesh, e, aa, bb, cc) : 0;
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      float v = 0.0f;
      if (valid) {
        long long g = f * nn + n;
        const auto xv = ldg(a.x + g);
        const bool fixed = masked && ldg(a.mask + g);
        if (!fixed) v = xv;
      }
      bufA[f * Q3 + idx] = v;
    }
  }
}

// Forward: gather x into bufA, interpolate to Gauss points into bufB.
template <int P, int Q>
__device__ __forceinline__ void forward(const ElemArgs<float>& a, const ElemSmem& s, int e, bool valid, int ij) {
  constexpr int Q2 = Q * Q, Q3 = Q * Q * Q;
  gather<P, Q>(a, s.bufA, e, valid, ij);
  __syncthreads();
  // x: [c][b][a] -> [c][b][i]
  for (int idx = ij; idx < P * P * Q; idx += Q2) {
    int i = idx % Q, r = idx / Q;  // r = b + P c
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const float* in = s.bufA + f * Q3 + r * P;
      float acc = 0.0f;
#pragma unroll
      for (int k = 0; k < P; ++k) acc = madd(acc, s.B[i * P + k], in[k]);
      s.bufB[f * Q3 + idx] = acc;
    }
  }
  __syncthreads();
  // y: [c][b][i] -> [c][j][i]
  for (int idx = ij; idx < P * Q * Q; idx += Q2) {
    int i = idx % Q, j = (idx / Q) % Q, c = idx / Q2;
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const float* in = s.bufB + f * Q3 + c * (P * Q) + i;
      float acc = 0.0f;
#pragma unroll
      for (int k = 0; k < P; ++k) acc = madd(acc, s.B[j * P + k], in[k * Q]);
      s.bufA[f * Q3 + idx] = acc;
    }
  }
  __syncthreads();
  // z: [c][j][i] -> [k][j][i]
  {
    const int i = ij % Q, j = ij / Q;
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      float col[P];
#pragma unroll
      for (int c = 0; c < P; ++c) col[c] = s.bufA[f * Q3 + c * Q2 + j * Q + i];
#pragma unroll
      for (int k = 0; k < Q; ++k) {
        float acc = 0.0f;
#pragma unroll
        for (int c = 0; c < P; ++c) acc = madd(acc, s.B[k * P + c], col[c]);
        s.bufB[f * Q3 + k * Q2 + j * Q + i] = acc;
      }
    }
  }
  __syncthreads();
}

// Parent-frame gradients of the four fields at point (i, j, k) from bufB.
template <int Q>
__device__ __forceinline__ void grad_at(const ElemSmem& s, int i, int j, int k, float g[4][3], float& phi) {
  constexpr int Q2 = Q * Q, Q3 = Q * Q * Q;
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    const float* V = s.bufB + f * Q3;
    float gx = 0.0f, gy = 0.0f, gz = 0.0f;
#pragma unroll
    for (int m = 0; m < Q; ++m) {
      gx = madd(gx, s.Dc[i * Q + m], V[k * Q2 + j * Q + m]);
      gy = madd(gy, s.Dc[j * Q + m], V[k * Q2 + m * Q + i]);
      gz = madd(gz, s.Dc[k * Q + m], V[m * Q2 + j * Q + i]);
    }
    g[f][0] = gx; g[f][1] = gy; g[f][2] = gz;
  }
  phi = s.bufB[3 * Q3 + k * Q2 + j * Q + i];
}

// Backward: from accumulated column values Y[f][k] (transposed derivative
// already applied) to nodal element values, then scatter-add.
template <int P, int Q>
__device__ __forceinline__ void backward(const ElemArgs<float>& a, const ElemSmem& s, int e, bool valid, int ij,
                                         float Y[4][Q]) {
  constexpr int Q2 = Q * Q, Q3 = Q * Q * Q, P3 = P * P * P;
  const int i = ij % Q, j = ij / Q;
  // z (registers): [k][j][i] -> [c][j][i]
#pragma unroll
  for (int f = 0; f < 4; ++f)
#pragma unroll
    for (int c = 0; c < P; ++c) {
      float acc = 0.0f;
#pragma unroll
      for (int k = 0; k < Q; ++k) acc = madd(acc, s.B[k * P + c], Y[f][k]);
      s.bufA[f * Q3 + c * Q2 + j * Q + i] = acc;
    }
  __syncthreads();
  // y: [c][j][i] -> [c][b][i]
  for (int idx = ij; idx < P * P * Q; idx += Q2) {
    int ii = idx % Q, bb = (idx / Q) % P, c = idx / (P * Q);
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const float* in = s.bufA + f * Q3 + c * Q2 + ii;
      float acc = 0.0f;
#pragma unroll
      for (int jj = 0; jj < Q; ++jj) acc = madd(acc, s.B[jj * P + bb], in[jj * Q]);
      s.bufB[f * Q3 + idx] = acc;
    }
  }
  __syncthreads();
  // x: [c][b][i] -> [c][b][a]
  for (int idx = ij; idx < P3; idx += Q2) {
    int aa = idx % P, r = idx / P;
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const float* in = s.bufB + f * Q3 + r * Q;
      float acc = 0.0f;
#pragma unroll
      for (int ii = 0; ii < Q; ++ii) acc = madd(acc, s.B[ii * P + aa], in[ii]);
      s.bufA[f * Q3 + idx] = acc;
    }
  }
  __syncthreads();
  if (!valid) return;
  if (a.evec) {  // deterministic transpose: element-local values, summed per node by k_node_gather
    float* ev = static_cast<float*>(a.evec) + (long long)e * 4 * P3;
    for (int idx = ij; idx < P3; idx += Q2)
#pragma unroll
      for (int f = 0; f < 4; ++f) ev[f * P3 + idx] = (s.bufA[f * Q3 + idx]);
    return;
  }
  const long long nn = a.mesh.nn;
  const bool masked = a.mask && (!a.emask || a.emask[e]);
#pragma unroll
  for (int r = 0; r < (P3 + Q2 - 1) / Q2; ++r) {
    const int idx = ij + r * Q2;
    if (idx >= P3) break;
    int aa = idx % P, bb = (idx / P) % P, cc = idx / (P * P);
    long long n = node_of<P, Q>(a.mesh, e, aa, bb, cc);
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      long long g = f * nn + n;
      if (masked && ldg(a.mask + g)) continue;
      atomicAdd(a.y + g, (s.bufA[f * Q3 + idx]));
    }
  }
}

// Pointwise linear map of the Jacobian with the stored FP64 words (already scaled
// by the quadrature weight and the parent-to-reference factors).
__device__ __forceinline__ void jac_point(const double* lin, const double* linP, const double* linC, long long stride,
                                          int kx, const double g[4][3], double phi, double o[4][3], double& o0) {
  double gu[9];
#pragma unroll
  for (int f = 0; f < 3; ++f)
#pragma unroll
    for (int al = 0; al < 3; ++al) gu[3 * f + al] = g[f][al];
  double ou[9];
#pragma unroll
  for (int m = 0; m < 9; ++m) ou[m] = ldg(linP + m * stride) * phi;
  // symmetric 9x9 block
#pragma unroll
  for (int m = 0; m < 9; ++m) {
#pragma unroll
    for (int n = m; n < 9; ++n) {
      const double A = ldg(lin + (long long)sym9(m, n) * stride);
      ou[m] = madd(ou[m], A, gu[n]);
      if (n != m) ou[n] = madd(ou[n], A, gu[m]);
    }
  }
  double s0 = ldg(lin + kWD * stride) * phi;
#pragma unroll
  for (int m = 0; m < 9; ++m) s0 = madd(s0, ldg(linC + m * stride), gu[m]);
  o0 = s0;
#pragma unroll
  for (int f = 0; f < 3; ++f)
#pragma unroll
    for (int al = 0; al < 3; ++al) o[f][al] = ou[3 * f + al];
#pragma unroll
  for (int al = 0; al < 3; ++al) o[3][al] = ldg(lin + (kWK + al) * stride) * g[3][al];
  if (kx) {  // mapped mesh: symmetric off-diagonal coefficients 01, 02, 12
    const double k01 = ldg(lin + (kWKX + 0) * stride);
    const double k02 = ldg(lin + (kWKX + 1) * stride);
    const double k12 = ldg(lin + (kWKX + 2) * stride);
    o[3][0] = madd(madd(o[3][0], k01, g[3][1]), k02, g[3][2]);
    o[3][1] = madd(madd(o[3][1], k01, g[3][0]), k12, g[3][2]);
    o[3][2] = madd(madd(o[3][2], k02, g[3][0]), k12, g[3][1]);
  }
}

// The same map reading the FP32 plane in the quad layout: q = the point's first
// quad (quads at stride qs), tl = its word 64 (tail words at stride ts).  Every
// quad is used as it arrives, in word order: the 9x9 block, dP/dphi and
// d(s_phi L)/dF (their roles swapped for the transpose, TR), d(s_phi L)/dphi.
template <bool TR>
__device__ __forceinline__ void jac_point_q(const float* q, long long qs, const float* tl, long long ts, int kx,
                                            const float g[4][3], float phi, float o[4][3], float& o0) {
  float gu[9];
#pragma unroll
  for (int f = 0; f < 3; ++f)
#pragma unroll
    for (int al = 0; al < 3; ++al) gu[3 * f + al] = g[f][al];
  float ou[9], s0 = 0.0f;
#pragma unroll
  for (int m = 0; m < 9; ++m) ou[m] = 0.0f;
  float4 quad;
  auto word = [&](int wd) {
    if ((wd & 3) == 0) quad = ld_quad(q + (wd >> 2) * qs);
    return (wd & 3) == 0 ? quad.x : (wd & 3) == 1 ? quad.y : (wd & 3) == 2 ? quad.z : quad.w;
  };
#pragma unroll
  for (int m = 0; m < 9; ++m) {  // upper triangle of the symmetric 9x9 block, row-major
#pragma unroll
    for (int n = m; n < 9; ++n) {
      const float w = word(sym9(m, n));
      ou[m] = madd(ou[m], w, gu[n]);
      if (n != m) ou[n] = madd(ou[n], w, gu[m]);
    }
  }
#pragma unroll
  for (int wd = kWP; wd < kLinQuadWords; ++wd) {  // the quad of word 44 is loaded
    const float w = word(wd);
    if (wd < kWC) {
      if (TR) s0 = madd(s0, w, gu[wd - kWP]);
      else ou[wd - kWP] = madd(ou[wd - kWP], w, phi);
    } else if (wd < kWD) {
      if (TR) ou[wd - kWC] = madd(ou[wd - kWC], w, phi);
      else s0 = madd(s0, w, gu[wd - kWC]);
    } else {
      s0 = madd(s0, w, phi);
    }
  }
  o0 = s0;
#pragma unroll
  for (int f = 0; f < 3; ++f)
#pragma unroll
    for (int al = 0; al < 3; ++al) o[f][al] = ou[3 * f + al];
#pragma unroll
  for (int al = 0; al < 3; ++al) o[3][al] = ldg(tl + al * ts) * g[3][al];
  if (kx) {  // mapped mesh: symmetric off-diagonal coefficients 01, 02, 12
    const float k01 = ldg(tl + 3 * ts), k02 = ldg(tl + 4 * ts), k12 = ldg(tl + 5 * ts);
    o[3][0] = madd(madd(o[3][0], k01, g[3][1]), k02, g[3][2]);
    o[3][1] = madd(madd(o[3][1], k01, g[3][0]), k12, g[3][2]);
    o[3][2] = madd(madd(o[3][2], k02, g[3][0]), k12, g[3][1]);
  }
}

// L2 prefetch of slice k of this block's stored linearisation (FP32 action):
// threads 0..15 request the contiguous run of one quad plane (4 Q^2 EB words),
// the next three (six on mapped meshes) the run of one tail word (Q^2 EB words),
// each with one bulk prefetch, so the next slice streams from HBM while this
// one computes (64^3 Q4: 3.76 -> 3.48 ms; two or three slices ahead measured
// slower).  Tail runs start on 8-byte boundaries; the request is widened to
// 16-byte boundaries and clipped to the plane.
constexpr int kPrefetchAhead = 1;  // slices requested ahead of the one computed
__device__ __forceinline__ void prefetch_run(uintptr_t base, long long first, long long run, long long plane) {
  const uintptr_t lo = (base + 4 * first) & ~uintptr_t(15);
  uintptr_t hi = (base + 4 * (first + run) + 15) & ~uintptr_t(15);
  const uintptr_t end = (base + 4 * plane) & ~uintptr_t(15);
  if (hi > end) hi = end;
  if (hi <= lo) return;
  asm volatile(
      "{\n\t.reg .u64 ga;\n\tcvta.to.global.u64 ga, %0;\n\tcp.async.bulk.prefetch.L2.global [ga], %1;\n\t}"
      :: "l"(lo), "r"((unsigned)(hi - lo)) : "memory");
}
template <int Q>
__device__ __forceinline__ void prefetch_slice(const ElemArgs<float>& a, int k, int t) {
  constexpr int EB = elems_per_block(Q);
  constexpr long long run = (long long)Q * Q * EB;   // words of one (word, slice) run
  constexpr int NQ = kLinQuadWords / 4;
  if (t >= NQ + (a.kx ? kLinWords - kLinQuadWords : kWKX - kLinQuadWords) || k >= Q) return;
  const long long nblk = (a.mesh.nel + EB - 1) / EB;
  const long long plane = nblk * kLinWords * Q * Q * Q * EB;
  const long long blk = (a.blk0 + blockIdx.x) * kLinWords * Q * run;
  const uintptr_t base = reinterpret_cast<uintptr_t>(a.lin);
  if (t < NQ) prefetch_run(base, blk + lin32_word(4 * t, k, 0, Q * run, run), 4 * run, plane);
  else prefetch_run(base, blk + lin32_word(kLinQuadWords + t - NQ, k, 0, Q * run, run), run, plane);
}

// FP32-word action without the persistent kernel's shared-memory ring (mapped
// meshes at Q = 5, whose two slots leave no room for a second block): three
// resident blocks per SM (<= 85 registers), no barriers in the pointwise stage.
template <int P, int Q>
__global__ void __launch_bounds__(Q * Q * elems_per_block(Q), 3)
k_elem(const ElemArgs<float> a) {
  constexpr int EB = elems_per_block(Q);
  constexpr int Q2 = Q * Q, Q3 = Q * Q * Q;
  constexpr long long run = (long long)Q2 * EB, stride = run * Q;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* sm = reinterpret_cast<float*>(smem_raw);
  const int t = threadIdx.x;
  const int el = t / Q2, ij = t % Q2;
  const int i = ij % Q, j = ij / Q;
  const int e = (a.blk0 + blockIdx.x) * EB + el;
  const bool valid = e < a.mesh.nel;

  float* Bs = sm;
  float* Dcs = Bs + Q * P;
  for (int idx = t; idx < Q * P; idx += blockDim.x) Bs[idx] = a.B[idx];
  for (int idx = t; idx < Q * Q; idx += blockDim.x) Dcs[idx] = a.Dc[idx];
  float* base = sm + mat_smem_words<P, Q>() + el * elem_smem_words<Q>();
  // bufB first (read by every slice's gradients), then bufA which extends to the
  // 8 x Q^3 derivative outputs of the pointwise stage
  const ElemSmem s{base + 4 * Q3, base, Bs, Dcs};
  __syncthreads();
  for (int k = 0; k < kPrefetchAhead; ++k) prefetch_slice<Q>(a, k, t);
  forward<P, Q>(a, s, e, valid, ij);

  float Y[4][Q];
#pragma unroll
  for (int f = 0; f < 4; ++f)
#pragma unroll
    for (int k = 0; k < Q; ++k) Y[f][k] = 0.0f;
  // pointwise stage of all slices: z-derivative and value terms into the
  // registers of the own column, x- and y-derivative outputs to shared memory
  const float* blk = a.lin + (a.blk0 + blockIdx.x) * (long long)kLinWords * stride;
  float* oxy = s.bufA;  // [8][Q^3]
#pragma unroll
  for (int k = 0; k < Q; ++k) {
    float g[4][3], phi, o[4][3], o0 = 0.0f;
    prefetch_slice<Q>(a, k + kPrefetchAhead, t);
    grad_at<Q>(s, i, j, k, g, phi);
    if (valid) {
      const float* q = blk + lin32_word(0, k, t, stride, run);
      const float* tl = blk + lin32_word(kLinQuadWords, k, t, stride, run);
      if (a.transpose) jac_point_q<true>(q, 4 * stride, tl, stride, a.kx, g, phi, o, o0);
      else jac_point_q<false>(q, 4 * stride, tl, stride, a.kx, g, phi, o, o0);
    } else {
#pragma unroll
      for (int f = 0; f < 4; ++f) o[f][0] = o[f][1] = o[f][2] = 0.0f;
    }
#pragma unroll
    for (int f = 0; f < 4; ++f) {
#pragma unroll
      for (int kk = 0; kk < Q; ++kk) Y[f][kk] = madd(Y[f][kk], s.Dc[k * Q + kk], o[f][2]);
      oxy[(2 * f) * Q3 + k * Q2 + ij] = o[f][0];
      oxy[(2 * f + 1) * Q3 + k * Q2 + ij] = o[f][1];
    }
    Y[3][k] += o0;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < Q; ++k)
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const float* ox = oxy + (2 * f) * Q3 + k * Q2;
      const float* oy = oxy + (2 * f + 1) * Q3 + k * Q2;
      float acc = Y[f][k];
#pragma unroll
      for (int m = 0; m < Q; ++m) {
        acc = madd(acc, s.Dc[m * Q + i], ox[j * Q + m]);
        acc = madd(acc, s.Dc[m * Q + j], oy[m * Q + i]);
      }
      Y[f][k] = acc;
    }
  __syncthreads();  // the derivative outputs are read; backward reuses the buffers
  backward<P, Q>(a, s, e, valid, ij, Y);
}

// Diagonal of the element operators: for each field f and node a,
//   sum_q sum_{alpha,beta} D_{f alpha, f beta}(q) d_alpha N_a d_beta N_a
// (+ the value term of the phase field), sum-factorised with the 1D products
// BB, BD, DD of the basis and its derivative (kinds 0, 1, 2 per direction).
//
// The (alpha, beta) terms of a field meet as early as their kinds allow: the
// six (kx, ky, kz) = 200, 110, 101, 020, 011, 002 leave the z contraction
// separately (the value term, 000, joins 002 there), the y contraction sums
// them by kx into three, the x contraction into one.  A field takes three
// barriers, and its words (whole quads in FP32) are requested while the former
// field is contracted.  Term by term, as before, a block passed 66 barriers and
// waited for each term's words: 290 us at 24x24x72 Q3 FP32, 113 us now (the
// quads that hold the words are 456 MB, 68 us at the copy rate).
//
// In FP64 the pipe binds (16 clocks per warp instruction and SM), so that idle
// lanes and products with zeros count: there the lines of the y and x stages are
// spread over the block's warps (at order 1 and Q4 half and a quarter of an
// element's threads have one), and the terms that a field does not have are left
// out (the value term of a displacement, the mixed terms of the phase field on a
// box).  41x40x37 Q3, FP64: order 1 1155 -> 685 us, order 3 2206 -> 1919 us (term
// by term 973 and 2339 us).  In FP32 an element's threads keep their own lines.
constexpr int kDiagTerms = 6;
// Words of field f at the thread's points, one value per term (f = 3: term 5
// gets the value word besides, in v).
template <int Q, typename T>
__device__ __forceinline__ void diag_words(const ElemArgs<T>& a, int f, int t, bool valid, T w[kDiagTerms][Q], T v[Q]) {
  constexpr long long EB = elems_per_block(Q), run = (long long)Q * Q * EB, stride = run * Q;
  const T* lin = a.lin + (a.blk0 + blockIdx.x) * (long long)kLinWords * stride;
#pragma unroll
  for (int k = 0; k < Q; ++k) {
#pragma unroll
    for (int m = 0; m < kDiagTerms; ++m) w[m][k] = T(0);
    v[k] = T(0);
  }
  if (!valid) return;
  // first derivative pairs (alpha, beta) of the terms: 00, 01, 02, 11, 12, 22
  if (f < 3) {
#pragma unroll
    for (int k = 0; k < Q; ++k) {
      if constexpr (sizeof(T) == 4) {
        // the six words lie in three quads; f is uniform, so are the selections
        const float* p = lin + (long long)k * 4 * run + 4 * t;
        const int q0 = f == 0 ? 0 : f == 1 ? 6 : 9;   // quads of words (f0, f0 .. f2)
        const int q1 = f == 0 ? 2 : f == 1 ? 7 : 10;
        const int q2 = f == 0 ? 4 : f == 1 ? 8 : 11;
        const float4 A = ld_quad(p + q0 * 4 * stride), B = ld_quad(p + q1 * 4 * stride),
                     C = ld_quad(p + q2 * 4 * stride);
        if (f == 0) {         // words 0, 1, 2, 9, 10, 17
          w[0][k] = A.x; w[1][k] = A.y; w[2][k] = A.z; w[3][k] = B.y; w[4][k] = B.z; w[5][k] = C.y;
        } else if (f == 1) {  // words 24, 25, 26, 30, 31, 35
          w[0][k] = A.x; w[1][k] = A.y; w[2][k] = A.z; w[3][k] = B.z; w[4][k] = B.w; w[5][k] = C.w;
        } else {              // words 39, 40, 41, 42, 43, 44
          w[0][k] = A.w; w[1][k] = B.x; w[2][k] = B.y; w[3][k] = B.z; w[4][k] = B.w; w[5][k] = C.x;
        }
      } else {
        const T* p = lin + (long long)k * run + t;
        int m = 0;
#pragma unroll
        for (int al = 0; al < 3; ++al)
#pragma unroll
          for (int be = al; be < 3; ++be) w[m++][k] = ldg(p + (long long)sym9(3 * f + al, 3 * f + be) * stride);
      }
    }
#pragma unroll
    for (int k = 0; k < Q; ++k) {
      w[1][k] *= T(2); w[2][k] *= T(2); w[4][k] *= T(2);
    }
  } else {
#pragma unroll
    for (int k = 0; k < Q; ++k) {
      auto word = [&](int wd) {
        return ldg(lin + (sizeof(T) == 4 ? lin32_word(wd, k, t, stride, run) : (long long)wd * stride + (long long)k * run + t));
      };
      w[0][k] = word(kWK); w[3][k] = word(kWK + 1); w[5][k] = word(kWK + 2); v[k] = word(kWD);
      if (a.kx) {  // mapped mesh: 2 K_al,be d_al N d_be N
        w[1][k] = T(2) * word(kWKX); w[2][k] = T(2) * word(kWKX + 1); w[4][k] = T(2) * word(kWKX + 2);
      }
    }
  }
}
// The 1D products [kind][q][node] as kernel parameters (constant-bank operands;
// from shared memory they took a load per two multiply-adds: 153 us at the size
// above, 113 us now), rounded once from the FP64 products.
template <typename T, int P, int Q> struct DiagMats { T m[3 * Q * P]; };
template <int P, int Q> __host__ __device__ constexpr int diag_smem_words() {
  return kDiagTerms * P * Q * Q + 3 * P * P * Q;
}

template <int P, int Q, typename T>
__global__ void __launch_bounds__(Q * Q * elems_per_block(Q), 2)
k_diag(const ElemArgs<T> a, const DiagMats<T, P, Q> mats) {
  constexpr int EB = elems_per_block(Q);
  constexpr int Q2 = Q * Q, P3 = P * P * P;
  constexpr bool kPipe64 = sizeof(T) == 8;  // bound by the FP64 pipe
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sm = reinterpret_cast<T*>(smem_raw);
  const int t = threadIdx.x;
  const int el = t / Q2, ij = t % Q2;
  const int e = (a.blk0 + blockIdx.x) * EB + el;
  const bool valid = e < a.mesh.nel;
  constexpr int W = diag_smem_words<P, Q>(), NT = Q2 * EB;
  T* Zb = sm + el * W;  // [term][c][j][i], then [c][b][a]; behind it Yb [kx][c][b][i]
  const bool masked = a.mask && valid && (!a.emask || a.emask[e]);
  const long long nn = a.mesh.nn;
  // kinds of the terms 00, 01, 02, 11, 12, 22
  constexpr int KX[kDiagTerms] = {2, 1, 1, 0, 0, 0}, KY[kDiagTerms] = {0, 1, 0, 2, 1, 0}, KZ[kDiagTerms] = {0, 0, 1, 0, 1, 2};
  T w[kDiagTerms][Q], v[Q];
  diag_words<Q, T>(a, 0, t, valid, w, v);
#pragma unroll 1
  for (int f = 0; f < 4; ++f) {
    auto absent = [&](int m) { return kPipe64 && f == 3 && !a.kx && (m == 1 || m == 2 || m == 4); };
#pragma unroll
    for (int c = 0; c < P; ++c)
#pragma unroll
      for (int m = 0; m < kDiagTerms; ++m) {
        if (absent(m)) continue;
        T s = T(0);
#pragma unroll
        for (int k = 0; k < Q; ++k) s += mats.m[(KZ[m] * Q + k) * P + c] * w[m][k];
        if (m == 5 && (!kPipe64 || f == 3)) {
          T u = T(0);
#pragma unroll
          for (int k = 0; k < Q; ++k) u += mats.m[k * P + c] * v[k];
          s += u;
        }
        Zb[(m * P + c) * Q2 + ij] = s;
      }
    __syncthreads();
    if (f < 3) diag_words<Q, T>(a, f + 1, t, valid, w, v);
    // lines of the thread's own element, or (kPipe64) of the whole block in turn
    auto lines = [&](int per_element, auto line) {
      if constexpr (kPipe64)
        for (int idx = t; idx < EB * per_element; idx += NT) line(sm + idx / per_element * W, idx % per_element);
      else
        for (int idx = ij; idx < per_element; idx += Q2) line(Zb, idx);
    };
    lines(P * Q, [&](T* Zb, int idx) {  // y: lines (c, i)
      T* Yb = Zb + kDiagTerms * P * Q2;
      const int i = idx % Q, c = idx / Q;
      T s[3][P];
#pragma unroll
      for (int g = 0; g < 3; ++g)
#pragma unroll
        for (int bb = 0; bb < P; ++bb) s[g][bb] = T(0);
#pragma unroll
      for (int m = 0; m < kDiagTerms; ++m) {
        if (absent(m)) continue;
        T u[P];  // each term's sum by itself (short chains keep FP32's error at the former level)
#pragma unroll
        for (int bb = 0; bb < P; ++bb) u[bb] = T(0);
#pragma unroll
        for (int j = 0; j < Q; ++j) {
          const T z = Zb[(m * P + c) * Q2 + j * Q + i];
#pragma unroll
          for (int bb = 0; bb < P; ++bb) u[bb] += mats.m[(KY[m] * Q + j) * P + bb] * z;
        }
#pragma unroll
        for (int bb = 0; bb < P; ++bb) s[KX[m]][bb] += u[bb];
      }
#pragma unroll
      for (int g = 0; g < 3; ++g)
#pragma unroll
        for (int bb = 0; bb < P; ++bb) Yb[((g * P + c) * P + bb) * Q + i] = s[g][bb];
    });
    __syncthreads();
    lines(P * P, [&](T* Zb, int idx) {  // x: lines (c, b)
      const T* Yb = Zb + kDiagTerms * P * Q2;
      T s[P];
#pragma unroll
      for (int aa = 0; aa < P; ++aa) s[aa] = T(0);
#pragma unroll
      for (int g = 0; g < 3; ++g) {
        T u[P];
#pragma unroll
        for (int aa = 0; aa < P; ++aa) u[aa] = T(0);
#pragma unroll
        for (int i = 0; i < Q; ++i) {
          const T y = Yb[(g * P * P + idx) * Q + i];
#pragma unroll
          for (int aa = 0; aa < P; ++aa) u[aa] += mats.m[(g * Q + i) * P + aa] * y;
        }
#pragma unroll
        for (int aa = 0; aa < P; ++aa) s[aa] += u[aa];
      }
#pragma unroll
      for (int aa = 0; aa < P; ++aa) Zb[idx * P + aa] = s[aa];
    });
    __syncthreads();
    if (valid) {
      if (a.evec) {  // deterministic: element-local values, summed per node by k_node_gather
        T* ev = static_cast<T*>(a.evec) + ((long long)e * 4 + f) * P3;
        for (int idx = ij; idx < P3; idx += Q2) ev[idx] = Zb[idx];
      } else {
        for (int idx = ij; idx < P3; idx += Q2) {
          const long long g = f * nn + node_of<P, Q>(a.mesh, e, idx % P, (idx / P) % P, idx / (P * P));
          if (masked && a.mask[g]) continue;
          atomicAdd(a.y + g, Zb[idx]);
        }
      }
    }
    __syncthreads();  // the next field's terms overwrite Zb
  }
}

}  // namespace pff

#include "pff_elem_fix.cuh"
#include "pff_elem_pipe.cuh"

namespace pff {

// FP64: fixed-point contractions, every mode.  FP32 arithmetic: the action only,
// in the persistent kernel where its slots fit.
template <int P, int Q, typename T>
cudaError_t launch_elem_pq(int mode, const ElemArgs<T>& a, cudaStream_t st) {
  constexpr int EB = elems_per_block(Q);
  int nblk = a.nblk > 0 ? a.nblk : (a.mesh.nel + EB - 1) / EB;
  if (nblk == 0) return cudaSuccess;
  if constexpr (sizeof(T) == 8) {
    if (mode == kApply) return launch_elem_fix<P, Q, kApply>(a, nblk, st);
    if (mode == kEval) return launch_elem_fix<P, Q, kEval>(a, nblk, st);
    return launch_elem_fix<P, Q, kBack>(a, nblk, st);
  } else {
    if (mode != kApply) return cudaErrorInvalidValue;
    cudaError_t err = cudaSuccess;
    if (launch_level_pipe<P, Q>(a, nblk, st, &err)) return err;
    if constexpr (!pipe_fits<P, Q, false, true>()) {
      const size_t smem = sizeof(float) * (size_t)(mat_smem_words<P, Q>() + EB * elem_smem_words<Q>());
      auto k = k_elem<P, Q>;
      cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      k<<<nblk, Q * Q * EB, smem, st>>>(a); note_launch();
      return cudaGetLastError();
    }
    return cudaErrorInvalidValue;
  }
}

template <int P, int Q, typename T>
cudaError_t launch_diag_pq(const ElemArgs<T>& a, const double* B, const double* D, cudaStream_t st) {
  DiagMats<T, P, Q> mats;
  for (int i = 0; i < Q * P; ++i) {
    mats.m[i] = (T)(B[i] * B[i]);
    mats.m[Q * P + i] = (T)(B[i] * D[i]);
    mats.m[2 * Q * P + i] = (T)(D[i] * D[i]);
  }
  constexpr int EB = elems_per_block(Q);
  int nblk = (a.mesh.nel + EB - 1) / EB;
  if (nblk == 0) return cudaSuccess;
  size_t smem = sizeof(T) * (size_t)(EB * diag_smem_words<P, Q>());
  auto k = k_diag<P, Q, T>;
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  k<<<nblk, Q * Q * EB, smem, st>>>(a, mats); note_launch();
  return cudaGetLastError();
}

}  // namespace pff
