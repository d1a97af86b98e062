// Vector kernels: Dirichlet initialisation, the FP32 and BF16 copies of the
// stored linearisation, the
// Chebyshev smoother updates, the export of the linearisation, reaction sums
// and the geometric factors of mapped meshes.
#include <cuda_bf16.h>

#include <initializer_list>

#include "pff_df.cuh"
#include "pff_internal.h"

namespace pff {

constexpr int kVecThreads = 256;

static unsigned grid_for(long long n) {
  long long b = (n + kVecThreads - 1) / kVecThreads;
  if (b > 152LL * 64) b = 152LL * 64;  // grid-stride beyond 64 blocks per SM
  return (unsigned)(b > 0 ? b : 1);
}

// mode 0: y = mask ? x : 0      (Jacobian action: identity rows of Dirichlet DoFs)
// mode 1: y = mask ? x - u : 0  (residual: z - ubar on Dirichlet DoFs)
// mode 2: y = mask ? 1 : 0      (diagonal)
// Bound by the store of y (x is read where masked only).  V entries per thread:
// FP32 takes four where n is a multiple of four and the addresses allow 16-byte
// stores and 4-byte mask loads (every vector from its allocation's start): 3.7 M
// entries 12.3 -> 6.2 us, 17 M 28 -> 20 us.  FP64 goes one by one: with four,
// 68 M entries took 103 us instead of 101.
template <typename T, int V>
__global__ void k_init_masked(T* __restrict__ y, const T* __restrict__ x, const double* __restrict__ ubar,
                              const uint8_t* __restrict__ mask, long long n, int mode) {
  struct alignas(V * sizeof(T)) Out { T v[V]; };
  const long long nv = n / V;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nv; i += (long long)gridDim.x * blockDim.x) {
    unsigned m = 0;  // V mask bytes
    if (mask) m = V == 4 ? *reinterpret_cast<const unsigned*>(mask + 4 * i) : mask[i];
    Out o;
#pragma unroll
    for (int c = 0; c < V; ++c) {
      T v = T(0);
      if (m >> (8 * c) & 255u) {
        const long long k = i * V + c;
        if (mode == 0) v = x[k];
        else if (mode == 1) v = x[k] - (ubar ? (T)ubar[k] : T(0));
        else v = T(1);
      }
      o.v[c] = v;
    }
    *reinterpret_cast<Out*>(y + i * V) = o;
  }
}

template <typename T>
static void init_masked(T* y, const T* x, const double* ubar, const uint8_t* mask, long long n, int mode,
                        cudaStream_t st) {
  if constexpr (sizeof(T) == 4) {
    if (n % 4 == 0 && (reinterpret_cast<uintptr_t>(y) & 15) == 0 && (reinterpret_cast<uintptr_t>(mask) & 3) == 0) {
      k_init_masked<T, 4><<<grid_for(n / 4), kVecThreads, 0, st>>>(y, x, ubar, mask, n, mode);
      return;
    }
  }
  k_init_masked<T, 1><<<grid_for(n), kVecThreads, 0, st>>>(y, x, ubar, mask, n, mode);
}

cudaError_t launch_init_masked(int prec, void* y, const void* x, const double* ubar, const uint8_t* mask,
                               long long n, int mode, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  if (prec == 0) init_masked((double*)y, (const double*)x, ubar, mask, n, mode, st);
  else init_masked((float*)y, (const float*)x, ubar, mask, n, mode, st);
  note_launch();
  return cudaGetLastError();
}

// Deterministic transpose E^T: every node sums the values its incident
// elements left in evec, always in the same order (elements ascending), so
// reruns are bitwise identical.  Node (I, J, K) lies in elements
// ex = I / p (local a = I mod p) and, on an element boundary (I mod p = 0),
// also ex - 1 (local a = p); likewise in y and z.
template <typename T>
__global__ void k_node_gather(MeshDev m, const T* __restrict__ evec, const uint8_t* __restrict__ mask, int mode,
                              const T* __restrict__ x, const double* __restrict__ ubar, T* __restrict__ y, long long n0,
                              long long n1) {
  const long long n = n0 + blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (n >= n1) return;
  const int p = m.p, P = p + 1, P3 = P * P * P;
  const int I = (int)(n % m.nnx), J = (int)((n / m.nnx) % m.nny), K = (int)(n / ((long long)m.nnx * m.nny));
  int ex[2], ax[2], nxc = 0, ey[2], ay[2], nyc = 0, ez[2], az[2], nzc = 0;
  if (I % p == 0 && I > 0) { ex[nxc] = I / p - 1; ax[nxc++] = p; }
  if (I / p < m.nx) { ex[nxc] = I / p; ax[nxc++] = I % p; }
  if (J % p == 0 && J > 0) { ey[nyc] = J / p - 1; ay[nyc++] = p; }
  if (J / p < m.ny) { ey[nyc] = J / p; ay[nyc++] = J % p; }
  if (K % p == 0 && K > 0) { ez[nzc] = K / p - 1; az[nzc++] = p; }
  if (K / p < m.nz) { ez[nzc] = K / p; az[nzc++] = K % p; }
  for (int f = 0; f < 4; ++f) {
    const long long g = f * m.nn + n;
    T v = T(0);
    if (mask && mask[g]) {
      v = (mode == 0) ? x[g] : (mode == 1) ? x[g] - (ubar ? (T)ubar[g] : T(0)) : (mode == 2) ? T(1) : T(0);
    } else {
      for (int cz = 0; cz < nzc; ++cz)
        for (int cy = 0; cy < nyc; ++cy)
          for (int cx = 0; cx < nxc; ++cx) {
            const long long e = ex[cx] + (long long)m.nx * (ey[cy] + (long long)m.ny * ez[cz]);
            v += evec[(e * 4 + f) * P3 + ax[cx] + P * (ay[cy] + P * az[cz])];
          }
    }
    y[g] = v;
  }
}
cudaError_t launch_node_gather(int prec, const MeshDev& m, const void* evec, const uint8_t* mask, int mode,
                               const void* x, const double* ubar, void* y, long long n0, long long n1,
                               cudaStream_t st) {
  if (n1 <= n0) return cudaSuccess;
  const unsigned blocks = (unsigned)((n1 - n0 + 255) / 256);
  if (prec == 0)
    k_node_gather<double><<<blocks, 256, 0, st>>>(m, (const double*)evec, mask, mode, (const double*)x, ubar,
                                                  (double*)y, n0, n1);
  else
    k_node_gather<float><<<blocks, 256, 0, st>>>(m, (const float*)evec, mask, mode, (const float*)x, ubar,
                                                 (float*)y, n0, n1);
  note_launch();
  return cudaGetLastError();
}

// emask[e] = 1 if any of element e's nodes has a prescribed (masked) DoF in
// any field, else 0: the element kernels read the node mask only for flagged
// elements (on a box with Dirichlet faces, a few percent of them).
__global__ void k_elem_mask(MeshDev m, const uint8_t* __restrict__ mask, uint8_t* __restrict__ emask) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= m.nel) return;
  const int P = m.p + 1;
  const int ex = (int)(e % m.nx), t = (int)(e / m.nx), ey = t % m.ny, ez = t / m.ny;
  uint8_t any = 0;
  for (int c = 0; c < P && !any; ++c)
    for (int b = 0; b < P && !any; ++b)
      for (int a = 0; a < P; ++a) {
        const long long n = m.offsets ? (long long)m.offsets[e * P * P * P + a + P * (b + P * c)]
                                      : (long long)(m.p * ex + a) +
                                            (long long)m.nnx * ((long long)(m.p * ey + b) + (long long)m.nny * (m.p * ez + c));
        for (int f = 0; f < 4; ++f) any |= mask[f * m.nn + n];
        if (any) break;
      }
  emask[e] = any ? 1 : 0;
}
cudaError_t launch_elem_mask(const MeshDev& m, const uint8_t* mask, uint8_t* emask, cudaStream_t st) {
  if (m.nel == 0) return cudaSuccess;
  k_elem_mask<<<(unsigned)((m.nel + 255) / 256), 256, 0, st>>>(m, mask, emask); note_launch();
  return cudaGetLastError();
}

// y = mask ? x : 0 on the nodes [n0, n1) of each of the four fields (rows of
// one range of node layers; the pipelined action through host buffers).
template <typename T>
__global__ void k_init_rows(T* __restrict__ y, const T* __restrict__ x, const uint8_t* __restrict__ mask, long long nn,
                            long long n0, long long cnt) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < 4 * cnt; i += (long long)gridDim.x * blockDim.x) {
    const long long g = (i / cnt) * nn + n0 + i % cnt;
    y[g] = (mask && mask[g]) ? x[g] : T(0);
  }
}
cudaError_t launch_init_rows(int prec, void* y, const void* x, const uint8_t* mask, long long nn, long long n0,
                             long long n1, cudaStream_t st) {
  const long long cnt = n1 - n0;
  if (cnt <= 0) return cudaSuccess;
  if (prec == 0) k_init_rows<double><<<grid_for(4 * cnt), kVecThreads, 0, st>>>((double*)y, (const double*)x, mask, nn, n0, cnt);
  else k_init_rows<float><<<grid_for(4 * cnt), kVecThreads, 0, st>>>((float*)y, (const float*)x, mask, nn, n0, cnt);
  note_launch();
  return cudaGetLastError();
}

// BF16 word of x, round to nearest even, by integer operations on the FP64
// bit pattern (zero and FP64 subnormals give signed zero; the rare |x| outside
// the normal FP32 range goes through the library conversion).
__device__ __forceinline__ unsigned bf16_rne(double x) {
  const unsigned hw = (unsigned)__double2hiint(x), lw = (unsigned)__double2loint(x);
  const unsigned sgn = (hw >> 16) & 0x8000u;
  const int e = (int)((hw >> 20) & 0x7ffu);
  if (e == 0) return sgn;
  const int ef = e - 896;
  if (ef <= 0 || ef >= 255) return __bfloat16_as_ushort(__double2bfloat16(x));
  const unsigned top = ((unsigned)ef << 7) | ((hw & 0xfffffu) >> 13);  // exponent and 7 significand bits
  const unsigned r = hw & 0x1fffu;                                      // significand bits 44..32 (44: half)
  const unsigned inc = (r > 0x1000u || (r == 0x1000u && (lw != 0u || (top & 1u)))) ? 1u : 0u;
  return sgn | (top + inc);  // a carry moves into the exponent
}

// FP32 word of x, round to nearest even, by integer operations (zero and FP64
// subnormals give zero; |x| outside the normal FP32 range goes through the
// conversion instruction).
__device__ __forceinline__ float f32_rne(double x) {
  const unsigned hw = (unsigned)__double2hiint(x), lw = (unsigned)__double2loint(x);
  const int e = (int)((hw >> 20) & 0x7ffu), ef = e - 896;
  if (e == 0) return 0.0f;
  if (ef <= 0 || ef >= 254) return __double2float_rn(x);
  const unsigned m23 = ((hw & 0xfffffu) << 3) | (lw >> 29), rem = lw & 0x1fffffffu;
  const unsigned inc = (rem > 0x10000000u || (rem == 0x10000000u && (m23 & 1u))) ? 1u : 0u;
  return __uint_as_float(((hw & 0x80000000u) | ((unsigned)ef << 23) | m23) + inc);  // a carry moves into the exponent
}

// The level copies of the stored linearisation in one pass over the FP64 words:
// the FP32 plane (lin32_word layout) and the BF16 words (lin16_word layout;
// words 70 and 71 zero), each optional.  All conversions are integer operations,
// so that the pass runs at HBM speed rather than at the FP64 rate of the
// conversion instructions.  One thread per octet of a point's words [0, 64)
// (eight coalesced FP64 reads; two 128-bit writes for the plane, one for the BF16
// octet), then one per tail plane of four words.  Writing these copies from the
// pointwise kernel instead measured slower (64^3 Q4 residual 154 -> 176 ms): its
// scattered narrow stores cost more than this pass.
__global__ void k_level_words(const double* __restrict__ a, float* __restrict__ w32, uint16_t* __restrict__ b16,
                              long long nblk, long long q3eb) {
  const long long bw = (long long)kLinWords * q3eb, ow = (long long)kLin16Words * q3eb;
  const long long opb = 8 * q3eb, tpb = 2 * q3eb;  // octet / tail units per block
  const long long no = nblk * opb, n = no + nblk * tpb;
  for (long long u = blockIdx.x * (long long)blockDim.x + threadIdx.x; u < n; u += (long long)gridDim.x * blockDim.x) {
    if (u < no) {
      const long long b = u / opb, rem = u % opb;
      const long long oc = rem / q3eb, r2 = rem % q3eb;
      const double* src = a + b * bw + 8 * oc * q3eb + r2;
      double x[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) x[c] = src[c * q3eb];
      if (w32) {
#pragma unroll
        for (int g = 0; g < 2; ++g)
          *reinterpret_cast<float4*>(w32 + b * bw + (2 * oc + g) * 4 * q3eb + 4 * r2) =
              make_float4(f32_rne(x[4 * g]), f32_rne(x[4 * g + 1]), f32_rne(x[4 * g + 2]), f32_rne(x[4 * g + 3]));
      }
      if (b16) {
        unsigned v[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) v[c] = bf16_rne(x[2 * c]) | (bf16_rne(x[2 * c + 1]) << 16);
        *reinterpret_cast<uint4*>(b16 + b * ow + oc * 8 * q3eb + 8 * r2) = make_uint4(v[0], v[1], v[2], v[3]);
      }
    } else {
      const long long w = u - no, b = w / tpb, rem = w % tpb;
      const long long tp = rem / q3eb, r2 = rem % q3eb;
      unsigned v[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int wd = 64 + 4 * (int)tp + c;
        v[c] = 0u;
        if (wd < kLinWords) {
          const long long i = b * bw + wd * q3eb + r2;
          const double x = a[i];
          if (w32) w32[i] = f32_rne(x);
          v[c] = bf16_rne(x);
        }
      }
      if (b16)
        *reinterpret_cast<uint2*>(b16 + b * ow + (64 + 4 * tp) * q3eb + 4 * r2) =
            make_uint2(v[0] | (v[1] << 16), v[2] | (v[3] << 16));
    }
  }
}
cudaError_t launch_level_words(const double* a, float* w32, uint16_t* b16, long long nblk, int Q, cudaStream_t st) {
  if (nblk == 0 || (!w32 && !b16)) return cudaSuccess;
  const long long q3eb = (long long)Q * Q * Q * elems_per_block(Q);
  const long long n = nblk * 10 * q3eb;
  k_level_words<<<grid_for(n), kVecThreads, 0, st>>>(a, w32, b16, nblk, q3eb); note_launch();
  return cudaGetLastError();
}

// Chebyshev iteration (Saad, Alg. 12.1) on D^-1 A, between products:
//   first: r = D^-1 (b - A x),  d = r / theta          (A x absent: x = 0)
//   next:  x += d (xset: x = d);  r -= D^-1 A d;  d = c_d d + c_r r
//          last: x += that d too, which ends the smoothing (r, d not written)
//   only:  x += D^-1 (b - A x) / theta, a smoothing of degree one (xset: x = that)
// The first two leave in Ad what the action expects there, its next input's prescribed
// entries and zeros elsewhere, so that no pass of its own prepares it.  Bound by
// HBM: a degree-3 smoothing moves 21 vectors instead of 30 (64 bit or 32 bit;
// 40^3 Q4 FP32, 67 MB each: 383 -> 226 us with the clears).  V entries per thread, 16-byte
// accesses where every pointer allows them.
template <typename T, int V> struct alignas(sizeof(T) * V) VecOf { T v[V]; };

// As first with an axpby in FP64 arithmetic, which moves ten vectors instead of five,
// a smoothing of degree one took 354 us at 32x31x33 Q4 FP32 (341 us with separate
// updates), now 264 us.
template <typename T, int V>
__global__ void __launch_bounds__(kVecThreads) k_cheb_only(long long n, const T* b, const T* Ax, const T* diag, T* x,
                                                           T inv_theta, int xset) {
  using W = VecOf<T, V>;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n / V; i += (long long)gridDim.x * blockDim.x) {
    const W bi = reinterpret_cast<const W*>(b)[i], gi = reinterpret_cast<const W*>(diag)[i];
    W ax, xi;
    if (Ax) ax = reinterpret_cast<const W*>(Ax)[i];
    if (!xset) xi = reinterpret_cast<const W*>(x)[i];
#pragma unroll
    for (int c = 0; c < V; ++c) {
      const T d = (Ax ? bi.v[c] - ax.v[c] : bi.v[c]) / gi.v[c] * inv_theta;
      xi.v[c] = xset ? d : xi.v[c] + d;
    }
    reinterpret_cast<W*>(x)[i] = xi;
  }
}
template <typename T, int V>
__global__ void __launch_bounds__(kVecThreads) k_cheb_first(long long n, const T* b, const T* Ax, const T* diag,
                                                            const uint8_t* mask, T* r, T* d, T* Ad, T inv_theta) {
  using W = VecOf<T, V>;
  using M = VecOf<uint8_t, V>;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n / V; i += (long long)gridDim.x * blockDim.x) {
    const W bi = reinterpret_cast<const W*>(b)[i], gi = reinterpret_cast<const W*>(diag)[i];
    W ax, ri, di, ai;
    M m;
    if (Ax) ax = reinterpret_cast<const W*>(Ax)[i];
    if (mask) m = reinterpret_cast<const M*>(mask)[i];
#pragma unroll
    for (int c = 0; c < V; ++c) {
      ri.v[c] = (Ax ? bi.v[c] - ax.v[c] : bi.v[c]) / gi.v[c];
      di.v[c] = ri.v[c] * inv_theta;
      ai.v[c] = mask && m.v[c] ? di.v[c] : T(0);
    }
    reinterpret_cast<W*>(r)[i] = ri;
    reinterpret_cast<W*>(d)[i] = di;
    reinterpret_cast<W*>(Ad)[i] = ai;
  }
}
template <typename T, int V, bool LAST>
__global__ void __launch_bounds__(kVecThreads) k_cheb_next(long long n, T* x, T* d, T* r, T* Ad, const T* diag,
                                                           const uint8_t* mask, T c_d, T c_r, int xset) {
  using W = VecOf<T, V>;
  using M = VecOf<uint8_t, V>;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n / V; i += (long long)gridDim.x * blockDim.x) {
    W di = reinterpret_cast<const W*>(d)[i], ri = reinterpret_cast<const W*>(r)[i];
    const W gi = reinterpret_cast<const W*>(diag)[i];
    W ai = reinterpret_cast<const W*>(Ad)[i], xi;
    M m;
    if (!xset) xi = reinterpret_cast<const W*>(x)[i];
    if (!LAST && mask) m = reinterpret_cast<const M*>(mask)[i];
#pragma unroll
    for (int c = 0; c < V; ++c) {
      xi.v[c] = xset ? di.v[c] : xi.v[c] + di.v[c];
      ri.v[c] -= ai.v[c] / gi.v[c];
      di.v[c] = c_d * di.v[c] + c_r * ri.v[c];
      if (LAST) xi.v[c] += di.v[c];
      else ai.v[c] = mask && m.v[c] ? di.v[c] : T(0);
    }
    reinterpret_cast<W*>(x)[i] = xi;
    if (!LAST) {
      reinterpret_cast<W*>(r)[i] = ri;
      reinterpret_cast<W*>(d)[i] = di;
      reinterpret_cast<W*>(Ad)[i] = ai;
    }
  }
}
static bool aligned16(std::initializer_list<const void*> ps) {
  uintptr_t u = 0;
  for (const void* p : ps) u |= reinterpret_cast<uintptr_t>(p);
  return u % 16 == 0;
}
template <typename T>
cudaError_t launch_cheb_first(long long n, const T* b, const T* Ax, const T* diag, const uint8_t* mask, T* r, T* d,
                              T* Ad, double inv_theta, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  constexpr int V = 16 / sizeof(T);
  if (n % V == 0 && aligned16({b, Ax, diag, mask, r, d, Ad}))
    k_cheb_first<T, V><<<grid_for(n / V), kVecThreads, 0, st>>>(n, b, Ax, diag, mask, r, d, Ad, (T)inv_theta);
  else
    k_cheb_first<T, 1><<<grid_for(n), kVecThreads, 0, st>>>(n, b, Ax, diag, mask, r, d, Ad, (T)inv_theta);
  note_launch();
  return cudaGetLastError();
}
template <typename T>
cudaError_t launch_cheb_only(long long n, const T* b, const T* Ax, const T* diag, T* x, double inv_theta, int xset,
                             cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  constexpr int V = 16 / sizeof(T);
  if (n % V == 0 && aligned16({b, Ax, diag, x}))
    k_cheb_only<T, V><<<grid_for(n / V), kVecThreads, 0, st>>>(n, b, Ax, diag, x, (T)inv_theta, xset);
  else
    k_cheb_only<T, 1><<<grid_for(n), kVecThreads, 0, st>>>(n, b, Ax, diag, x, (T)inv_theta, xset);
  note_launch();
  return cudaGetLastError();
}
template <typename T>
cudaError_t launch_cheb_next(long long n, T* x, T* d, T* r, T* Ad, const T* diag, const uint8_t* mask, double c_d,
                             double c_r, int xset, int last, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  constexpr int V = 16 / sizeof(T);
  const bool wide = n % V == 0 && aligned16({x, d, r, Ad, diag, mask});
  const unsigned nb = grid_for(wide ? n / V : n);
  if (wide && last) k_cheb_next<T, V, true><<<nb, kVecThreads, 0, st>>>(n, x, d, r, Ad, diag, mask, (T)c_d, (T)c_r, xset);
  else if (wide) k_cheb_next<T, V, false><<<nb, kVecThreads, 0, st>>>(n, x, d, r, Ad, diag, mask, (T)c_d, (T)c_r, xset);
  else if (last) k_cheb_next<T, 1, true><<<nb, kVecThreads, 0, st>>>(n, x, d, r, Ad, diag, mask, (T)c_d, (T)c_r, xset);
  else k_cheb_next<T, 1, false><<<nb, kVecThreads, 0, st>>>(n, x, d, r, Ad, diag, mask, (T)c_d, (T)c_r, xset);
  note_launch();
  return cudaGetLastError();
}
template cudaError_t launch_cheb_first<double>(long long, const double*, const double*, const double*, const uint8_t*,
                                               double*, double*, double*, double, cudaStream_t);
template cudaError_t launch_cheb_first<float>(long long, const float*, const float*, const float*, const uint8_t*,
                                              float*, float*, float*, double, cudaStream_t);
template cudaError_t launch_cheb_only<double>(long long, const double*, const double*, const double*, double*, double,
                                              int, cudaStream_t);
template cudaError_t launch_cheb_only<float>(long long, const float*, const float*, const float*, float*, double, int,
                                             cudaStream_t);
template cudaError_t launch_cheb_next<double>(long long, double*, double*, double*, double*, const double*,
                                              const uint8_t*, double, double, int, int, cudaStream_t);
template cudaError_t launch_cheb_next<float>(long long, float*, float*, float*, float*, const float*, const uint8_t*,
                                             double, double, int, int, cudaStream_t);


// Stored linearisation from the tiled layout to the canonical order [67][N_q]
// (the off-diagonal phase-gradient words of mapped meshes are not exported).
__global__ void k_untile(const double* __restrict__ lin, double* __restrict__ out, long long nq, int Q) {
  const long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (q >= nq) return;
  const int Q2 = Q * Q, Q3 = Q2 * Q, EB = elems_per_block(Q);
  const long long e = q / Q3;
  const int lq = (int)(q % Q3);
  const int i = lq % Q, j = (lq / Q) % Q, k = lq / Q2;
  const long long stride = (long long)Q3 * EB;
  const long long base = (e / EB) * kLinWords * stride + (long long)k * Q2 * EB + (e % EB) * Q2 + j * Q + i;
  for (int w = 0; w < kLinWordsExport; ++w) out[w * nq + q] = lin[base + w * stride];
}
cudaError_t launch_untile(const double* lin, double* out, long long nq, int Q, cudaStream_t st) {
  if (nq == 0) return cudaSuccess;
  k_untile<<<(unsigned)((nq + 255) / 256), 256, 0, st>>>(lin, out, nq, Q); note_launch();
  return cudaGetLastError();
}


// z = ubar on Dirichlet DoFs (other entries untouched).
__global__ void k_apply_dirichlet(double* __restrict__ z, const double* __restrict__ ubar,
                                  const uint8_t* __restrict__ mask, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    if (mask[i]) z[i] = ubar ? ubar[i] : 0.0;
}
cudaError_t launch_apply_dirichlet(double* z, const double* ubar, const uint8_t* mask, long long n, cudaStream_t st) {
  if (n == 0 || !mask) return cudaSuccess;
  k_apply_dirichlet<<<grid_for(n), kVecThreads, 0, st>>>(z, ubar, mask, n); note_launch();
  return cudaGetLastError();
}

// out[f] += sum over nodes n with sel[f][n] of v[f][n] (FP64, per-block partial
// sums combined with atomics).
__global__ void k_masked_field_sums(const double* __restrict__ v, const uint8_t* __restrict__ sel, long long nn,
                                    double* __restrict__ out) {
  __shared__ double red[4][kVecThreads / 32];
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nn; i += (long long)gridDim.x * blockDim.x)
    for (int f = 0; f < 4; ++f)
      if (sel[f * nn + i]) s[f] += v[f * nn + i];
  for (int f = 0; f < 4; ++f) {
    double t = s[f];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) red[f][threadIdx.x >> 5] = t;
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    double t = 0.0;
    for (int w = 0; w < kVecThreads / 32; ++w) t += red[threadIdx.x][w];
    atomicAdd(out + threadIdx.x, t);
  }
}
cudaError_t launch_masked_field_sums(const double* v, const uint8_t* sel, long long nn, double* out, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(out, 0, 4 * sizeof(double), st);
  if (e != cudaSuccess || nn == 0) return e;
  k_masked_field_sums<<<grid_for(nn), kVecThreads, 0, st>>>(v, sel, nn, out); note_launch();
  return cudaGetLastError();
}

// State summary of a load step (the per-step log): out[0..2] = points whose
// flags have bit 0 (Prandtl yield), bit 1 (history active), bit 2 (theta >=
// 0); out[3], out[4] = largest and smallest nodal phase field; out[5] = nodes
// with phi > 0.9; out[6], out[7] = largest accumulated plastic strain and
// history field of the given history.  One block-reduced pass per quantity.
__device__ __forceinline__ void atomic_max_d(double* a, double v) {
  unsigned long long* p = reinterpret_cast<unsigned long long*>(a);
  unsigned long long old = *p;
  while (v > __longlong_as_double((long long)old)) {
    const unsigned long long prev = atomicCAS(p, old, (unsigned long long)__double_as_longlong(v));
    if (prev == old) break;
    old = prev;
  }
}
__device__ __forceinline__ void atomic_min_d(double* a, double v) {
  unsigned long long* p = reinterpret_cast<unsigned long long*>(a);
  unsigned long long old = *p;
  while (v < __longlong_as_double((long long)old)) {
    const unsigned long long prev = atomicCAS(p, old, (unsigned long long)__double_as_longlong(v));
    if (prev == old) break;
    old = prev;
  }
}
__global__ void k_state_summary(const uint8_t* __restrict__ flags, const double* __restrict__ hist, long long nq,
                                const double* __restrict__ phi, long long nn, double* __restrict__ out) {
  double cnt[3] = {0.0, 0.0, 0.0}, hi = -INFINITY, lo = INFINITY, n9 = 0.0, ep = -INFINITY, H = -INFINITY;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < nq; q += stride) {
    const unsigned f = flags[q];
    cnt[0] += (f & 1u) ? 1.0 : 0.0;
    cnt[1] += (f & 2u) ? 1.0 : 0.0;
    cnt[2] += (f & 4u) ? 1.0 : 0.0;
    ep = fmax(ep, hist[12 * nq + q]);
    H = fmax(H, hist[13 * nq + q]);
  }
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < nn; n += stride) {
    const double v = phi[n];
    hi = fmax(hi, v);
    lo = fmin(lo, v);
    n9 += (v > 0.9) ? 1.0 : 0.0;
  }
  for (int off = 16; off > 0; off >>= 1) {
    for (int c = 0; c < 3; ++c) cnt[c] += __shfl_down_sync(0xffffffffu, cnt[c], off);
    hi = fmax(hi, __shfl_down_sync(0xffffffffu, hi, off));
    lo = fmin(lo, __shfl_down_sync(0xffffffffu, lo, off));
    n9 += __shfl_down_sync(0xffffffffu, n9, off);
    ep = fmax(ep, __shfl_down_sync(0xffffffffu, ep, off));
    H = fmax(H, __shfl_down_sync(0xffffffffu, H, off));
  }
  if ((threadIdx.x & 31) == 0) {
    for (int c = 0; c < 3; ++c) atomicAdd(out + c, cnt[c]);
    atomic_max_d(out + 3, hi);
    atomic_min_d(out + 4, lo);
    atomicAdd(out + 5, n9);
    atomic_max_d(out + 6, ep);
    atomic_max_d(out + 7, H);
  }
}
__global__ void k_state_summary_init(double* out) {
  if (threadIdx.x < 8) out[threadIdx.x] = (threadIdx.x == 3 || threadIdx.x >= 6) ? -INFINITY
                                          : (threadIdx.x == 4 ? INFINITY : 0.0);
}
cudaError_t launch_state_summary(const uint8_t* flags, const double* hist, long long nq, const double* phi,
                                 long long nn, double* out, cudaStream_t st) {
  k_state_summary_init<<<1, 32, 0, st>>>(out); note_launch();
  k_state_summary<<<grid_for(nq > nn ? nq : nn), kVecThreads, 0, st>>>(flags, hist, nq, phi, nn, out); note_launch();
  return cudaGetLastError();
}


// Geometry of a mapped mesh at every quadrature point from the parent Jacobian
// J = dX / dxi (rows 3 f + al of an eval of the nodal coordinates):
// geo[3 al + A] = (J^-1)[al][A] = d xi_al / dX_A, geo[9] = w_q det J.
__global__ void k_geometry(const double* __restrict__ J, double* __restrict__ geo, Geom g, int Q, long long nq,
                           int* __restrict__ status) {
  const long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (q >= nq) return;
  double A[3][3];
  for (int f = 0; f < 3; ++f)
    for (int al = 0; al < 3; ++al) A[f][al] = J[(3 * f + al) * nq + q];
  const double det = A[0][0] * (A[1][1] * A[2][2] - A[1][2] * A[2][1]) - A[0][1] * (A[1][0] * A[2][2] - A[1][2] * A[2][0]) +
                     A[0][2] * (A[1][0] * A[2][1] - A[1][1] * A[2][0]);
  if (!(det > 0.0)) atomicOr(status, 2);
  const double r = 1.0 / det;
  double G[3][3];
  G[0][0] = (A[1][1] * A[2][2] - A[1][2] * A[2][1]) * r;
  G[0][1] = (A[0][2] * A[2][1] - A[0][1] * A[2][2]) * r;
  G[0][2] = (A[0][1] * A[1][2] - A[0][2] * A[1][1]) * r;
  G[1][0] = (A[1][2] * A[2][0] - A[1][0] * A[2][2]) * r;
  G[1][1] = (A[0][0] * A[2][2] - A[0][2] * A[2][0]) * r;
  G[1][2] = (A[0][2] * A[1][0] - A[0][0] * A[1][2]) * r;
  G[2][0] = (A[1][0] * A[2][1] - A[1][1] * A[2][0]) * r;
  G[2][1] = (A[0][1] * A[2][0] - A[0][0] * A[2][1]) * r;
  G[2][2] = (A[0][0] * A[1][1] - A[0][1] * A[1][0]) * r;
  for (int al = 0; al < 3; ++al)
    for (int B = 0; B < 3; ++B) geo[(3 * al + B) * nq + q] = G[al][B];
  const int Q2 = Q * Q;
  const int lq = (int)(q % ((long long)Q2 * Q));
  geo[9 * nq + q] = g.wq[lq % Q] * g.wq[(lq / Q) % Q] * g.wq[lq / Q2] * det;
}
cudaError_t launch_geometry(const double* J, double* geo, const Geom& g, int Q, long long nq, int* status,
                            cudaStream_t st) {
  if (nq == 0) return cudaSuccess;
  k_geometry<<<(unsigned)((nq + 255) / 256), 256, 0, st>>>(J, geo, g, Q, nq, status); note_launch();
  return cudaGetLastError();
}

}  // namespace pff
