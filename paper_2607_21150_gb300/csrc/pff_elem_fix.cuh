// FP64 element kernels (Sec. 4): the Jacobian action, the evaluation of the state
// at the Gauss points and the transposed contraction of the residual integrands,
// with the tensor contractions in 64-bit fixed point on the integer pipes.
//
// What bounds them on GB300 is the FP64 pipe: two multiply-adds per clock and SM,
// 64 issue slots per warp instruction, of which a contraction needs 240 per
// point (Q4) and the pointwise map 103.  A contraction with a constant 1D matrix
// needs no floating point, though: the values of a field in an element share one
// exponent (that of its largest entry), a matrix entry is an integer b = B 2^s,
// and with both split into 30-bit halves a multiply-add is three 32 x 32 + 64-bit
// integer ones (high x high, two cross products; low x low is below one unit in
// the last place), about a quarter of the FP64 pipe's time, on a pipe that works
// beside it.  The map of the stored words stays in FP64.
//
// Precision: an entry keeps about 59 bits (FixTab) below its element's largest, or
// below the bound of the derivative sums in the transposed direction; every
// product sum is exact up to one rounding of the last place.  Against 128-bit
// arithmetic with the same words (Q2..Q4, uniform, smooth and widely varying
// vectors) the action errs no more than FP64 contractions did.  Values are
// converted by integer operations too, rounded to nearest.  Non-finite entries
// make their field's values NaN in the element, as the dense contractions did.
//
// A block takes fix_elems(Q) elements (128 to 192 threads) of a group of
// elems_per_block(Q) that the stored words are tiled by.  A thread is a node in
// the gather and the scatter, a line in the contractions (4 Q^2 lines) and a
// Gauss point in the map, Q^3 threads per element: up to 30 warps per SM whose
// integer and FP64 phases overlap, and short serial chains on meshes of a few
// elements.  The 1D matrices are kernel parameters (constant-bank operands).
//
// Measured, 64^3 Q4 action: 20.08 ms with FP64 contractions (88.7 % of the FP64
// pipe), 7.64 ms now; the map alone is 5.4 ms of that pipe (ncu, 24^3: pipe 74 %
// busy, issue 55 %, DRAM 31 %).  With one thread per column of points (12 warps
// per SM, as the FP64 kernel had it) 17 ms; with one copy of the line code per
// direction instead of loops over the directions 9.1 ms (instruction cache).
// 4^3 Q2: 56 -> 13.3 us (64 elements in 21 blocks instead of three).
#pragma once
#include "pff_df.cuh"
#include "pff_internal.h"

namespace pff {

__device__ __forceinline__ void fx_split(long long x, int& h, int& l) {
  h = (int)((x + (1LL << 29)) >> 30);
  l = (int)((unsigned)x - ((unsigned)h << 30));
}

// c + a b in 64 bits, one instruction.
__device__ __forceinline__ long long fx_mad(int a, int b, long long c) {
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}
// out[q] = sum_p M[q][p] in[p] (TR: sum over the matrix's first index) in units
// of the last place, rounded to nearest; in and out at the given strides.
template <int NI, int NO, bool TR>
__device__ __forceinline__ void fx_line(const int* Mh, const int* Ml, const long long* in, int is, long long* out,
                                        int os) {
  int h[NI], l[NI];
#pragma unroll
  for (int p = 0; p < NI; ++p) fx_split(in[p * is], h[p], l[p]);
#pragma unroll
  for (int q = 0; q < NO; ++q) {
    long long A = 0, C = 1LL << 29;
#pragma unroll
    for (int p = 0; p < NI; ++p) {
      const int m = TR ? p * NO + q : q * NI + p;
      A = fx_mad(h[p], Mh[m], A);
      C = fx_mad(h[p], Ml[m], C);
      C = fx_mad(l[p], Mh[m], C);
    }
    out[q * os] = A + (C >> 30);
  }
}

// Biased exponent of x (subnormals count as 1, zero as 0, non-finite 2047).
__device__ __forceinline__ int fx_exponent(double x) {
  const unsigned hi = (unsigned)__double2hiint(x) & 0x7fffffffu;
  const int e = (int)(hi >> 20);
  return e ? e : (hi | (unsigned)__double2loint(x)) ? 1 : 0;
}
// x in units of 2^(emax - 1022 - w) (|x| < 2^(emax - 1022) is at most 2^w); the
// result is below 2^62.
__device__ __forceinline__ long long fx_from(double x, int emax, int w) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int e = (int)((hi >> 20) & 0x7ffu);
  // significand with its leading bit at 62, then one right shift (at least one)
  // and the rounding
  const unsigned sg = (hi & 0xfffffu) | (e ? 0x100000u : 0u);
  const unsigned long long m = ((unsigned long long)__funnelshift_l(lo, sg, 10) << 32) | (lo << 10);
  const int sh = emax - (e ? e : 1) + 62 - w;
  const unsigned long long r = sh > 63 ? 0ull : ((m >> sh) + 1) >> 1;
  return (int)hi < 0 ? -(long long)r : (long long)r;
}
// m 2^ex rounded to nearest; orv: bits set in the result (NaN of a non-finite
// field).  Results near the ends of the exponent range are scaled by the library.
static __device__ __noinline__ double fx_scale(double x, int ex) { return scalbn(x, ex); }
__device__ __forceinline__ double fx_to(long long m, int ex, int orv) {
  const unsigned long long u = m < 0 ? 0ull - (unsigned long long)m : (unsigned long long)m;
  unsigned hi = (unsigned)(u >> 32), lo = (unsigned)u;
  const bool far = ex < -1000 || ex > 900;
  int be = 1022 + 63 + (far ? 0 : ex);  // biased exponent of a leading bit at 63, less one
  if (hi == 0u) {
    hi = lo;
    lo = 0u;
    be -= 32;
  }
  const int lz = __clz((int)hi);
  be -= lz;
  hi = __funnelshift_l(lo, hi, lz);
  lo <<= lz & 31;
  // 53 bits with the leading one, rounded half up; a carry moves into the exponent
  const unsigned rl = __funnelshift_r(lo, hi, 11), up = (lo >> 10) & 1u;
  const unsigned sl = rl + up;
  unsigned sh = ((unsigned)be << 20) + (hi >> 11) + (sl < rl ? 1u : 0u);
  sh = hi ? sh : 0u;
  double r = __hiloint2double((int)(sh | (unsigned)((int)(m >> 32) & 0x80000000)), (int)(hi ? sl : 0u));
  if (far) r = fx_scale(r, ex);
  return __hiloint2double(__double2hiint(r) | orv, __double2loint(r));
}
constexpr int kFxNan = 0x7ff80000;
// *m = max(*m, v) over the threads of an element: by warp where a warp holds one
// element only (Q >= 4), so that the shared atomics do not queue up (for Q = 3 a
// reduction over the lanes of each element measured slower than the atomics).
// Every thread of the block calls it, and those warps are full (fix_threads): all
// lanes are named, so that lane 0 has the whole warp's maximum whatever branches
// went before.  With 29 lanes in the last warp of Q = 5 and their mask here,
// 64^3 Q4 took 7.95 ms instead of 7.72.
template <int Q> __device__ __forceinline__ void fx_max(int* m, int v) {
  if (Q >= 4) {
    v = __reduce_max_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) atomicMax(m, v);
  } else {
    atomicMax(m, v);
  }
}

// Shared memory per element: A, four fields of Q^3; B, eight of Q^3 (the x- and
// y-derivatives, or a ping-pong buffer of the contractions); C, Q^3 (the value
// term of the phase field).
template <int Q> __host__ __device__ constexpr int fix_elem_words() { return 13 * Q * Q * Q; }
// Resident blocks the register allocation is held to: about 30 warps per SM
// (40x33x37 elements, 20 / 24 / 30 / 36 warps: Q2 376 / 335 / 316 / 326 us, Q3 - /
// 657 / 645 / 681 us, Q4 - / 1493 / 1495 / 1564 us).
__host__ __device__ constexpr int fix_blocks(int threads) { return 30 / ((threads + 31) / 32); }

template <int P, int Q, int MODE, int EBS>
__global__ void __launch_bounds__(fix_threads(Q, EBS), fix_blocks(fix_threads(Q, EBS)))
k_elem_fix(const ElemArgs<double> a) {
  constexpr int EB = elems_per_block(Q), NSUB = EB / EBS;
  constexpr int Q2 = Q * Q, Q3 = Q * Q * Q, P2 = P * P, P3 = P * P * P;
  static_assert(NSUB * EBS == EB, "a block's elements divide the group");
  static_assert(Q < 4 || Q3 % 32 == 0 || EBS == 1, "fx_max: one element per warp");
  __shared__ long long sm[EBS * fix_elem_words<Q>()];
  __shared__ int emax[EBS][12];  // exponents: x per field, [4..7] gradient outputs, [8] value output
  constexpr int NT = fix_threads(Q, EBS);
  const int t = threadIdx.x;
  const bool live = NT == Q3 * EBS || t < Q3 * EBS;  // the others fill the last warp of Q = 5
  const int el = EBS == 1 ? 0 : t / Q3, pt = EBS == 1 ? t : t % Q3;  // element, and node or point of it
  const long long grp = a.blk0 + blockIdx.x / NSUB;
  const int sub = blockIdx.x % NSUB;
  const int e = (int)(grp * EB) + sub * EBS + el;
  const bool valid = live && e < a.mesh.nel;
  const long long nn = a.mesh.nn;
  const FixTab& fx = a.fix;
  const int dd = 60 - fx.sD;
  long long* A = sm + el * fix_elem_words<Q>();
  long long* B = A + 4 * Q3;
  double* C = reinterpret_cast<double*>(B + 8 * Q3);
  if (Q == 2 ? pt < 4 : pt < 12) emax[el][pt] = 0;
  if (Q == 2 && pt < 8) emax[el][4 + pt] = 0;
  __syncthreads();

  const bool masked = a.mask && valid && (!a.emask || a.emask[e]);
  const bool node = valid && pt < P3;
  long long n = 0;
  if (MODE != kEval || node) n = node ? node_of<P, Q>(a.mesh, e, pt % P, (pt / P) % P, pt / P2) : 0;
  // gather, and which entries are prescribed: bytes that only elements with
  // masked nodes load, all of them at once, and that the scatter finds here
  double phi = 0.0, xv[4] = {0.0, 0.0, 0.0, 0.0};
  bool fixed[4] = {false, false, false, false};
  if (MODE != kBack && node)
#pragma unroll
    for (int f = 0; f < 4; ++f) xv[f] = __ldg(a.x + f * nn + n);
  if (masked && node)
#pragma unroll
    for (int f = 0; f < 4; ++f) fixed[f] = __ldg(a.mask + f * nn + n);
  if constexpr (MODE != kBack) {
    // prescribed entries zero; the fields' exponents
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      if (fixed[f]) xv[f] = 0.0;
      fx_max<Q>(&emax[el][f], fx_exponent(xv[f]));
    }
    __syncthreads();
    if (pt < P3)
#pragma unroll
      for (int f = 0; f < 4; ++f) A[f * Q3 + pt] = fx_from(xv[f], emax[el][f], fx.wf);
    __syncthreads();
    // interpolation: x [c][b][a] -> B [c][b][i], y -> A [c][j][i], z in place
    // [k][j][i] (one copy of the line's code for the three: the instruction cache)
#pragma unroll 1
    for (int d = 0; d < 3; ++d) {
      const int lines = P == Q ? Q2 : d == 0 ? P2 : d == 1 ? P * Q : Q2, is = d == 0 ? 1 : d == 1 ? Q : Q2;
#pragma unroll 1
      for (int L = t; L < 4 * EBS * lines; L += NT) {
        const int ef = P == Q ? L / Q2 : d == 0 ? L / P2 : d == 1 ? L / (P * Q) : L / Q2, r = L - ef * lines;
        long long* S = sm + (EBS == 1 ? ef * Q3 : ef / 4 * fix_elem_words<Q>() + ef % 4 * Q3);
        const long long* in = (d == 1 ? S + 4 * Q3 : S) + (d == 0 ? r * P : d == 1 ? r / Q * (P * Q) + r % Q : r);
        long long* out = (d == 0 ? S + 4 * Q3 : S) + (d == 0 ? r * Q : d == 1 ? r / Q * Q2 + r % Q : r);
        fx_line<P, Q, false>(fx.Bh, fx.Bl, in, is, out, is);
      }
      __syncthreads();
    }
    // collocated derivatives: x and y into B, then (the point's phase field kept)
    // z in place
    phi = fx_to(A[3 * Q3 + pt], emax[el][3] - 1022 - fx.wf, emax[el][3] == 2047 ? kFxNan : 0);
#pragma unroll 1
    for (int d = 0; d < 3; ++d) {
      if (d == 2) __syncthreads();
#pragma unroll 1
      for (int L = t; L < 4 * EBS * Q2; L += NT) {
        const int ef = L / Q2, r = L % Q2, f = EBS == 1 ? ef : ef % 4;
        long long *A = sm + (EBS == 1 ? 0 : ef / 4 * fix_elem_words<Q>()), *B = A + 4 * Q3;
        const int o = d == 0 ? r * Q : d == 1 ? r / Q * Q2 + r % Q : r;  // lines (k, j), (k, i), (j, i)
        fx_line<Q, Q, false>(fx.Dh, fx.Dl, A + f * Q3 + o, d == 0 ? 1 : d == 1 ? Q : Q2,
                             d == 2 ? A + f * Q3 + o : B + (2 * f + d) * Q3 + o, d == 0 ? 1 : d == 1 ? Q : Q2);
      }
    }
    __syncthreads();
  }

  // the point's gradients from its slots; its outputs (FP64 bits) back into them
  {
    const long long q = (long long)e * Q3 + pt;
    double g[4][3], o[4][3], v0 = 0.0;
    if constexpr (MODE != kBack) {
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        const int ef = emax[el][f], ex = ef - 1022 - fx.wf + dd, nan = ef == 2047 ? kFxNan : 0;
        g[f][0] = fx_to(B[2 * f * Q3 + pt], ex, nan);
        g[f][1] = fx_to(B[(2 * f + 1) * Q3 + pt], ex, nan);
        g[f][2] = fx_to(A[f * Q3 + pt], ex, nan);
      }
    }
    if constexpr (MODE == kEval) {
      if (!valid) return;
      if (a.geo) {  // mapped mesh: reference gradient = parent gradient x d xi / dX
        double G[3][3];
#pragma unroll
        for (int al = 0; al < 3; ++al)
#pragma unroll
          for (int X = 0; X < 3; ++X) G[al][X] = a.geo[(3 * al + X) * a.nq + q];
#pragma unroll
        for (int f = 0; f < 4; ++f)
#pragma unroll
          for (int X = 0; X < 3; ++X)
            a.scratch[((f < 3) ? 3 * f + X : 10 + X) * a.nq + q] = g[f][0] * G[0][X] + g[f][1] * G[1][X] + g[f][2] * G[2][X];
      } else {
#pragma unroll
        for (int f = 0; f < 4; ++f)
#pragma unroll
          for (int al = 0; al < 3; ++al)
            a.scratch[((f < 3) ? 3 * f + al : 10 + al) * a.nq + q] = g[f][al] * a.s[al];
      }
      a.scratch[9 * a.nq + q] = phi;
      return;
    } else {
      if (valid) {
        if constexpr (MODE == kApply) {
          constexpr long long run = (long long)Q2 * EB, stride = run * Q;
          const long long off = grp * kLinWords * stride + (pt / Q2) * run + (sub * EBS + el) * Q2 + pt % Q2;
          jac_point(a.lin + off, a.linP + off, a.linC + off, stride, a.kx, g, phi, o, v0);
        } else {  // integrands from the pointwise kernel
#pragma unroll
          for (int f = 0; f < 4; ++f)
#pragma unroll
            for (int al = 0; al < 3; ++al) o[f][al] = a.scratch[((f < 3) ? 3 * f + al : 10 + al) * a.nq + q];
          v0 = a.scratch[9 * a.nq + q];
        }
      } else {
#pragma unroll
        for (int f = 0; f < 4; ++f) o[f][0] = o[f][1] = o[f][2] = 0.0;
      }
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        if (live) {
          B[2 * f * Q3 + pt] = __double_as_longlong(o[f][0]);
          B[(2 * f + 1) * Q3 + pt] = __double_as_longlong(o[f][1]);
          A[f * Q3 + pt] = __double_as_longlong(o[f][2]);
        }
        fx_max<Q>(&emax[el][4 + f], max(fx_exponent(o[f][0]), max(fx_exponent(o[f][1]), fx_exponent(o[f][2]))));
      }
      if (live) C[pt] = v0;
      fx_max<Q>(&emax[el][8], fx_exponent(v0));
    }
  }
  __syncthreads();
  // exponent of the column sums of field f: three derivative sums (2^eD bounds
  // their weights) and, in the phase field, the value term
  auto sum_exponent = [&](int el, int f) {
    const int eg = emax[el][4 + f] + fx.eD;
    return f < 3 ? eg : max(eg, emax[el][8]) + 1;
  };
  // transposed derivatives: x and y lines in place, then the z lines, which sum
  // the three (and the value term) and contract z into A [c][j][i]
#pragma unroll 1
  for (int L = t; L < 4 * EBS * Q2; L += NT) {
    const int ef = L / Q2, r = L % Q2, f = EBS == 1 ? ef : ef % 4, ey = sum_exponent(EBS == 1 ? 0 : ef / 4, f);
    long long* B = sm + (EBS == 1 ? 0 : ef / 4 * fix_elem_words<Q>()) + 4 * Q3;
#pragma unroll 1
    for (int dir = 0; dir < 2; ++dir) {
      long long* ln = B + (2 * f + dir) * Q3 + (dir ? (r / Q) * Q2 + r % Q : r * Q);
      const int st = dir ? Q : 1;
      long long v[Q];
#pragma unroll
      for (int m = 0; m < Q; ++m) v[m] = fx_from(__longlong_as_double(ln[m * st]), ey, fx.wb + dd);
      fx_line<Q, Q, true>(fx.Dh, fx.Dl, v, 1, ln, st);
    }
  }
  __syncthreads();
#pragma unroll 1
  for (int L = t; L < 4 * EBS * Q2; L += NT) {
    const int ef = L / Q2, r = L % Q2, f = EBS == 1 ? ef : ef % 4, ey = sum_exponent(EBS == 1 ? 0 : ef / 4, f);
    long long *A = sm + (EBS == 1 ? 0 : ef / 4 * fix_elem_words<Q>()), *B = A + 4 * Q3;
    const double* C = reinterpret_cast<const double*>(B + 8 * Q3);
    long long* col = A + f * Q3 + r;
    long long v[Q], y[Q];
#pragma unroll
    for (int m = 0; m < Q; ++m) v[m] = fx_from(__longlong_as_double(col[m * Q2]), ey, fx.wb + dd);
    fx_line<Q, Q, true>(fx.Dh, fx.Dl, v, 1, y, 1);
#pragma unroll
    for (int m = 0; m < Q; ++m) {
      y[m] += B[2 * f * Q3 + m * Q2 + r] + B[(2 * f + 1) * Q3 + m * Q2 + r];
      if (f == 3) y[m] += fx_from(C[m * Q2 + r], ey, fx.wb);
    }
    fx_line<Q, P, true>(fx.Bh, fx.Bl, y, 1, col, Q2);
  }
  __syncthreads();
  // transposed interpolation: y -> B [c][b][i], x -> A [c][b][a]
#pragma unroll 1
  for (int d = 1; d >= 0; --d) {
    const int lines = d == 1 ? P * Q : P2;
#pragma unroll 1
    for (int L = t; L < 4 * EBS * lines; L += NT) {
      const int ef = P == Q ? L / Q2 : d == 1 ? L / (P * Q) : L / P2, r = L - ef * lines;
      long long* S = sm + (EBS == 1 ? ef * Q3 : ef / 4 * fix_elem_words<Q>() + ef % 4 * Q3);
      const long long* in = (d == 1 ? S : S + 4 * Q3) + (d == 1 ? r / Q * Q2 + r % Q : r * Q);
      long long* out = (d == 1 ? S + 4 * Q3 : S) + (d == 1 ? r / Q * (P * Q) + r % Q : r * P);
      fx_line<Q, P, true>(fx.Bh, fx.Bl, in, d == 1 ? Q : 1, out, d == 1 ? Q : 1);
    }
    __syncthreads();
  }
  if (!node) return;
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    const bool bad = emax[el][4 + f] == 2047 || (f == 3 && emax[el][8] == 2047);
    const double v = fx_to(A[f * Q3 + pt], sum_exponent(el, f) - 1022 - fx.wb, bad ? kFxNan : 0);
    if (a.evec)  // deterministic transpose: element-local values, summed per node by k_node_gather
      static_cast<double*>(a.evec)[((long long)e * 4 + f) * P3 + pt] = v;
    else if (!fixed[f])
      atomicAdd(a.y + f * nn + n, v);
  }
}

template <int P, int Q, int MODE, int EBS>
cudaError_t launch_fix(const ElemArgs<double>& a, int nblk, cudaStream_t st) {
  k_elem_fix<P, Q, MODE, EBS><<<(unsigned)nblk * (elems_per_block(Q) / EBS), fix_threads(Q, EBS), 0, st>>>(a); note_launch();
  return cudaGetLastError();
}
template <int P, int Q, int MODE>
cudaError_t launch_elem_fix(const ElemArgs<double>& a, int nblk, cudaStream_t st) {
  constexpr int big = fix_elems(Q, false), small = fix_elems(Q, true);
  if (small != big && nblk * (elems_per_block(Q) / big) < 2 * 152) return launch_fix<P, Q, MODE, small>(a, nblk, st);
  return launch_fix<P, Q, MODE, big>(a, nblk, st);
}

}  // namespace pff
