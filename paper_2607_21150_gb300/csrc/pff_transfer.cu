// p-transfer between a coarse level and a finer one on the same element grid:
// prolongation x_f = P x_c, P[f, c] = coarse Lagrange basis at the fine GLL node,
// and restriction r_c = P^T r_f (Sec. 5).
//
// Both are sum-factorised over a tile of elements in shared memory, one element
// layer and one field per block, and both are gathers: every fine (coarse) node
// is written by the one block that owns it, so that no transfer needs atomics, a
// cleared output or node multiplicities, and reruns give the same bits.  They are
// bound by the latency of the tiles' gathers and stages (L2 mostly: DRAM 4 % busy
// at 40x24x24).  The tile is 64 fine nodes wide (FP64: 32); its halo of one element
// width costs the restriction about a quarter more reads, and as a block takes one
// layer of vertices, it reads 2 p_f - 1 fine planes to own p_f (Q4: 7 for 4): about
// 2.2 times the fine vector in all.  Every loop has constant bounds
// (divisions by run-time widths made the kernels issue-bound: 107 and 87 us for the two) and
// the Dirichlet mask is read only by blocks that have flagged elements.  The end
// rows of the 1D matrix are those of the identity (both GLL sets hold -1 and 1),
// so shared nodes take no arithmetic.
//
// 48^3 Q4-Q2, FP32 (115 MB of fine vector): the former kernels evaluated the
// dense P^3 sums per fine node and per element-local coarse node from L2,
// 873 us for the prolongation and 829 us for the restriction; 81 and 90 us now.
#include <algorithm>
#include <type_traits>

#include "pff_internal.h"

namespace pff {

namespace {

template <typename T, int PF, int PC> struct XferW { T w[(PF + 1) * (PC + 1)]; };  // I1[a][b]

// Tile in elements: 64 fine nodes in x (FP64: 32), four element rows in y
// (prolongation in FP64: eight), so that a prolongation block has one item of its
// main stage per thread.
template <typename T, int PF> __host__ __device__ constexpr int tile_x() { return (sizeof(T) == 8 ? 32 : 64) / PF; }
template <typename T> __host__ __device__ constexpr int tile_yp() { return sizeof(T) == 8 ? 8 : 4; }
constexpr int kTileYr = 4;
constexpr int kXferThreads = 256;

// Whether an element of the box [x0, x1) x [y0, y1) x [z0, z1) has masked nodes
// (all of the block's threads get the answer; emask null: assume so).
__device__ __forceinline__ bool any_masked(const MeshDev& m, const uint8_t* emask, int x0, int x1, int y0, int y1,
                                           int z0, int z1) {
  x0 = max(x0, 0), y0 = max(y0, 0), z0 = max(z0, 0);
  x1 = min(x1, m.nx), y1 = min(y1, m.ny), z1 = min(z1, m.nz);
  int any = emask == nullptr;
  const int w = x1 - x0, h = y1 - y0;
  if (emask)
    for (int r = threadIdx.x / 32; r < h * (z1 - z0); r += kXferThreads / 32)
      for (int x = threadIdx.x % 32; x < w; x += 32)
        any |= emask[x0 + x + (long long)m.nx * (y0 + r % h + (long long)m.ny * (z0 + r / h))];
  return __syncthreads_or(any) != 0;
}

// Prolongation.  Stage x: coarse tile [c][J][I] -> [c][J][i] with i fine, one
// element of a row per item; then every thread takes a fine node i and an
// element row: y for its PF rows, z to the PF fine nodes of the layer (the
// weights are kernel parameters, constant-bank operands).
template <typename T, int PF, int PC, bool ADD>
__global__ void __launch_bounds__(kXferThreads)
k_prolong(MeshDev mc, MeshDev mf, const XferW<T, PF, PC> I1, const T* __restrict__ xc, T* xf,
          const uint8_t* __restrict__ maskc, const uint8_t* __restrict__ maskf, const uint8_t* __restrict__ emask) {
  constexpr int TX = tile_x<T, PF>(), TY = tile_yp<T>();
  constexpr int CX = PC * TX + 1, CY = PC * TY + 1, FX = PF * TX + 1;
  __shared__ T C[PC + 1][CY][CX];
  __shared__ T X[PC + 1][CY][FX];
  const int t = threadIdx.x, plane = mf.nnx * mf.nny;
  for (int zf = blockIdx.z; zf < 4 * mf.nz; zf += gridDim.z)
  for (int ey0 = blockIdx.y * TY; ey0 < mf.ny; ey0 += gridDim.y * TY) {
  const int ez = zf >> 2, f = zf & 3, ex0 = blockIdx.x * TX;
  __syncthreads();  // a former tile's values are read
  const int nex = min(TX, mf.nx - ex0), ney = min(TY, mf.ny - ey0);
  const int cw = PC * nex + 1, ch = PC * ney + 1;
  // a masked node of either level marks its elements (the fine flags cover the
  // fine mask, the coarse mask is read with the tile)
  const T* src = xc + f * mc.nn;
  const uint8_t* mk = maskc ? maskc + f * mc.nn : nullptr;
  const bool masked = maskf && any_masked(mf, emask, ex0, ex0 + TX, ey0, ey0 + TY, ez, ez + 1);
  for (int idx = t; idx < (PC + 1) * CY * CX; idx += kXferThreads) {
    const int I = idx % CX, r = idx / CX, J = r % CY, c = r / CY;
    if (I >= cw || J >= ch) continue;
    const long long n = PC * ex0 + I + (long long)mc.nnx * (PC * ey0 + J + (long long)mc.nny * (PC * ez + c));
    T v = src[n];
    if (mk && mk[n]) v = T(0);
    C[c][J][I] = v;
  }
  __syncthreads();
  for (int idx = t; idx < (PC + 1) * CY * TX; idx += kXferThreads) {
    const int e = idx % TX, r = idx / TX, J = r % CY, c = r / CY;
    if (e >= nex || J >= ch) continue;
    T v[PC + 1];
#pragma unroll
    for (int b = 0; b <= PC; ++b) v[b] = C[c][J][PC * e + b];
    T* out = &X[c][J][PF * e];
    out[0] = v[0];
#pragma unroll
    for (int a = 1; a < PF; ++a) {
      T s = T(0);
#pragma unroll
      for (int b = 0; b <= PC; ++b) s += I1.w[a * (PC + 1) + b] * v[b];
      out[a] = s;
    }
    if (e == nex - 1) out[PF] = v[PC];
  }
  __syncthreads();
  // fine nodes owned by the tile: the last one of the grid closes it
  const bool top = ez == mf.nz - 1;
  auto column = [&](int i, int e, auto with_mask) {
    const bool close = ey0 + e == mf.ny - 1;
    T in[PC + 1][PC + 1];
#pragma unroll
    for (int c = 0; c <= PC; ++c)
#pragma unroll
      for (int b = 0; b <= PC; ++b) in[c][b] = X[c][PC * e + b][i];
    const long long n0 = f * mf.nn + PF * ex0 + i + (long long)mf.nnx * PF * (ey0 + e) + (long long)plane * PF * ez;
#pragma unroll
    for (int a = 0; a <= PF; ++a) {
      if (a == PF && !close) break;
      T v[PC + 1];
#pragma unroll
      for (int c = 0; c <= PC; ++c) {
        v[c] = a == 0 ? in[c][0] : a == PF ? in[c][PC] : T(0);
        if (a > 0 && a < PF)
#pragma unroll
          for (int b = 0; b <= PC; ++b) v[c] += I1.w[a * (PC + 1) + b] * in[c][b];
      }
      T* out = xf + n0 + mf.nnx * a;
      const uint8_t* m = maskf + n0 + mf.nnx * a;
#pragma unroll
      for (int k = 0; k <= PF; ++k) {
        if (k == PF && !top) break;
        T s = k == 0 ? v[0] : k == PF ? v[PC] : T(0);
        if (k > 0 && k < PF)
#pragma unroll
          for (int c = 0; c <= PC; ++c) s += I1.w[k * (PC + 1) + c] * v[c];
        if (decltype(with_mask)::value && m[plane * k]) s = T(0);
        out[plane * k] = ADD ? out[plane * k] + s : s;
      }
    }
  };
  auto columns = [&](auto with_mask) {
    for (int idx = t; idx < PF * TX * TY; idx += kXferThreads) {
      const int i = idx % (PF * TX), e = idx / (PF * TX);
      if (i < PF * nex && e < ney) column(i, e, with_mask);
    }
    if (ex0 + nex == mf.nx && t < ney) column(PF * nex, t, with_mask);
  };
  if (masked) columns(std::true_type());
  else columns(std::false_type());
  }
}

// Restriction onto the coarse nodes of element slots [s0, s0 + ns) per
// direction: slot s holds the vertex PC s and the PC - 1 nodes inside element s;
// the last slot of a direction is the closing vertex.  Stage z: every thread
// takes fine columns of the tile and its halo and contracts the 2 PF - 1 fine
// nodes around the layer's vertex; then y and x in shared memory.
template <typename T, int PF, int PC, bool MINUS>
__global__ void __launch_bounds__(kXferThreads)
k_restrict(MeshDev mc, MeshDev mf, const XferW<T, PF, PC> I1, const T* __restrict__ rf, const T* __restrict__ b,
           T* __restrict__ rc, const uint8_t* __restrict__ maskc, const uint8_t* __restrict__ maskf,
           const uint8_t* __restrict__ emask) {
  constexpr int TX = tile_x<T, PF>(), TY = kTileYr;
  constexpr int FX = PF * (TX + 1) + PF - 1, FY = PF * (TY + 1) + PF - 1;
  __shared__ T Z[PC][FY][FX];
  __shared__ T Y[PC][PC * (TY + 1)][FX];
  const int t = threadIdx.x, plane = mf.nnx * mf.nny;
  for (int zf = blockIdx.z; zf < 4 * (mf.nz + 1); zf += gridDim.z)
  for (int sy0 = blockIdx.y * TY; sy0 < mf.ny; sy0 += gridDim.y * TY) {
  const int sz = zf >> 2, f = zf & 3, sx0 = blockIdx.x * TX;
  __syncthreads();  // a former tile's values are read
  const int nsx = sx0 + TX >= mf.nx ? mf.nx + 1 - sx0 : TX, nsy = sy0 + TY >= mf.ny ? mf.ny + 1 - sy0 : TY;
  const int fw = PF * nsx + PF - 1, fh = PF * nsy + PF - 1;
  const int i0 = PF * sx0 - (PF - 1), j0 = PF * sy0 - (PF - 1), k0 = PF * sz - (PF - 1), nnzf = PF * mf.nz + 1;
  const bool masked = maskf && any_masked(mf, emask, sx0 - 1, sx0 + TX, sy0 - 1, sy0 + TY, sz - 1, sz + 1);
  const bool inner = k0 >= 0 && k0 + 2 * PF - 2 < nnzf;
  auto vertex = [&](const T* v, int st) {  // weights of a vertex: its own node and both elements' interiors
    T s = v[(PF - 1) * st];
#pragma unroll
    for (int a = 1; a < PF; ++a) s += I1.w[a * (PC + 1) + PC] * v[(a - 1) * st] + I1.w[a * (PC + 1)] * v[(PF - 1 + a) * st];
    return s;
  };
  auto interior = [&](const T* v, int st, int q) {
    T s = T(0);
#pragma unroll
    for (int a = 1; a < PF; ++a) s += I1.w[a * (PC + 1) + q] * v[(PF - 1 + a) * st];
    return s;
  };
  auto column = [&](int i, int j, auto with_mask) {
    const int I = i0 + i, J = j0 + j;
    T v[2 * PF - 1];
#pragma unroll
    for (int k = 0; k < 2 * PF - 1; ++k) v[k] = T(0);
    if (I >= 0 && J >= 0 && I < mf.nnx && J < mf.nny) {
      const long long n0 = f * mf.nn + I + (long long)mf.nnx * J + (long long)plane * k0;
      const T *in = rf + n0, *bn = MINUS ? b + n0 : nullptr;
      auto at = [&](int k) {
        const int o = plane * k;
        if (decltype(with_mask)::value && maskf[n0 + o]) return T(0);
        return MINUS ? bn[o] - in[o] : in[o];
      };
      if (inner) {
#pragma unroll
        for (int k = 0; k < 2 * PF - 1; ++k) v[k] = at(k);
      } else {
#pragma unroll
        for (int k = 0; k < 2 * PF - 1; ++k)
          if (k0 + k >= 0 && k0 + k < nnzf) v[k] = at(k);
      }
    }
    Z[0][j][i] = vertex(v, 1);
#pragma unroll
    for (int c = 1; c < PC; ++c) Z[c][j][i] = interior(v, 1, c);
  };
  // (two widths known at compile time, so that no index needs a division)
  auto columns = [&](auto with_mask) {
    constexpr int GX = FX - PF, GY = FY - PF;
    if (nsx > TX || nsy > TY) {
      for (int idx = t; idx < FY * FX; idx += kXferThreads)
        if (idx % FX < fw && idx / FX < fh) column(idx % FX, idx / FX, with_mask);
    } else {
      for (int idx = t; idx < GY * GX; idx += kXferThreads)
        if (idx % GX < fw && idx / GX < fh) column(idx % GX, idx / GX, with_mask);
    }
  };
  if (masked) columns(std::true_type());
  else columns(std::false_type());
  __syncthreads();
  for (int idx = t; idx < PC * (TY + 1) * FX; idx += kXferThreads) {
    const int i = idx % FX, r = idx / FX, sl = r % (TY + 1), c = r / (TY + 1);
    if (i >= fw || sl >= nsy) continue;
    const T* in = &Z[c][PF * sl][i];
    Y[c][PC * sl][i] = vertex(in, FX);
#pragma unroll
    for (int q = 1; q < PC; ++q) Y[c][PC * sl + q][i] = interior(in, FX, q);
  }
  __syncthreads();
  // coarse nodes of the block: PC per slot, one for the closing vertex
  constexpr int CX = PC * (TX + 1), CY = PC * (TY + 1);
  const int cw = PC * nsx - (sx0 + nsx > mf.nx ? PC - 1 : 0), ch = PC * nsy - (sy0 + nsy > mf.ny ? PC - 1 : 0);
  const int cd = sz == mf.nz ? 1 : PC;
  for (int idx = t; idx < PC * CY * CX; idx += kXferThreads) {
    const int I = idx % CX, r = idx / CX, J = r % CY, c = r / CY;
    if (I >= cw || J >= ch || c >= cd) continue;
    const int sl = I / PC, q = I % PC;
    const T* in = &Y[c][J][PF * sl];
    T s = T(0);
    if (q == 0) {
      s = vertex(in, 1);
    } else {
#pragma unroll
      for (int qq = 1; qq < PC; ++qq)
        if (qq == q) s = interior(in, 1, qq);
    }
    const long long n = f * mc.nn + PC * sx0 + I + (long long)mc.nnx * (PC * sy0 + J + (long long)mc.nny * (PC * sz + c));
    if (maskc && maskc[n]) s = T(0);
    rc[n] = s;
  }
  }
}

// Blocks per tile direction (x unlimited; y and z walk their remainder).
template <int TX, int TY> dim3 xfer_grid(const MeshDev& m, int layers) {
  return dim3((m.nx + TX - 1) / TX, std::min((m.ny + TY - 1) / TY, 65535), std::min(4LL * layers, 65535LL));
}

template <typename T, int PF, int PC>
cudaError_t prolong_pq(const MeshDev& mc, const MeshDev& mf, const double* I1, const T* xc, T* xf,
                       const uint8_t* maskc, const uint8_t* maskf, const uint8_t* emask, int add, cudaStream_t st) {
  XferW<T, PF, PC> w;
  for (int k = 0; k < (PF + 1) * (PC + 1); ++k) w.w[k] = (T)I1[k];
  const dim3 grid = xfer_grid<tile_x<T, PF>(), tile_yp<T>()>(mf, mf.nz);
  if (add) k_prolong<T, PF, PC, true><<<grid, kXferThreads, 0, st>>>(mc, mf, w, xc, xf, maskc, maskf, emask);
  else k_prolong<T, PF, PC, false><<<grid, kXferThreads, 0, st>>>(mc, mf, w, xc, xf, maskc, maskf, emask);
  note_launch();
  return cudaGetLastError();
}
template <typename T, int PF, int PC>
cudaError_t restrict_pq(const MeshDev& mc, const MeshDev& mf, const double* I1, const T* rf, const T* b, T* rc,
                        const uint8_t* maskc, const uint8_t* maskf, const uint8_t* emaskf, cudaStream_t st) {
  XferW<T, PF, PC> w;
  for (int k = 0; k < (PF + 1) * (PC + 1); ++k) w.w[k] = (T)I1[k];
  const dim3 grid = xfer_grid<tile_x<T, PF>(), kTileYr>(mf, mf.nz + 1);
  if (b) k_restrict<T, PF, PC, true><<<grid, kXferThreads, 0, st>>>(mc, mf, w, rf, b, rc, maskc, maskf, emaskf);
  else k_restrict<T, PF, PC, false><<<grid, kXferThreads, 0, st>>>(mc, mf, w, rf, b, rc, maskc, maskf, emaskf);
  note_launch();
  return cudaGetLastError();
}

}  // namespace

// I1: host table [p_f + 1][p_c + 1] of the coarse basis at the fine nodes.
template <typename T>
cudaError_t launch_prolong(const MeshDev& mc, const MeshDev& mf, const double* I1, const T* xc, T* xf,
                           const uint8_t* maskc, const uint8_t* maskf, const uint8_t* emaskf, int add,
                           cudaStream_t st) {
  if (mf.nel == 0) return cudaSuccess;
  switch (10 * mf.p + mc.p) {
    case 21: return prolong_pq<T, 2, 1>(mc, mf, I1, xc, xf, maskc, maskf, emaskf, add, st);
    case 31: return prolong_pq<T, 3, 1>(mc, mf, I1, xc, xf, maskc, maskf, emaskf, add, st);
    case 32: return prolong_pq<T, 3, 2>(mc, mf, I1, xc, xf, maskc, maskf, emaskf, add, st);
    case 41: return prolong_pq<T, 4, 1>(mc, mf, I1, xc, xf, maskc, maskf, emaskf, add, st);
    case 42: return prolong_pq<T, 4, 2>(mc, mf, I1, xc, xf, maskc, maskf, emaskf, add, st);
    case 43: return prolong_pq<T, 4, 3>(mc, mf, I1, xc, xf, maskc, maskf, emaskf, add, st);
  }
  return cudaErrorInvalidValue;
}
template <typename T>
cudaError_t launch_restrict(const MeshDev& mc, const MeshDev& mf, const double* I1, const T* rf, const T* b, T* rc,
                            const uint8_t* maskc, const uint8_t* maskf, const uint8_t* emaskf, cudaStream_t st) {
  if (mf.nel == 0) return cudaSuccess;
  switch (10 * mf.p + mc.p) {
    case 21: return restrict_pq<T, 2, 1>(mc, mf, I1, rf, b, rc, maskc, maskf, emaskf, st);
    case 31: return restrict_pq<T, 3, 1>(mc, mf, I1, rf, b, rc, maskc, maskf, emaskf, st);
    case 32: return restrict_pq<T, 3, 2>(mc, mf, I1, rf, b, rc, maskc, maskf, emaskf, st);
    case 41: return restrict_pq<T, 4, 1>(mc, mf, I1, rf, b, rc, maskc, maskf, emaskf, st);
    case 42: return restrict_pq<T, 4, 2>(mc, mf, I1, rf, b, rc, maskc, maskf, emaskf, st);
    case 43: return restrict_pq<T, 4, 3>(mc, mf, I1, rf, b, rc, maskc, maskf, emaskf, st);
  }
  return cudaErrorInvalidValue;
}
#define PFF_TRANSFER(T)                                                                                            \
  template cudaError_t launch_prolong<T>(const MeshDev&, const MeshDev&, const double*, const T*, T*,              \
                                         const uint8_t*, const uint8_t*, const uint8_t*, int, cudaStream_t);       \
  template cudaError_t launch_restrict<T>(const MeshDev&, const MeshDev&, const double*, const T*, const T*, T*,   \
                                          const uint8_t*, const uint8_t*, const uint8_t*, cudaStream_t);
PFF_TRANSFER(double)
PFF_TRANSFER(float)

}  // namespace pff
