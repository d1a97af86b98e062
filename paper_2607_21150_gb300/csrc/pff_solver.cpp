// Newton-Krylov solver with p-multigrid preconditioning (Sec. 5: Newton,
// GMRES with adaptive classical Gram-Schmidt refinement, p-multigrid with
// Chebyshev smoothing), host-driven, every vector operation a device kernel.
//
// * Outer: Newton on the FP64 residual with a backtracking line search; each
//   linear solve is FGMRES(m) with FP64 vectors and inner products, its
//   operator the FP64 fine action (outer_prec), right-
//   preconditioned by one V-cycle (flexible because the coarse solve and the
//   mixed-precision cycle are not exactly linear in FP64).
// * V-cycle: Chebyshev(k) pre- and post-smoothing on D^-1 J of every
//   matrix-free level (FP64, or FP32 in the mixed variant), p-restriction /
//   prolongation between levels, and on an order-1 coarsest level an FP64
//   solve with the assembled Q1 Galerkin operator: Chebyshev-Jacobi,
//   Jacobi-GMRES, or GMRES preconditioned by a geometric h-multigrid V-cycle
//   on the structured Q1 grid (the paper's algebraic coarse solver replaced
//   by geometric coarsening, which the structured box allows).
// * Eigenvalue bounds: lambda_max of D^-1 J per level (and per h-level) as the
//   spectral radius of the Hessenberg matrix of a few Arnoldi steps from a
//   seeded random-sign vector, re-estimated every eig_every Newton iterations
//   (0: only on the first); smoothing interval [lo, hi] * lambda_max.
#include <algorithm>
#include <atomic>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "pff_handles.h"

using namespace pff;

namespace {

int sfail(int code, const std::string& msg) { return set_last_error(code, msg.c_str()); }

#define S_CK(call)                                                                                   \
  do {                                                                                              \
    cudaError_t e_ = (call);                                                                        \
    if (e_ != cudaSuccess) return sfail(PFF_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)
#define S_RC(call)            \
  do {                        \
    int r_ = (call);          \
    if (r_ != PFF_OK) return r_; \
  } while (0)

struct LevelWork {
  pff_level* L = nullptr;
  int p = 0;
  int prec = PFF_F64;
  size_t esz = 8;
  long long n = 0;
  void *diag = nullptr, *b = nullptr, *x = nullptr, *tmp = nullptr, *work = nullptr;
  double lmax = 1.0;
};

// One level of the geometric h-hierarchy below the assembled Q1 level (level 0
// aliases the Q1 level's operator, diagonal, element matrices and mask).
struct HLevel {
  MeshDev mesh;
  long long n = 0;
  double *Ke = nullptr, *A = nullptr, *dinv = nullptr;  // dinv: reciprocal diagonal
  float* A32 = nullptr;  // mixed solver: FP32 copy of A for the preconditioner's products
  const uint8_t* mask = nullptr;
  uint8_t* own_mask = nullptr;
  double *b = nullptr, *x = nullptr, *r = nullptr, *work = nullptr;
  double lmax = 1.0;
  bool owns = false;
};

// Page-locked sets of dot scalars: six of the Krylov solves; the Arnoldi process
// (not nested in one) uses two per step, up to 60 steps.
constexpr int kHostSlots = 128;

double now() {
  return std::chrono::duration<double>(std::chrono::steady_clock::now().time_since_epoch()).count();
}

}  // namespace

struct pff_solver {
  pff_op* op = nullptr;
  pff_solver_params prm;
  std::vector<LevelWork> lv;
  bool assembled = false;
  double *A = nullptr, *cdinv = nullptr, *cb = nullptr, *cx = nullptr, *cwork = nullptr;
  float* A32 = nullptr;                 // mixed solver: FP32 copy of the coarse stencil
  double *cV = nullptr, *cZ = nullptr;  // coarse GMRES basis
  double* Ke = nullptr;                 // coarse element matrices [nel][32][32]
  std::vector<HLevel> hl;               // geometric h-hierarchy (coarse_solver 2)
  long long coarse_iters = 0;
  double clmax = 1.0;
  long long n = 0;
  double *V = nullptr, *Z = nullptr, *r = nullptr, *dz = nullptr, *zold = nullptr;
  double* partial = nullptr;       // block shares of the dot products
  unsigned* arrived = nullptr;     // blocks of a dot-product launch that have finished
  DotScalars* sc = nullptr;        // six sets of dot scalars: outer Krylov (and Arnoldi), coarse Krylov
  DotScalars *host = nullptr, *host_dev = nullptr;  // page-locked copies and their device address
  unsigned long long seq = 0;
  double* pw64 = nullptr;  // power-iteration start vector (FP64, fine size)
  int transpose = 0;       // 1 while solving with J^T (adjoint)
  // adjoint work space (allocated on the first pff_adjoint_step)
  double *a_in = nullptr, *pbuf = nullptr, *qa = nullptr, *ag = nullptr, *alam = nullptr, *av = nullptr, *gth = nullptr;
};

namespace {

// Dot products out->dot[j] = V_j . w, j < k, with their host copy in slot
// `slot` under a new sequence number (returned in *seq).
int dots(pff_solver* s, const double* V, long long ldv, int k, const double* w, long long n, int gs,
         const DotScalars* gate, DotScalars* out, int slot, unsigned long long* seq, cudaStream_t st) {
  *seq = ++s->seq;
  S_CK((launch_mdot<double, double>(V, ldv, k, w, n, s->partial, s->arrived, gs, gate, out, s->host_dev + slot, *seq, st)));
  return PFF_OK;
}

// Waits for the host copy of a set of dot products: polls the sequence number
// that the kernel writes last, so that the work queued behind the products keeps
// running; the stream is queried now and then, which also ends the wait on an
// error.
int wait_dots(pff_solver* s, int slot, unsigned long long seq, cudaStream_t st) {
  const volatile DotScalars* h = s->host + slot;
  for (unsigned it = 1; h->seq != seq; ++it) {
    if (it % 2048) continue;
    const cudaError_t e = cudaStreamQuery(st);
    if (e == cudaErrorNotReady) continue;
    if (e != cudaSuccess) return sfail(PFF_ERR_CUDA, std::string("dot products: ") + cudaGetErrorString(e));
    if (h->seq != seq) return sfail(PFF_ERR_CUDA, "dot products: no result");
  }
  std::atomic_thread_fence(std::memory_order_acquire);
  return PFF_OK;
}

// ||v||^2 on the host.
int dev_norm2(pff_solver* s, const double* v, long long n, double* out, cudaStream_t st) {
  unsigned long long seq;
  S_RC(dots(s, v, 0, 1, v, n, 0, nullptr, s->sc, 0, &seq, st));
  S_RC(wait_dots(s, 0, seq, st));
  *out = s->host[0].dot[0];
  return PFF_OK;
}

int coarse_gmres(pff_solver* s, cudaStream_t st);

// The assembled coarse level in the form of an h-level.
HLevel coarse_level(pff_solver* s) {
  HLevel h;
  h.mesh = s->lv.back().L->mesh;
  h.n = s->lv.back().n;
  h.A = s->A;
  h.A32 = s->A32;
  h.dinv = s->cdinv;
  h.work = s->cwork;
  return h;
}

int level_apply(pff_solver* s, const LevelWork& w, const void* x, void* y, cudaStream_t st) {
  if (s->transpose) return pff_jacobian_transpose_apply(w.L, (pff_prec)w.prec, x, y, st);
  return pff_jacobian_apply(w.L, (pff_prec)w.prec, x, y, st);
}

// Chebyshev smoothing of J x = b or, in transposed mode, J^T x = b (same
// eigenvalue bounds: D^-1 J^T and D^-1 J have the same spectrum).
int cheb_level(pff_solver* s, LevelWork& w, bool from_zero, int degree, double lmin, double lmax, cudaStream_t st) {
  return smooth_level(w.L, w.prec, s->transpose != 0, from_zero, degree, lmin, lmax, w.diag, w.b, w.x, w.work, st);
}

// Stencil product of an assembled level with the update that consumes it: the
// FP64 stencil, or with the mixed solver its FP32 copy (the coarse level only
// preconditions; the transposed product of the adjoint stays FP64).
int h_stencil(pff_solver* s, const HLevel& h, int mode, StencilArgs a, cudaStream_t st) {
  const bool f32 = h.A32 && !s->transpose;
  a.mesh = h.mesh;
  a.A = f32 ? (const void*)h.A32 : (const void*)h.A;
  a.dinv = h.dinv;
  S_CK(launch_q1_stencil(mode, f32, s->transpose != 0, a, st));
  return PFF_OK;
}
int h_spmv(pff_solver* s, const HLevel& h, const double* x, double* y, cudaStream_t st) {
  StencilArgs a{};
  a.v = x;
  a.y = y;
  return h_stencil(s, h, kStProduct, a, st);
}

// Chebyshev-Jacobi smoothing (Saad, Alg. 12.1) of A x = b on an assembled
// level, degree - 1 products, each with its updates in one kernel.  from_zero:
// x = 0 on entry (its contents are not read) and h.work already holds
// r = D^-1 b and d = r / theta (launch_hrestrict or launch_jacobi).
int h_cheb(pff_solver* s, HLevel& h, const double* b, double* x, int degree, double lmin, double lmax, bool from_zero,
           cudaStream_t st) {
  const long long n = h.n;
  double *r = h.work, *d = h.work + n, *dn = h.work + 2 * n;
  const double theta = 0.5 * (lmax + lmin), delta = 0.5 * (lmax - lmin), sigma = theta / delta;
  double rho = 1.0 / sigma;
  StencilArgs a{};
  a.b = b;
  a.x = x;
  a.r = r;
  if (!from_zero) {
    a.v = x;
    a.y = d;
    a.cr = 1.0 / theta;
    S_RC(h_stencil(s, h, kStChebInit, a, st));
  }
  if (degree == 1) {
    if (from_zero) S_CK(cudaMemcpyAsync(x, d, sizeof(double) * n, cudaMemcpyDeviceToDevice, st));
    else S_CK(launch_axpby<double>(x, d, 1.0, 1.0, n, st));
  }
  for (int k = 0; k + 1 < degree; ++k) {
    const double rho_new = 1.0 / (2.0 * sigma - rho);
    a.v = d;
    a.y = dn;
    a.cd = rho_new * rho;
    a.cr = 2.0 * rho_new / delta;
    a.xset = from_zero && k == 0;
    a.last = k + 2 == degree;
    S_RC(h_stencil(s, h, kStChebStep, a, st));
    std::swap(d, dn);
    rho = rho_new;
  }
  return PFF_OK;
}

// Smoothing interval of h-level l: [lo, cheb_hi] lambda_max, with the coarsest
// grid's lower end; 1 / theta of it.
double h_inv_theta(const pff_solver* s, size_t l) {
  const double lo = l + 1 == s->hl.size() ? s->prm.coarse_lo : s->prm.cheb_lo;
  return 2.0 / (s->hl[l].lmax * (s->prm.cheb_hi + lo));
}

int coarse_cheb(pff_solver* s, cudaStream_t st) {
  if (s->prm.coarse_solver >= 1) return coarse_gmres(s, st);
  // FP64 Chebyshev-Jacobi on the assembled coarse operator, from x = 0.
  LevelWork& c = s->lv.back();
  const long long n = c.n;
  HLevel h = coarse_level(s);
  if (c.prec == PFF_F64) S_CK(cudaMemcpyAsync(s->cb, c.b, sizeof(double) * n, cudaMemcpyDeviceToDevice, st));
  else S_CK(launch_f2d(s->cb, (const float*)c.b, n, st));
  const double lmax = s->clmax * s->prm.cheb_hi, lmin = s->clmax * s->prm.coarse_lo;
  S_CK(launch_jacobi(n, s->cb, s->cdinv, h.work, h.work + n, 2.0 / (lmax + lmin), st));
  S_RC(h_cheb(s, h, s->cb, s->cx, s->prm.coarse_degree, lmin, lmax, true, st));
  if (c.prec == PFF_F64) S_CK(cudaMemcpyAsync(c.x, s->cx, sizeof(double) * n, cudaMemcpyDeviceToDevice, st));
  else S_CK(launch_d2f((float*)c.x, s->cx, n, st));
  return PFF_OK;
}

int vcycle(pff_solver* s, int l, cudaStream_t st) {
  LevelWork& w = s->lv[l];
  const bool coarsest = (l + 1 == (int)s->lv.size());
  if (coarsest && s->assembled) return coarse_cheb(s, st);
  const int deg = coarsest ? s->prm.coarse_degree : s->prm.cheb_degree;
  const double lo = coarsest ? s->prm.coarse_lo : s->prm.cheb_lo;
  S_RC(cheb_level(s, w, true, deg, lo * w.lmax, s->prm.cheb_hi * w.lmax, st));
  if (coarsest) return PFF_OK;
  // residual, restriction, coarse correction, prolongation
  S_RC(level_apply(s, w, w.x, w.tmp, st));
  LevelWork& c = s->lv[l + 1];
  S_RC(transfer_restrict(c.L, w.L, w.prec, w.tmp, w.b, c.b, st));
  S_RC(vcycle(s, l + 1, st));
  S_RC(transfer_prolong(c.L, w.L, w.prec, c.x, w.x, true, st));
  S_RC(cheb_level(s, w, false, s->prm.cheb_degree, s->prm.cheb_lo * w.lmax, s->prm.cheb_hi * w.lmax, st));
  return PFF_OK;
}

// ---- geometric h-multigrid on the assembled order-1 grid ------------------
// V-cycle on h-level l for A_l x = b (x from zero; h.work holds the first
// smoothing vectors, see h_cheb): Chebyshev pre- and post-smoothing, residual
// restriction by P^T, coarse correction, trilinear prolongation; the coarsest
// grid takes Chebyshev(coarse_degree).
int hcycle(pff_solver* s, int l, const double* b, double* x, cudaStream_t st) {
  HLevel& h = s->hl[l];
  const pff_solver_params& p = s->prm;
  if (l + 1 == (int)s->hl.size())
    return h_cheb(s, h, b, x, p.coarse_degree, p.coarse_lo * h.lmax, p.cheb_hi * h.lmax, true, st);
  S_RC(h_cheb(s, h, b, x, p.cheb_degree, p.cheb_lo * h.lmax, p.cheb_hi * h.lmax, true, st));
  StencilArgs a{};
  a.v = x;
  a.b = b;
  a.y = h.r;
  S_RC(h_stencil(s, h, kStResidual, a, st));
  HLevel& c = s->hl[l + 1];
  S_CK(launch_hrestrict(c.mesh, h.mesh, h.r, c.b, c.mask, h.mask, c.dinv, h_inv_theta(s, l + 1), c.work, c.work + c.n,
                        st));
  S_RC(hcycle(s, l + 1, c.b, c.x, st));
  S_CK(launch_hprolong_add(c.mesh, h.mesh, c.x, x, c.mask, h.mask, st));
  return h_cheb(s, h, b, x, p.cheb_degree, p.cheb_lo * h.lmax, p.cheb_hi * h.lmax, false, st);
}

// One V-cycle x = M_h^-1 b on h-level 0 (x and b distinct).
int hcycle_top(pff_solver* s, const double* b, double* x, cudaStream_t st) {
  HLevel& h = s->hl[0];
  S_CK(launch_jacobi(h.n, b, h.dinv, h.work, h.work + h.n, h_inv_theta(s, 0), st));
  return hcycle(s, 0, b, x, st);
}

// Spectral radius of a small dense matrix (row-major k x k) by power iteration
// on the host, with the growth rate averaged over the last iterations so that a
// dominant complex pair is measured too.
double small_spectral_radius(const std::vector<double>& H, int k) {
  std::vector<double> v(k, 1.0), y(k);
  for (int i = 0; i < k; ++i) v[i] = 1.0 + 0.01 * i;
  double logsum = 0.0;
  int counted = 0;
  for (int it = 0; it < 2000; ++it) {
    double nrm = 0.0;
    for (int i = 0; i < k; ++i) {
      double s = 0.0;
      for (int j = 0; j < k; ++j) s += H[i * k + j] * v[j];
      y[i] = s;
      nrm += s * s;
    }
    nrm = std::sqrt(nrm);
    if (!(nrm > 0.0) || !std::isfinite(nrm)) return 0.0;
    for (int i = 0; i < k; ++i) v[i] = y[i] / nrm;
    if (it >= 1000) { logsum += std::log(nrm); ++counted; }
  }
  return std::exp(logsum / counted);
}

// lambda_max of D^-1 A: k Arnoldi steps (Gram-Schmidt twice, FP64 basis in the
// FGMRES storage) from a seeded random-sign vector; the estimate is the spectral
// radius of the k x k Hessenberg block (the reading of the eigenvalue bound of
// a Chebyshev smoother: a few Arnoldi/Lanczos steps).  op(v, w) sets
// w = D^-1 A v on FP64 vectors of length n.
template <typename Op>
int arnoldi_lmax(pff_solver* s, long long n, Op&& op, double* out, cudaStream_t st) {
  // Nothing waits on the host between the steps: the second pass's kernels run
  // or return at once by the first pass's scalars on the device, and the
  // Hessenberg matrix is put together from the host copies at the end.
  const int k = std::min(s->prm.power_iters, s->prm.krylov_restart);
  double* V = s->V;  // (restart + 1) fine vectors >= (k + 1) level vectors
  unsigned long long seq = 0;
  std::vector<unsigned long long> seqs(2 * k + 1, 0);
  S_RC(dots(s, s->pw64, 0, 1, s->pw64, n, 0, nullptr, s->sc, 0, &seq, st));
  S_CK(launch_normalise(V, s->pw64, s->sc, n, st));
  for (int j = 0; j < k; ++j) {
    double* wv = V + (long long)(j + 1) * n;
    S_RC(op(V + (long long)j * n, wv));
    // classical Gram-Schmidt with the second pass only when the first removed
    // more than half of ||w||^2 (the criterion of the outer FGMRES); the dots
    // include w . w itself (wv is V_{j+1})
    for (int pass = 0; pass < 2; ++pass) {
      const DotScalars* gate = pass ? s->sc : nullptr;
      S_RC(dots(s, V, n, j + 2, wv, n, 1, gate, s->sc + pass, 1 + 2 * j + pass, &seqs[2 * j + pass], st));
      S_CK(launch_gs_update(wv, V, n, j + 1, s->sc + pass, gate, n, st));
    }
  }
  S_CK(cudaStreamSynchronize(st));
  std::vector<double> H((k + 1) * k, 0.0);
  int kk = k;
  for (int j = 0; j < k; ++j) {
    double ww2 = 0.0;
    for (int pass = 0; pass < 2; ++pass) {
      const DotScalars& h = s->host[1 + 2 * j + pass];
      if (h.seq != seqs[2 * j + pass]) break;  // no second pass
      for (int i = 0; i <= j; ++i) H[i * k + j] += h.dot[i];
      ww2 = h.ww2;
    }
    const double hn = std::sqrt(ww2);
    if (!std::isfinite(hn)) return sfail(PFF_ERR_DEVICE, "Arnoldi eigenvalue estimate: non-finite vector");
    H[(j + 1) * k + j] = hn;
    if (hn <= 1e-14 * std::fabs(H[j * k + j]) + 1e-300) { kk = j + 1; break; }
  }
  std::vector<double> Hk(kk * kk);
  for (int i = 0; i < kk; ++i)
    for (int j = 0; j < kk; ++j) Hk[i * kk + j] = H[i * k + j];
  const double lam = small_spectral_radius(Hk, kk);
  if (!(lam > 0.0) || !std::isfinite(lam)) return sfail(PFF_ERR_DEVICE, "Arnoldi eigenvalue estimate failed");
  *out = lam;
  return PFF_OK;
}

int arnoldi_level(pff_solver* s, LevelWork& w, cudaStream_t st) {
  const long long n = w.n;
  auto op = [&](const double* vj, double* wv) -> int {
    if (w.prec == PFF_F64) {
      S_RC(pff_jacobian_apply(w.L, PFF_F64, vj, wv, st));
      S_CK(launch_dscale<double>(wv, wv, (const double*)w.diag, n, st));
    } else {
      S_CK(launch_d2f((float*)w.x, vj, n, st));
      S_RC(pff_jacobian_apply(w.L, (pff_prec)w.prec, w.x, w.tmp, st));
      S_CK(launch_dscale<float>((float*)w.tmp, (const float*)w.tmp, (const float*)w.diag, n, st));
      S_CK(launch_f2d(wv, (const float*)w.tmp, n, st));
    }
    return PFF_OK;
  };
  return arnoldi_lmax(s, n, op, &w.lmax, st);
}

int arnoldi_hlevel(pff_solver* s, HLevel& h, cudaStream_t st) {
  auto op = [&](const double* vj, double* wv) -> int {
    StencilArgs a{};
    a.v = vj;
    a.y = wv;
    return h_stencil(s, h, kStScaled, a, st);
  };
  return arnoldi_lmax(s, h.n, op, &h.lmax, st);
}

int power_coarse(pff_solver* s, cudaStream_t st) {
  const HLevel lev = coarse_level(s);
  const long long n = lev.n;
  double* v = s->cx;
  double* y = s->cb;
  S_CK(cudaMemcpyAsync(v, s->pw64, sizeof(double) * n, cudaMemcpyDeviceToDevice, st));
  double h;
  S_RC(dev_norm2(s, v, n, &h, st));
  S_CK(launch_axpby<double>(v, v, 1.0 / std::sqrt(h), 0.0, n, st));
  double lam = 1.0;
  for (int it = 0; it < s->prm.power_iters; ++it) {
    StencilArgs a{};
    a.v = v;
    a.y = y;
    S_RC(h_stencil(s, lev, kStScaled, a, st));
    S_RC(dev_norm2(s, y, n, &h, st));
    lam = std::sqrt(h);
    if (!(lam > 0.0) || !std::isfinite(lam)) return sfail(PFF_ERR_DEVICE, "coarse power iteration failed");
    S_CK(launch_axpby<double>(v, y, 1.0 / lam, 0.0, n, st));
  }
  s->clmax = lam;
  return PFF_OK;
}

// Flexible GMRES(m), right preconditioned (Saad, Alg. 9.6), FP64; classical
// Gram-Schmidt with a second pass when the first one loses accuracy (the
// adaptive CGS refinement of Sec. 5).  V: (m+1) n, Z: m n device doubles.
// sc, slot: its three sets of dot scalars on the device and in host memory (an
// inner solve runs between an outer one's and must not share them).  late: the
// host learns ||b|| with the first Hessenberg column only, which saves an inner
// solve a wait per call; a zero b then costs one preconditioner and one product.
struct Krylov {
  long long n = 0;
  int m = 0;
  double *V = nullptr, *Z = nullptr;
  DotScalars* sc = nullptr;
  int slot = 0;
  bool late = false;
};

template <typename ApplyA, typename ApplyM>
int gmres_flex(pff_solver* s, const Krylov& kw, ApplyA&& applyA, ApplyM&& applyM, const double* b, double* x,
               double rtol, int maxit, int* iters, double* relres, cudaStream_t st) {
  const long long n = kw.n;
  const int m = kw.m;
  std::vector<double> H((m + 1) * m, 0.0), cs(m, 0.0), sn(m, 0.0), g(m + 1, 0.0);
  const DotScalars* host = s->host + kw.slot;
  double beta0 = -1.0, res = 0.0;
  int total = 0;
  bool first = true;
  while (true) {
    double* v0 = kw.V;
    if (!first) {
      S_RC(applyA(x, v0));
      S_CK(launch_bminus<double>(v0, b, n, st));
    }
    // ||r|| and v0 = r / ||r|| on the device
    const double* r0 = first ? b : v0;
    unsigned long long seq_b = 0;
    S_RC(dots(s, r0, 0, 1, r0, n, 0, nullptr, kw.sc, kw.slot, &seq_b, st));
    double beta = 0.0;
    bool known = false;
    auto read_beta = [&]() -> int {
      S_RC(wait_dots(s, kw.slot, seq_b, st));
      beta = std::sqrt(host[0].dot[0]);
      if (beta0 < 0) beta0 = beta;
      known = true;
      return PFF_OK;
    };
    if (!first || !kw.late || !(rtol < 1.0) || total >= maxit) {
      S_RC(read_beta());
      if (beta == 0.0 || beta0 == 0.0) { res = 0.0; break; }
      res = beta;
      if (beta <= rtol * beta0 || total >= maxit) break;
    }
    S_CK(launch_normalise(v0, r0, kw.sc, n, st));
    int jend = 0;
    bool ended = false;
    for (int j = 0; j < m && total < maxit; ++j) {
      double* vj = kw.V + (long long)j * n;
      double* zj = kw.Z + (long long)j * n;
      double* w = kw.V + (long long)(j + 1) * n;
      S_RC(applyM(vj, zj));
      S_RC(applyA(zj, w));
      if (!known) {
        S_RC(read_beta());
        if (beta <= rtol * beta0) { ended = true; break; }  // zero, or a square beyond FP64: x = 0
      }
      if (j == 0) {
        std::fill(g.begin(), g.end(), 0.0);
        g[0] = beta;
      }
      // ||w||^2 after the projection is ww - hsq; a second pass only when the
      // first one removed more than half of ||w||^2 (cancellation has cost
      // accuracy: Daniel-Gragg-Kaufman-Stewart criterion), otherwise the
      // estimate is accurate to a few rounding errors and no further
      // reduction is needed
      unsigned long long seq;
      S_RC(dots(s, kw.V, n, j + 2, w, n, 1, nullptr, kw.sc + 1, kw.slot + 1, &seq, st));
      S_CK(launch_gs_update(w, kw.V, n, j + 1, kw.sc + 1, nullptr, n, st));
      S_RC(wait_dots(s, kw.slot + 1, seq, st));
      for (int i = 0; i <= j; ++i) H[i * m + j] = host[1].dot[i];
      double ww2 = host[1].ww2;
      if (host[1].second) {
        S_RC(dots(s, kw.V, n, j + 2, w, n, 1, kw.sc + 1, kw.sc + 2, kw.slot + 2, &seq, st));
        S_CK(launch_gs_update(w, kw.V, n, j + 1, kw.sc + 2, kw.sc + 1, n, st));
        S_RC(wait_dots(s, kw.slot + 2, seq, st));
        for (int i = 0; i <= j; ++i) H[i * m + j] += host[2].dot[i];
        ww2 = host[2].ww2;
      }
      const double hn = std::sqrt(ww2);
      H[(j + 1) * m + j] = hn;
      for (int i = 0; i < j; ++i) {
        double a = H[i * m + j], c = H[(i + 1) * m + j];
        H[i * m + j] = cs[i] * a + sn[i] * c;
        H[(i + 1) * m + j] = -sn[i] * a + cs[i] * c;
      }
      double a = H[j * m + j], c = H[(j + 1) * m + j];
      double den = std::hypot(a, c);
      cs[j] = den > 0 ? a / den : 1.0;
      sn[j] = den > 0 ? c / den : 0.0;
      H[j * m + j] = den;
      H[(j + 1) * m + j] = 0.0;
      g[j + 1] = -sn[j] * g[j];
      g[j] = cs[j] * g[j];
      ++total;
      jend = j + 1;
      res = std::fabs(g[j + 1]);
      if (res <= rtol * beta0 || hn == 0.0) break;
    }
    if (ended) { res = beta; break; }
    LinCoef y;
    for (int i = jend - 1; i >= 0; --i) {
      double sum = g[i];
      for (int k = i + 1; k < jend; ++k) sum -= H[i * m + k] * y.c[k];
      y.c[i] = sum / H[i * m + i];
    }
    S_CK(launch_lincomb(x, kw.Z, n, jend, y, first ? 0 : 1, n, st));
    first = false;
    if (res <= rtol * beta0 || total >= maxit) break;
  }
  if (first) S_CK(cudaMemsetAsync(x, 0, sizeof(double) * n, st));  // zero right-hand side, or no iteration allowed
  *iters = total;
  *relres = beta0 > 0 ? res / beta0 : 0.0;
  return PFF_OK;
}

int precondition(pff_solver* s, const double* v, double* z, cudaStream_t st);

int fgmres(pff_solver* s, const double* b, double* x, double rtol, int maxit, int* iters, double* relres,
           cudaStream_t st) {
  pff_level* F = s->lv[0].L;
  Krylov kw;
  kw.n = s->n;
  kw.m = s->prm.krylov_restart;
  kw.V = s->V;
  kw.Z = s->Z;
  kw.sc = s->sc;
  kw.slot = 0;
  const pff_prec outer = (pff_prec)s->prm.outer_prec;
  auto A = [&](const double* in, double* out) {
    if (s->transpose) return pff_jacobian_transpose_apply(F, outer, in, out, st);
    return pff_jacobian_apply(F, outer, in, out, st);
  };
  auto M = [&](const double* in, double* out) { return precondition(s, in, out, st); };
  return gmres_flex(s, kw, A, M, b, x, rtol, maxit, iters, relres, st);
}

// z = M^-1 v on FP64 fine vectors: one V-cycle (FP32 levels in the mixed variant).
int precondition(pff_solver* s, const double* v, double* z, cudaStream_t st) {
  LevelWork& f = s->lv[0];
  const long long n = s->n;
  if (f.prec == PFF_F64) S_CK(cudaMemcpyAsync(f.b, v, sizeof(double) * n, cudaMemcpyDeviceToDevice, st));
  else S_CK(launch_d2f((float*)f.b, v, n, st));
  S_RC(vcycle(s, 0, st));
  if (f.prec == PFF_F64) S_CK(cudaMemcpyAsync(z, f.x, sizeof(double) * n, cudaMemcpyDeviceToDevice, st));
  else S_CK(launch_f2d(z, (const float*)f.x, n, st));
  return PFF_OK;
}

// Coarsest level: GMRES on the assembled FP64 operator to coarse_rtol (at most
// coarse_maxit iterations), from x = 0, preconditioned by Jacobi
// (coarse_solver 1) or by one h-multigrid V-cycle (coarse_solver 2).
int coarse_gmres(pff_solver* s, cudaStream_t st) {
  LevelWork& c = s->lv.back();
  const HLevel lev = coarse_level(s);
  const long long n = c.n;
  if (c.prec == PFF_F64) S_CK(cudaMemcpyAsync(s->cb, c.b, sizeof(double) * n, cudaMemcpyDeviceToDevice, st));
  else S_CK(launch_f2d(s->cb, (const float*)c.b, n, st));
  Krylov kw;
  kw.n = n;
  kw.m = s->prm.krylov_restart;
  kw.V = s->cV;
  kw.Z = s->cZ;
  kw.sc = s->sc + 3;
  kw.slot = 3;
  kw.late = true;
  auto A = [&](const double* in, double* out) -> int { return h_spmv(s, lev, in, out, st); };
  auto M = [&](const double* in, double* out) -> int {
    if (s->prm.coarse_solver == 2) return hcycle_top(s, in, out, st);
    S_CK(launch_jacobi(n, in, s->cdinv, nullptr, out, 1.0, st));
    return PFF_OK;
  };
  int its = 0;
  double rel = 0.0;
  S_RC(gmres_flex(s, kw, A, M, s->cb, s->cx, s->prm.coarse_rtol, s->prm.coarse_maxit, &its, &rel, st));
  s->coarse_iters += its;
  if (c.prec == PFF_F64) S_CK(cudaMemcpyAsync(c.x, s->cx, sizeof(double) * n, cudaMemcpyDeviceToDevice, st));
  else S_CK(launch_d2f((float*)c.x, s->cx, n, st));
  return PFF_OK;
}

// Diagonals, coarse operators and eigenvalue bounds for the current stored
// linearisation.  `eig` = false keeps the previous lambda_max estimates (the
// eig_every option of a Newton solve).
int setup(pff_solver* s, cudaStream_t st, bool eig = true) {
  const int L = (int)s->lv.size();
  for (int l = 0; l < L; ++l) {
    LevelWork& w = s->lv[l];
    if (l + 1 == L && s->assembled) continue;
    S_RC(pff_assemble_diagonal(w.L, (pff_prec)w.prec, w.diag, st));
  }
  if (s->assembled) {
    LevelWork& c = s->lv.back();
    pff_op* op = s->op;
    // the mixed solver assembles its (preconditioning) coarse level from the
    // FP32 words in FP32 arithmetic, the FP64 solver from the FP64 words
    S_CK(launch_q1_assemble_sf(c.L->mesh, op->Q, op->lin64, s->prm.mixed ? op->lin32 : nullptr, c.L->tab.B64,
                               c.L->tab.Dt64, c.L->mask, s->Ke, s->A,
                               op->geo != nullptr, st));
    S_CK(launch_q1_dinv(c.L->mesh, s->A, s->cdinv, st));
    if (s->A32) S_CK(launch_d2f(s->A32, s->A, 27LL * 16 * c.L->mesh.nn, st));
    if (s->prm.coarse_solver == 0 && eig) S_RC(power_coarse(s, st));
    if (s->prm.coarse_solver == 2) {
      for (size_t l = 1; l < s->hl.size(); ++l) {
        HLevel& f = s->hl[l - 1];
        HLevel& h = s->hl[l];
        S_CK(launch_hmask(f.mesh, h.mesh, f.mask, h.own_mask, st));
        S_CK(launch_q1_coarsen(f.mesh, h.mesh, f.mask, f.Ke, h.Ke, s->prm.mixed != 0, st));
        S_CK(launch_q1_gather(h.mesh, h.Ke, h.mask, h.A, st));
        S_CK(launch_q1_dinv(h.mesh, h.A, h.dinv, st));
        if (h.A32) S_CK(launch_d2f(h.A32, h.A, 27LL * 16 * h.mesh.nn, st));
      }
      if (eig)
        for (HLevel& h : s->hl) S_RC(arnoldi_hlevel(s, h, st));
    }
  }
  for (int l = 0; l < L && eig; ++l) {
    if (l + 1 == L && s->assembled) continue;
    S_RC(arnoldi_level(s, s->lv[l], st));
  }
  return PFF_OK;
}

void free_solver(pff_solver* s) {
  for (auto& w : s->lv) {
    cudaFree(w.diag); cudaFree(w.b); cudaFree(w.x); cudaFree(w.tmp); cudaFree(w.work);
  }
  cudaFree(s->A); cudaFree(s->A32); cudaFree(s->cdinv); cudaFree(s->cb); cudaFree(s->cx); cudaFree(s->cwork);
  cudaFree(s->cV); cudaFree(s->cZ); cudaFree(s->Ke);
  for (HLevel& h : s->hl) {
    if (h.owns) { cudaFree(h.Ke); cudaFree(h.A); cudaFree(h.A32); cudaFree(h.dinv); cudaFree(h.own_mask); }
    cudaFree(h.b); cudaFree(h.x); cudaFree(h.r); cudaFree(h.work);
  }
  cudaFree(s->V); cudaFree(s->Z); cudaFree(s->r); cudaFree(s->dz); cudaFree(s->zold);
  cudaFree(s->partial); cudaFree(s->arrived); cudaFree(s->sc); cudaFreeHost(s->host);
  cudaFree(s->pw64);
  cudaFree(s->a_in); cudaFree(s->pbuf); cudaFree(s->qa); cudaFree(s->ag); cudaFree(s->alam); cudaFree(s->av);
  cudaFree(s->gth);
}

}  // namespace

extern "C" {

int pff_solver_default_params(pff_solver_params* p) {
  if (!p) return sfail(PFF_ERR_INVALID, "pff_solver_default_params: null");
  p->mixed = 1;
  p->cheb_degree = 3;
  p->cheb_lo = 0.1;
  p->cheb_hi = 1.1;
  p->coarse_degree = 16;
  p->coarse_lo = 0.02;
  p->power_iters = 10;
  p->krylov_restart = 30;
  p->krylov_maxit = 200;
  p->krylov_rtol = 1e-3;
  p->newton_maxit = 20;
  p->newton_rtol = 1e-8;
  p->line_search_max = 8;
  p->coarse_solver = 2;
  p->coarse_rtol = 1e-2;
  p->coarse_maxit = 200;
  p->verbose = 0;
  p->outer_prec = PFF_F64;
  p->newton_stall = 0;
  p->eig_every = 1;
  p->level_words = 32;
  return PFF_OK;
}

int pff_create_solver(pff_op* op, int nlevels, pff_level* const* levels, const pff_solver_params* prm,
                      pff_solver** out) {
  if (!op || !levels || !prm || !out || nlevels < 1) return sfail(PFF_ERR_INVALID, "pff_create_solver: bad argument");
  if (prm->krylov_restart < 1 || prm->krylov_restart > 60) return sfail(PFF_ERR_INVALID, "pff_create_solver: 1 <= restart <= 60");
  if (prm->cheb_degree < 1 || prm->coarse_degree < 1) return sfail(PFF_ERR_INVALID, "pff_create_solver: degrees >= 1");
  if (!(prm->cheb_hi > prm->cheb_lo && prm->cheb_lo > 0 && prm->coarse_lo > 0 && prm->coarse_lo < prm->cheb_hi))
    return sfail(PFF_ERR_INVALID, "pff_create_solver: need 0 < lo < hi");
  if (levels[0]->op != op || !levels[0]->is_fine) return sfail(PFF_ERR_INVALID, "pff_create_solver: levels[0] must be the fine level of op");
  for (int l = 1; l < nlevels; ++l)
    if (levels[l]->op != op || levels[l]->p >= levels[l - 1]->p)
      return sfail(PFF_ERR_INVALID, "pff_create_solver: levels must share op with decreasing order");
  if (prm->mixed && !op->lin32) return sfail(PFF_ERR_INVALID, "pff_create_solver: mixed precision needs pff_op_enable_f32");
  if (prm->coarse_solver < 0 || prm->coarse_solver > 2)
    return sfail(PFF_ERR_INVALID, "pff_create_solver: coarse_solver must be 0, 1 or 2");
  if (prm->outer_prec != PFF_F64 && prm->outer_prec != PFF_DF64)
    return sfail(PFF_ERR_INVALID, "pff_create_solver: outer_prec must be PFF_F64 or PFF_DF64");
  if (prm->outer_prec == PFF_DF64 && !op->df)
    return sfail(PFF_ERR_INVALID, "pff_create_solver: outer_prec PFF_DF64 needs pff_op_enable_df");
  if (prm->level_words != 32 && prm->level_words != 16)
    return sfail(PFF_ERR_INVALID, "pff_create_solver: level_words must be 32 or 16");
  if (prm->mixed && prm->level_words == 16 && !(op->bf16 && op->lin16))
    return sfail(PFF_ERR_INVALID, "pff_create_solver: level_words 16 needs pff_op_enable_bf16");
  pff_solver* s = new pff_solver();
  s->op = op;
  s->prm = *prm;
  s->n = 4 * op->mesh.nn;
  s->assembled = (levels[nlevels - 1]->p == 1 && nlevels > 1);
  cudaError_t e = cudaSuccess;
  for (int l = 0; l < nlevels; ++l) {
    LevelWork w;
    w.L = levels[l];
    w.p = levels[l]->p;
    w.prec = prm->mixed ? (prm->level_words == 16 ? PFF_F32_BF16 : PFF_F32) : PFF_F64;
    w.esz = (w.prec == PFF_F64) ? 8 : 4;
    w.n = 4 * levels[l]->mesh.nn;
    if (e == cudaSuccess) e = cudaMalloc(&w.diag, w.esz * w.n);
    if (e == cudaSuccess) e = cudaMalloc(&w.b, w.esz * w.n);
    if (e == cudaSuccess) e = cudaMalloc(&w.x, w.esz * w.n);
    if (e == cudaSuccess) e = cudaMalloc(&w.tmp, w.esz * w.n);
    if (e == cudaSuccess) e = cudaMalloc(&w.work, 3 * w.esz * w.n);
    s->lv.push_back(w);
  }
  if (s->assembled) {
    const long long nc = s->lv.back().n;
    if (e == cudaSuccess) e = cudaMalloc(&s->A, sizeof(double) * 27 * 16 * (nc / 4));
    if (e == cudaSuccess && prm->mixed) e = cudaMalloc(&s->A32, sizeof(float) * 27 * 16 * (nc / 4));
    if (e == cudaSuccess) e = cudaMalloc(&s->cdinv, sizeof(double) * nc);
    if (e == cudaSuccess) e = cudaMalloc(&s->cb, sizeof(double) * nc);
    if (e == cudaSuccess) e = cudaMalloc(&s->cx, sizeof(double) * nc);
    if (e == cudaSuccess) e = cudaMalloc(&s->cwork, sizeof(double) * 3 * nc);
    if (e == cudaSuccess) e = cudaMalloc(&s->Ke, sizeof(double) * 1024 * (size_t)op->nel);
    if (e == cudaSuccess && prm->coarse_solver >= 1) e = cudaMalloc(&s->cV, sizeof(double) * (prm->krylov_restart + 1) * nc);
    if (e == cudaSuccess && prm->coarse_solver >= 1) e = cudaMalloc(&s->cZ, sizeof(double) * prm->krylov_restart * nc);
    if (prm->coarse_solver == 2) {
      // h-levels: the Q1 level, then full coarsening while every direction has
      // an even number of elements and keeps at least two
      pff_level* Lc = s->lv.back().L;
      HLevel h0;
      h0.mesh = Lc->mesh;
      h0.n = nc;
      h0.Ke = s->Ke;
      h0.A = s->A;
      h0.A32 = s->A32;
      h0.dinv = s->cdinv;
      h0.mask = Lc->is_fine ? op->mask : Lc->mask;
      s->hl.push_back(h0);
      while (true) {
        const MeshDev& mf = s->hl.back().mesh;
        if (mf.nx % 2 || mf.ny % 2 || mf.nz % 2 || mf.nx < 4 || mf.ny < 4 || mf.nz < 4) break;
        HLevel h;
        h.mesh = mf;
        h.mesh.nx = mf.nx / 2; h.mesh.ny = mf.ny / 2; h.mesh.nz = mf.nz / 2;
        h.mesh.nel = h.mesh.nx * h.mesh.ny * h.mesh.nz;
        h.mesh.nnx = h.mesh.nx + 1; h.mesh.nny = h.mesh.ny + 1;
        h.mesh.nn = (long long)h.mesh.nnx * h.mesh.nny * (h.mesh.nz + 1);
        h.mesh.offsets = nullptr;
        h.n = 4 * h.mesh.nn;
        h.owns = true;
        if (e == cudaSuccess) e = cudaMalloc(&h.Ke, sizeof(double) * 1024 * (size_t)h.mesh.nel);
        if (e == cudaSuccess) e = cudaMalloc(&h.A, sizeof(double) * 27 * 16 * (size_t)h.mesh.nn);
        if (e == cudaSuccess && prm->mixed) e = cudaMalloc(&h.A32, sizeof(float) * 27 * 16 * (size_t)h.mesh.nn);
        if (e == cudaSuccess) e = cudaMalloc(&h.dinv, sizeof(double) * h.n);
        if (e == cudaSuccess) e = cudaMalloc(&h.own_mask, h.n);
        h.mask = h.own_mask;
        s->hl.push_back(h);
        if (e != cudaSuccess) break;
      }
      for (HLevel& h : s->hl) {
        if (e == cudaSuccess) e = cudaMalloc(&h.b, sizeof(double) * h.n);
        if (e == cudaSuccess) e = cudaMalloc(&h.x, sizeof(double) * h.n);
        if (e == cudaSuccess) e = cudaMalloc(&h.r, sizeof(double) * h.n);
        if (e == cudaSuccess) e = cudaMalloc(&h.work, sizeof(double) * 3 * h.n);
      }
    }
  }
  const int m = prm->krylov_restart;
  if (e == cudaSuccess) e = cudaMalloc(&s->V, sizeof(double) * (m + 1) * s->n);
  if (e == cudaSuccess) e = cudaMalloc(&s->Z, sizeof(double) * m * s->n);
  if (e == cudaSuccess) e = cudaMalloc(&s->r, sizeof(double) * s->n);
  if (e == cudaSuccess) e = cudaMalloc(&s->dz, sizeof(double) * s->n);
  if (e == cudaSuccess) e = cudaMalloc(&s->zold, sizeof(double) * s->n);
  if (e == cudaSuccess) e = cudaMalloc(&s->partial, sizeof(double) * 64 * kReduceBlocks);
  if (e == cudaSuccess) e = cudaMalloc(&s->arrived, sizeof(unsigned));
  if (e == cudaSuccess) e = cudaMemset(s->arrived, 0, sizeof(unsigned));
  if (e == cudaSuccess) e = cudaMalloc(&s->sc, sizeof(DotScalars) * 6);
  if (e == cudaSuccess) e = cudaHostAlloc((void**)&s->host, sizeof(DotScalars) * kHostSlots, cudaHostAllocMapped);
  if (e == cudaSuccess) std::memset(s->host, 0, sizeof(DotScalars) * kHostSlots);
  if (e == cudaSuccess) e = cudaHostGetDevicePointer((void**)&s->host_dev, s->host, 0);
  if (e == cudaSuccess) e = cudaMalloc(&s->pw64, sizeof(double) * s->n);
  if (e == cudaSuccess) {
    // seeded start vector of the eigenvalue estimates (xorshift64*, random signs)
    std::vector<double> h(s->n);
    unsigned long long st = 0x9E3779B97F4A7C15ull;
    for (long long i = 0; i < s->n; ++i) {
      st ^= st >> 12; st ^= st << 25; st ^= st >> 27;
      double u = (double)((st * 0x2545F4914F6CDD1Dull) >> 11) * (1.0 / 9007199254740992.0);
      h[i] = (u < 0.5) ? -1.0 : 1.0;
    }
    e = cudaMemcpy(s->pw64, h.data(), sizeof(double) * s->n, cudaMemcpyHostToDevice);
  }
  if (e != cudaSuccess) {
    free_solver(s);
    delete s;
    return sfail(PFF_ERR_CUDA, std::string("pff_create_solver: ") + cudaGetErrorString(e));
  }
  *out = s;
  return PFF_OK;
}

int pff_vec_axpby(pff_prec prec, int64_t n, double a, const void* x, double b, void* y, void* stream) {
  if (!x || !y || n < 0) return sfail(PFF_ERR_INVALID, "pff_vec_axpby: bad argument");
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (prec == PFF_F64) S_CK(launch_axpby<double>((double*)y, (const double*)x, a, b, n, st));
  else if (prec == PFF_F32) S_CK(launch_axpby<float>((float*)y, (const float*)x, a, b, n, st));
  else return sfail(PFF_ERR_INVALID, "pff_vec_axpby: unknown precision");
  return PFF_OK;
}

int pff_destroy_solver(pff_solver* s) {
  if (!s) return PFF_OK;
  free_solver(s);
  delete s;
  return PFF_OK;
}

int pff_solver_setup(pff_solver* s, void* stream) {
  if (!s) return sfail(PFF_ERR_INVALID, "pff_solver_setup: null solver");
  return setup(s, reinterpret_cast<cudaStream_t>(stream));
}

int pff_solver_level_lambda(const pff_solver* s, int level, double* lmax) {
  if (!s || !lmax || level < 0 || level >= (int)s->lv.size()) return sfail(PFF_ERR_INVALID, "pff_solver_level_lambda: bad argument");
  *lmax = (level + 1 == (int)s->lv.size() && s->assembled) ? s->clmax : s->lv[level].lmax;
  return PFF_OK;
}

int pff_solver_vcycle(pff_solver* s, const double* r, double* z, void* stream) {
  if (!s || !r || !z) return sfail(PFF_ERR_INVALID, "pff_solver_vcycle: null argument");
  return precondition(s, r, z, reinterpret_cast<cudaStream_t>(stream));
}

int pff_solver_coarse_apply(pff_solver* s, const double* x, double* y, void* stream) {
  if (!s || !x || !y || !s->assembled) return sfail(PFF_ERR_INVALID, "pff_solver_coarse_apply: needs an assembled coarse level");
  StencilArgs a{};
  a.mesh = s->lv.back().L->mesh;
  a.A = s->A;
  a.v = x;
  a.y = y;
  S_CK(launch_q1_stencil(kStProduct, false, false, a, reinterpret_cast<cudaStream_t>(stream)));
  return PFF_OK;
}

int pff_solver_num_hlevels(const pff_solver* s) { return s ? (int)s->hl.size() : 0; }

int pff_solver_hlevel_info(const pff_solver* s, int level, int* dims, double* lmax) {
  if (!s || !dims || !lmax || level < 0 || level >= (int)s->hl.size())
    return sfail(PFF_ERR_INVALID, "pff_solver_hlevel_info: bad argument");
  const HLevel& h = s->hl[level];
  dims[0] = h.mesh.nx; dims[1] = h.mesh.ny; dims[2] = h.mesh.nz;
  *lmax = h.lmax;
  return PFF_OK;
}

int pff_solver_hlevel_apply(pff_solver* s, int level, const double* x, double* y, void* stream) {
  if (!s || !x || !y || level < 0 || level >= (int)s->hl.size())
    return sfail(PFF_ERR_INVALID, "pff_solver_hlevel_apply: bad argument");
  StencilArgs a{};
  a.mesh = s->hl[level].mesh;
  a.A = s->hl[level].A;
  a.v = x;
  a.y = y;
  S_CK(launch_q1_stencil(kStProduct, false, false, a, reinterpret_cast<cudaStream_t>(stream)));
  return PFF_OK;
}

int pff_solver_hcycle(pff_solver* s, const double* b, double* x, void* stream) {
  if (!s || !b || !x || s->hl.empty()) return sfail(PFF_ERR_INVALID, "pff_solver_hcycle: needs coarse_solver 2");
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  HLevel& h0 = s->hl[0];
  S_CK(cudaMemcpyAsync(h0.b, b, sizeof(double) * h0.n, cudaMemcpyDeviceToDevice, st));
  S_RC(hcycle_top(s, h0.b, h0.x, st));
  S_CK(cudaMemcpyAsync(x, h0.x, sizeof(double) * h0.n, cudaMemcpyDeviceToDevice, st));
  return PFF_OK;
}

int pff_solver_krylov(pff_solver* s, const double* b, double* x, double rtol, int maxit, int* iters, double* relres,
                      void* stream) {
  if (!s || !b || !x || !iters || !relres) return sfail(PFF_ERR_INVALID, "pff_solver_krylov: null argument");
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  S_RC(fgmres(s, b, x, rtol, maxit, iters, relres, st));
  S_CK(cudaStreamSynchronize(st));
  return PFF_OK;
}

int pff_newton_solve(pff_solver* s, double* z, pff_newton_stats* stats, void* stream) {
  if (!s || !z || !stats) return sfail(PFF_ERR_INVALID, "pff_newton_solve: null argument");
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  std::memset(stats, 0, sizeof(*stats));
  s->coarse_iters = 0;
  const long long n = s->n;
  double r0 = -1.0;
  for (int it = 0;; ++it) {
    double t0 = now();
    if (it == 0 || s->prm.line_search_max == 0) {
      S_RC(pff_residual(s->op, z, s->r, st));
      int status = 0;
      S_RC(pff_get_status(s->op, stream, &status));
      if (status) {
        stats->status = status;
        return sfail(PFF_ERR_DEVICE, "pff_newton_solve: residual kernel status " + std::to_string(status));
      }
    }
    double rr;
    S_RC(dev_norm2(s, s->r, n, &rr, st));
    double rn = std::sqrt(rr);
    stats->t_residual += now() - t0;
    if (r0 < 0) r0 = rn;
    if (it < 64) stats->res_history[it] = rn;
    stats->res0 = r0;
    stats->res = rn;
    if (rn <= s->prm.newton_rtol * r0 || rn == 0.0) { stats->converged = 1; break; }
    if (it >= s->prm.newton_maxit) break;
    const int k = s->prm.newton_stall;
    if (k > 0 && it >= k && it - k < 64 && rn > 0.5 * stats->res_history[it - k]) break;  // stagnation
    t0 = now();
    const int ev = s->prm.eig_every;
    S_RC(setup(s, st, ev > 0 ? (it % ev == 0) : (it == 0)));
    S_CK(cudaStreamSynchronize(st));
    stats->t_setup += now() - t0;
    t0 = now();
    int its = 0;
    double rel = 0.0;
    S_RC(fgmres(s, s->r, s->dz, s->prm.krylov_rtol, s->prm.krylov_maxit, &its, &rel, st));
    S_CK(cudaStreamSynchronize(st));
    stats->t_krylov += now() - t0;
    stats->krylov_iterations += its;
    stats->newton_iterations = it + 1;
    stats->last_krylov_relres = rel;
    stats->coarse_iterations = (int)s->coarse_iters;
    if (s->prm.verbose)
      std::fprintf(stderr, "[pff newton] it %d |r| %.6e |r|/|r0| %.3e krylov %d (rel %.2e) coarse its %lld t_res %.3f t_setup %.3f t_krylov %.3f\n",
                   it, rn, rn / r0, its, rel, s->coarse_iters, stats->t_residual, stats->t_setup, stats->t_krylov);
    // backtracking line search (Sec. 5): accept z - alpha dz once the residual is
    // finite, every det F > 0 and ||r|| <= (1 - 1e-4 alpha) ||r_prev||; halve alpha
    // otherwise.  The residual of the accepted point is the next iteration's.
    t0 = now();
    S_CK(cudaMemcpyAsync(s->zold, z, sizeof(double) * n, cudaMemcpyDeviceToDevice, st));
    double alpha = 1.0;
    bool accepted = false;
    for (int ls = 0; ls <= s->prm.line_search_max; ++ls) {
      S_CK(cudaMemcpyAsync(z, s->zold, sizeof(double) * n, cudaMemcpyDeviceToDevice, st));
      S_CK(launch_axpby<double>(z, s->dz, -alpha, 1.0, n, st));
      if (s->prm.line_search_max == 0) { accepted = true; break; }
      S_RC(pff_residual(s->op, z, s->r, st));
      int lst = 0;
      S_RC(pff_get_status(s->op, stream, &lst));
      double r2 = 0.0;
      if (!lst) S_RC(dev_norm2(s, s->r, n, &r2, st));
      const double rt = std::sqrt(r2);
      if (!lst && std::isfinite(rt) && rt <= (1.0 - 1e-4 * alpha) * rn) { accepted = true; break; }
      if (!lst && std::isfinite(rt) && ls == s->prm.line_search_max) { accepted = true; break; }
      alpha *= 0.5;
      stats->line_search_cuts += 1;
    }
    stats->t_residual += now() - t0;
    if (!accepted) {
      S_CK(cudaMemcpyAsync(z, s->zold, sizeof(double) * n, cudaMemcpyDeviceToDevice, st));
      return sfail(PFF_ERR_DEVICE, "pff_newton_solve: line search found no admissible step");
    }
  }
  return PFF_OK;
}

}  // extern "C"

namespace {

template <typename T>
cudaError_t elem_launch(int Q, int P, int mode, const ElemArgs<T>& a, cudaStream_t st) {
  switch (Q) {
    case 2: return launch_elem_q2<T>(P, mode, a, st);
    case 3: return launch_elem_q3<T>(P, mode, a, st);
    case 4: return launch_elem_q4<T>(P, mode, a, st);
    case 5: return launch_elem_q5<T>(P, mode, a, st);
  }
  return cudaErrorInvalidValue;
}

ElemArgs<double> fine_args(pff_op* op) {
  ElemArgs<double> a;
  std::memset(&a, 0, sizeof(a));
  a.mesh = op->mesh;
  a.fix = op->tab.fix;
  a.lin = op->lin64;
  a.nq = op->nq;
  a.geo = op->geo;
  a.kx = op->geo != nullptr;
  for (int d = 0; d < 3; ++d) a.s[d] = op->geom.s[d];
  return a;
}

AdjArgs adj_args(pff_op* op) {
  AdjArgs a;
  std::memset(&a, 0, sizeof(a));
  for (int i = 0; i < op->ctx->nphase; ++i) a.phase[i] = op->ctx->phase[i];
  a.glob = op->ctx->glob;
  a.geom = op->geom;
  a.Q = op->Q;
  a.nphase = op->ctx->nphase;
  a.nq = op->nq;
  a.hist = op->hist_c;
  a.phase_id = op->phase;
  a.status = op->status;
  a.geo = op->geo;
  return a;
}

}  // namespace

extern "C" int pff_adjoint_step(pff_solver* s, const double* z, const double* hist_prev, const uint8_t* sel,
                                double wF, const double* hbar_n, double* hbar_prev, double* grad, double rtol,
                                int maxit, int* iters, void* stream) {
  if (!s || !z || !hist_prev || !sel || !hbar_prev || !grad || !iters)
    return sfail(PFF_ERR_INVALID, "pff_adjoint_step: null argument");
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  pff_op* op = s->op;
  const long long nq = op->nq, n = s->n;
  cudaError_t e = cudaSuccess;
  if (!s->a_in) {
    if (e == cudaSuccess) e = cudaMalloc(&s->a_in, sizeof(double) * 13 * nq);
    if (e == cudaSuccess) e = cudaMalloc(&s->pbuf, sizeof(double) * 13 * nq);
    if (e == cudaSuccess) e = cudaMalloc(&s->qa, sizeof(double) * 13 * nq);
    if (e == cudaSuccess) e = cudaMalloc(&s->ag, sizeof(double) * n);
    if (e == cudaSuccess) e = cudaMalloc(&s->alam, sizeof(double) * n);
    if (e == cudaSuccess) e = cudaMalloc(&s->av, sizeof(double) * n);
    if (e == cudaSuccess) e = cudaMalloc(&s->gth, sizeof(double) * kMaxPhase * 6);
    if (e != cudaSuccess) return sfail(PFF_ERR_CUDA, std::string("pff_adjoint_step: ") + cudaGetErrorString(e));
  }
  // 1. linearisation at (z_n, h_{n-1}): recomputed from the checkpoint
  S_CK(cudaMemcpyAsync(op->hist_c, hist_prev, sizeof(double) * 15 * nq, cudaMemcpyDeviceToDevice, st));
  S_RC(pff_residual(op, z, s->r, st));
  int status = 0;
  S_RC(pff_get_status(op, stream, &status));
  if (status) return sfail(PFF_ERR_DEVICE, "pff_adjoint_step: residual kernel status " + std::to_string(status));
  S_RC(setup(s, st));
  // point inputs a(q)
  ElemArgs<double> ea = fine_args(op);
  ea.x = z;
  ea.scratch = s->a_in;
  S_CK(elem_launch<double>(op->Q, op->p + 1, kEval, ea, st));
  // 2. right-hand side g = wF J_int^T sel + B^T [(dPhi/da)^T hbar_n], zero on Dirichlet DoFs
  S_CK(cudaMemsetAsync(s->ag, 0, sizeof(double) * n, st));
  if (hbar_n) {
    AdjArgs aa = adj_args(op);
    aa.mode = 0;
    aa.a_in = s->a_in;
    aa.hbar = hbar_n;
    aa.qa_out = s->qa;
    S_CK(launch_adjoint_point(aa, st));
    ElemArgs<double> eb = fine_args(op);
    eb.y = s->ag;
    eb.scratch = s->qa;
    S_CK(elem_launch<double>(op->Q, op->p + 1, kBack, eb, st));
  }
  S_CK(launch_sel_scale(s->av, sel, wF, n, st));
  {
    ElemArgs<double> et = fine_args(op);
    const long long stride = (long long)op->Q * op->Q * op->Q * elems_per_block(op->Q);
    et.x = s->av;
    et.y = s->ag;
    et.linP = op->lin64 + kWC * stride;
    et.linC = op->lin64 + kWP * stride;
    et.transpose = 1;
    S_CK(elem_launch<double>(op->Q, op->p + 1, kApply, et, st));
  }
  S_CK(launch_zero_masked(s->ag, op->mask, n, st));
  // 3. adjoint solve J_n^T lam = g (Dirichlet rows/columns identity, g = 0 there)
  s->transpose = 1;
  double rel = 0.0;
  int rc = fgmres(s, s->ag, s->alam, rtol, maxit, iters, &rel, st);
  s->transpose = 0;
  if (rc) return rc;
  // 4. pull-back p = interpolation of (wF sel - lam) to the Gauss points
  S_CK(launch_axpby<double>(s->av, s->alam, -1.0, 1.0, n, st));
  ElemArgs<double> ep = fine_args(op);
  ep.x = s->av;
  ep.scratch = s->pbuf;
  S_CK(elem_launch<double>(op->Q, op->p + 1, kEval, ep, st));
  // 5. history adjoint of the previous step and parameter gradient
  S_CK(cudaMemsetAsync(s->gth, 0, sizeof(double) * kMaxPhase * 6, st));
  AdjArgs ab = adj_args(op);
  ab.mode = 1;
  ab.a_in = s->a_in;
  ab.p = s->pbuf;
  ab.hbar = hbar_n;
  ab.hbar_out = hbar_prev;
  ab.gtheta = s->gth;
  S_CK(launch_adjoint_point(ab, st));
  std::vector<double> h(kMaxPhase * 6);
  S_CK(cudaMemcpyAsync(h.data(), s->gth, sizeof(double) * kMaxPhase * 6, cudaMemcpyDeviceToHost, st));
  S_CK(cudaStreamSynchronize(st));
  for (int i = 0; i < op->ctx->nphase * 6; ++i) grad[i] += h[i];
  S_RC(pff_get_status(op, stream, &status));
  if (status) return sfail(PFF_ERR_DEVICE, "pff_adjoint_step: adjoint kernel status " + std::to_string(status));
  return PFF_OK;
}
