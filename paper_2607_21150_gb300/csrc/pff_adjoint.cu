// Adjoint of the pointwise update: the derivatives of the residual integrands f
// and of the trial history Phi (Box 1 step 4) with respect to the point inputs
// a = (grad_X u, phi, grad_X phi), the committed history h and the point's own
// phase parameters (E_inf, nu_inf, sigma0, eta_d, Gc, l0), contracted with the
// adjoint weights of the load-step recursion by one reverse pass per point.
//
// The paper linearises only in (u, phi) (Appendix B/C).  The derivatives here
// extend the same principal-frame construction: for a perturbation db of the
// trial b of a branch (db = ell b + b ell^T + F dC F^T, ell = dF F^-1), the
// eigenvalue terms follow Box A1 and the eigenvector terms the divided
// differences (t_i - t_j)/(b_i - b_j) = mu a log1p(x)/(x b_j) for the stress
// and (g_i - g_j)/(b_i - b_j) = g_j/b_j expm1(a log1p(x))/x for the committed
// b^e = N diag(g) N^T, g_i = exp(2 (a eps_d,i + theta/3)) = K b_i^a; both stay
// smooth where eigenvalues coincide.
//
// In the eigenframe of a branch the reverse pass needs two 3x3 matrices only:
//   That = N^T (g S) N,   S = adjoint of the degraded stress, and
//   Ghat = N^T (F^-T Hb F^-1) N,   Hb = adjoint of the committed C_in^-1,
// from which the adjoints of the branch factor a, of the principal strains and
// of db follow in closed form.  Bound by the FP64 pipe: about 3000 FP64
// operations per point with three branches.  The forward form it replaces took
// each of the 10 (mode 0) or 21 (mode 1) input directions through every branch:
// 29.0 ms per call on 373 k points (24^3 Q2), spilling its 3x3 temporaries.
#include <cmath>

#include "pff_internal.h"
#include "pff_point.cuh"

namespace pff {

namespace {

struct Branch {
  bool has, plastic;
  double mu, af, s2, q, c;  // c: Maxwell mu dt / eta_d
  double dgam, H, esig0;    // Prandtl: plastic increment, slope of sigma_y, d sigma_y / d sigma0 at ep_n + dgam
  double N[3][3], x[3], ed[3];
};

// (b_p^a - b_q^a) / (b_p - b_q) * K with K b_q^a = ghat_q, from x = b - 1.
__device__ double power_ratio(double a, double xp, double xq, double gq) {
  const double bq = 1.0 + xq;
  const double y = (xp - xq) / bq;
  double r;
  if (fabs(y) < 1e-4) r = a * (1.0 + 0.5 * (a - 1.0) * y * (1.0 + (a - 2.0) * y / 3.0));
  else r = expm1(a * log1p(y)) / y;
  return gq / bq * r;
}

// C = N^T S N
__device__ __forceinline__ void to_frame(const double N[3][3], const double S[3][3], double C[3][3]) {
  double T[3][3];
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int c = 0; c < 3; ++c) T[r][c] = S[r][0] * N[0][c] + S[r][1] * N[1][c] + S[r][2] * N[2][c];
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int c = 0; c < 3; ++c) C[r][c] = N[0][r] * T[0][c] + N[1][r] * T[1][c] + N[2][r] * T[2][c];
}

}  // namespace

template <int MODE>
__global__ void __launch_bounds__(128) k_adjoint_point(const AdjArgs a) {
  __shared__ double red[kMaxPhase * 6];
  if (MODE == 1) {
    for (int i = threadIdx.x; i < kMaxPhase * 6; i += blockDim.x) red[i] = 0.0;
    __syncthreads();
  }
  const long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  int pid = -1;
  double gpar[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  if (q < a.nq) {
    const long long nq = a.nq;
    int status = 0;
    pid = a.phase_id[q];
    if (pid >= a.nphase) { status |= 8; pid = 0; }
    const PhaseDev& ph = a.phase[pid];
    const GlobDev& gl = a.glob;

    // ---------------- primal
    double F[3][3], Fi[3][3], GG[3][3];
    double theta;
    {
      double Hm[3][3];
#pragma unroll
      for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          Hm[r][c] = a.a_in[(3 * r + c) * nq + q];
          F[r][c] = Hm[r][c] + (r == c ? 1.0 : 0.0);
        }
      const double trH = Hm[0][0] + Hm[1][1] + Hm[2][2];
      double trHH = 0.0;
#pragma unroll
      for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) trHH += Hm[r][c] * Hm[c][r];
      const double detH = Hm[0][0] * (Hm[1][1] * Hm[2][2] - Hm[1][2] * Hm[2][1]) -
                          Hm[0][1] * (Hm[1][0] * Hm[2][2] - Hm[1][2] * Hm[2][0]) +
                          Hm[0][2] * (Hm[1][0] * Hm[2][1] - Hm[1][1] * Hm[2][0]);
      const double Jm1 = trH + 0.5 * (trH * trH - trHH) + detH;
      if (!(Jm1 > -1.0)) status |= 2;
      theta = 2.0 * half_log1p(Jm1);
      const double rJ = rcp64(1.0 + Jm1);
#pragma unroll
      for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const int r1 = (r + 1) % 3, r2 = (r + 2) % 3, c1 = (c + 1) % 3, c2 = (c + 2) % 3;
          Fi[r][c] = (F[c1][r1] * F[c2][r2] - F[c1][r2] * F[c2][r1]) * rJ;
          GG[r][c] = Hm[r][c] + Hm[c][r] + Hm[r][0] * Hm[c][0] + Hm[r][1] * Hm[c][1] + Hm[r][2] * Hm[c][2];
        }
    }
    const double phi = a.a_in[9 * nq + q];
    const double omp = 1.0 - phi;
    const double g = omp * omp + gl.eta;
    const double gp = -2.0 * omp;
    const double epn = a.hist[12 * nq + q];

    Branch Bs[3];
    double psid = 0.0;
#pragma unroll
    for (int br = 0; br < 3; ++br) {
      Branch& B = Bs[br];
      B.has = ph.has[br] != 0;
      B.plastic = false;
      if (!B.has) continue;
      B.mu = ph.mu[br];
      double X[3][3];
#pragma unroll
      for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) X[r][c] = GG[r][c];
      if (br > 0) {
        double M[3][3], FM[3][3];
#pragma unroll
        for (int v = 0; v < 6; ++v) {
          int r, c;
          vo_idx(v, r, c);
          const double m = a.hist[(6 * (br - 1) + v) * nq + q] - (v < 3 ? 1.0 : 0.0);
          M[r][c] = m; M[c][r] = m;
        }
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
          for (int c = 0; c < 3; ++c) FM[r][c] = F[r][0] * M[0][c] + F[r][1] * M[1][c] + F[r][2] * M[2][c];
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
          for (int c = r; c < 3; ++c) {
            const double sm = FM[r][0] * F[c][0] + FM[r][1] * F[c][1] + FM[r][2] * F[c][2];
            X[r][c] += sm;
            if (c != r) X[c][r] += sm;
          }
      }
      if (!eigh3(X, B.N, B.x)) status |= 1;
      double tr = 0.0;
#pragma unroll
      for (int p = 0; p < 3; ++p) {
        B.ed[p] = half_log1p(B.x[p]);
        tr += B.ed[p];
      }
#pragma unroll
      for (int p = 0; p < 3; ++p) B.ed[p] -= tr * (1.0 / 3.0);
      B.s2 = B.ed[0] * B.ed[0] + B.ed[1] * B.ed[1] + B.ed[2] * B.ed[2];
      B.af = 1.0;
      B.c = 0.0;
      if (br == 1) {
        B.c = ph.cmax;
        B.af = 1.0 / (1.0 + B.c * g);
      } else if (br == 2) {
        B.q = 2.0 * B.mu * sqrt(1.5 * B.s2);
        if (g * B.q - yield_stress(ph, epn) > 0.0) {
          int ok;
          B.dgam = return_map(ph, g, B.mu, B.q, epn, &ok);
          if (!ok) status |= 16;
          B.H = yield_slope(ph, epn + B.dgam);
          B.esig0 = ph.hard ? exp(-ph.beta * (epn + B.dgam)) : 1.0;
          B.af = 1.0 - 3.0 * B.mu * B.dgam / B.q;
          B.plastic = true;
        }
      }
      psid += B.mu * B.af * B.af * B.s2;
    }
    const bool tens = theta >= 0.0;
    const double psip = tens ? psid + 0.5 * ph.kap_tot * theta * theta : psid;
    const double Hn = a.hist[13 * nq + q];
    const bool active = psip > Hn;

    // ---------------- reverse pass
    const double h12 = a.hbar ? a.hbar[12 * nq + q] : 0.0;
    const double h13 = a.hbar ? a.hbar[13 * nq + q] : 0.0;
    double Hbar = h13;       // adjoint of the trial history field H
    double St[3][3];         // mode 1: g times the adjoint of the degraded stress
    double out12 = h12;      // adjoint of ep_n
    if (MODE == 1) {
      const int Q = a.Q, Q2 = Q * Q, Q3 = Q2 * Q;
      const int lq = (int)(q % Q3);
      const double wdet = a.geo ? a.geo[9 * nq + q]
                                : a.geom.wq[lq % Q] * a.geom.wq[(lq / Q) % Q] * a.geom.wq[lq / Q2] * a.geom.detJ;
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        const double p0 = wdet * a.p[(3 * r) * nq + q], p1 = wdet * a.p[(3 * r + 1) * nq + q],
                     p2 = wdet * a.p[(3 * r + 2) * nq + q];
#pragma unroll
        for (int c = 0; c < 3; ++c) St[r][c] = p0 * Fi[0][c] + p1 * Fi[1][c] + p2 * Fi[2][c];
      }
      const double Lbar = wdet * a.p[9 * nq + q] * gl.s_phi;
      double kbar = 0.0;
#pragma unroll
      for (int A = 0; A < 3; ++A) kbar += wdet * a.p[(10 + A) * nq + q] * a.a_in[(10 + A) * nq + q];
      Hbar += gp * Lbar;
      const double alphap = (gl.at == 1) ? 1.0 : 2.0 * phi;
      const double gcbar = alphap * Lbar / ph.c0, kpbar = 2.0 * gl.s_phi * kbar / ph.c0;
      gpar[4] = gcbar / ph.l0 + kpbar * ph.l0;
      gpar[5] = kpbar * ph.Gc - gcbar * ph.Gc / (ph.l0 * ph.l0);
      const double tvbar = (tens ? g : 1.0) * (St[0][0] + St[1][1] + St[2][2]);
      const double kap0bar = theta * tvbar + ((tens && active) ? 0.5 * theta * theta * Hbar : 0.0);
      const double tnu = 1.0 - 2.0 * ph.nu0;
      gpar[0] = kap0bar / (3.0 * tnu);
      gpar[1] = 2.0 * kap0bar * ph.E0 / (3.0 * tnu * tnu);
      a.hbar_out[13 * nq + q] = active ? 0.0 : Hbar;
      a.hbar_out[14 * nq + q] = -gl.zdt * Lbar;
#pragma unroll
      for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) St[r][c] *= g;
    }
    const double psibar = active ? Hbar : 0.0;  // adjoint of psi+
    double gbar = 0.0;                          // mode 0: adjoint of g(phi)
    double thbar = (MODE == 0 && tens) ? ph.kap_tot * theta * psibar : 0.0;
    double eb[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};  // mode 0: adjoint of ell
#pragma unroll
    for (int br = 0; br < 3; ++br) {
      const Branch& B = Bs[br];
      if (!B.has) {
        if (MODE == 1 && br > 0)  // absent branch: the history words pass through
          for (int v = 0; v < 6; ++v)
            a.hbar_out[(6 * (br - 1) + v) * nq + q] = a.hbar ? a.hbar[(6 * (br - 1) + v) * nq + q] : 0.0;
        continue;
      }
      double abar = 0.0, edbar[3] = {0.0, 0.0, 0.0}, off[3] = {0.0, 0.0, 0.0};  // off: pairs (0,1), (0,2), (1,2) of db
      double eddebar = 2.0 * psibar * B.mu * B.af * B.af;  // adjoint of eps_d . d eps
      const double rp[3] = {B.x[0], B.x[0], B.x[1]}, rq[3] = {B.x[1], B.x[2], B.x[2]};
      double G[3][3], ghat[3];
      if (MODE == 1) {
        double T[3][3];
        to_frame(B.N, St, T);
        const double ted = B.ed[0] * T[0][0] + B.ed[1] * T[1][1] + B.ed[2] * T[2][2];
        if (br == 0) {
          const double onu = 1.0 + ph.nu0;
          const double mubar = 2.0 * B.af * ted + psibar * B.af * B.af * B.s2;
          gpar[0] += mubar / (2.0 * onu);
          gpar[1] -= mubar * ph.E0 / (2.0 * onu * onu);
          continue;
        }
        abar = 2.0 * B.mu * ted;
#pragma unroll
        for (int p = 0; p < 3; ++p) edbar[p] = 2.0 * B.mu * B.af * T[p][p];
        const double mua = B.mu * B.af;
        off[0] = mua * log_ratio(rp[0], rq[0]) * (T[0][1] + T[1][0]);
        off[1] = mua * log_ratio(rp[1], rq[1]) * (T[0][2] + T[2][0]);
        off[2] = mua * log_ratio(rp[2], rq[2]) * (T[1][2] + T[2][1]);
      }
      if (br > 0) {
        abar += 2.0 * psibar * B.mu * B.af * B.s2;
        if (a.hbar) {
          double Hb[3][3], M[3][3];
#pragma unroll
          for (int v = 0; v < 6; ++v) {
            int r, c;
            vo_idx(v, r, c);
            const double hv = a.hbar[(6 * (br - 1) + v) * nq + q] * (v < 3 ? 1.0 : 0.5);
            Hb[r][c] = hv; Hb[c][r] = hv;
          }
          to_frame(Fi, Hb, M);
          to_frame(B.N, M, G);
#pragma unroll
          for (int p = 0; p < 3; ++p) {
            ghat[p] = exp_near(2.0 * (B.af * B.ed[p] + theta * (1.0 / 3.0)));
            const double gg = 2.0 * ghat[p] * G[p][p];
            abar += gg * B.ed[p];
            edbar[p] += gg * B.af;
            if (MODE == 0) thbar += gg * (1.0 / 3.0);
          }
          off[0] += 2.0 * power_ratio(B.af, rp[0], rq[0], ghat[1]) * G[0][1];
          off[1] += 2.0 * power_ratio(B.af, rp[1], rq[1], ghat[2]) * G[0][2];
          off[2] += 2.0 * power_ratio(B.af, rp[2], rq[2], ghat[2]) * G[1][2];
        }
        if (br == 1) {
          if (MODE == 0) gbar -= abar * B.af * B.af * B.c;
          else if (B.c != 0.0) gpar[3] += abar * B.af * B.af * B.c * g / ph.eta_d;
        } else if (B.plastic) {
          // implicit derivative of the degraded consistency condition
          // g q - 3 g mu dgam - sigma_y(ep_n + dgam; sigma0) = 0
          const double rden = 1.0 / (3.0 * g * B.mu + B.H);
          const double dgbar = (h12 - 3.0 * B.mu * abar / B.q) * rden;
          const double qbar = 3.0 * B.mu * B.dgam * abar / (B.q * B.q) + dgbar * g;
          eddebar += qbar * B.q / B.s2;
          if (MODE == 0) {
            gbar += dgbar * (B.q - 3.0 * B.mu * B.dgam);
          } else {
            gpar[2] -= dgbar * B.esig0;
            out12 -= dgbar * B.H;
          }
        }
      }
      const double em = (edbar[0] + edbar[1] + edbar[2]) * (1.0 / 3.0);
      double dep[3];  // adjoint of the principal strain increments
#pragma unroll
      for (int p = 0; p < 3; ++p) dep[p] = edbar[p] - em + B.ed[p] * eddebar;
      if (MODE == 0) {
        // d eps_p = lh_pp, db_pr = lh_pr b_r + b_p lh_rp with lh = N^T ell N, and
        // dF^-1 = -F^-1 ell in the committed history
        double lb[3][3];
        lb[0][0] = dep[0]; lb[1][1] = dep[1]; lb[2][2] = dep[2];
        lb[0][1] = off[0] * (1.0 + B.x[1]); lb[1][0] = off[0] * (1.0 + B.x[0]);
        lb[0][2] = off[1] * (1.0 + B.x[2]); lb[2][0] = off[1] * (1.0 + B.x[0]);
        lb[1][2] = off[2] * (1.0 + B.x[2]); lb[2][1] = off[2] * (1.0 + B.x[1]);
        if (br > 0 && a.hbar)
#pragma unroll
          for (int p = 0; p < 3; ++p)
#pragma unroll
            for (int r = 0; r < 3; ++r) lb[p][r] -= 2.0 * G[p][r] * ghat[r];
        double NL[3][3];
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
          for (int r = 0; r < 3; ++r) NL[i][r] = B.N[i][0] * lb[0][r] + B.N[i][1] * lb[1][r] + B.N[i][2] * lb[2][r];
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
          for (int j = 0; j < 3; ++j)
            eb[i][j] += NL[i][0] * B.N[j][0] + NL[i][1] * B.N[j][1] + NL[i][2] * B.N[j][2];
      } else {
        // db = W^T dC W, W = F^T N
        double W[3][3], V[3][3];
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
          for (int p = 0; p < 3; ++p) W[r][p] = F[0][r] * B.N[0][p] + F[1][r] * B.N[1][p] + F[2][r] * B.N[2][p];
#pragma unroll
        for (int p = 0; p < 3; ++p) dep[p] /= 2.0 * (1.0 + B.x[p]);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          V[i][0] = dep[0] * W[i][0];
          V[i][1] = dep[1] * W[i][1] + off[0] * W[i][0];
          V[i][2] = dep[2] * W[i][2] + off[1] * W[i][0] + off[2] * W[i][1];
        }
#pragma unroll
        for (int v = 0; v < 6; ++v) {
          int r, c;
          vo_idx(v, r, c);
          double cb = V[r][0] * W[c][0] + V[r][1] * W[c][1] + V[r][2] * W[c][2];
          if (r != c) cb += V[c][0] * W[r][0] + V[c][1] * W[r][1] + V[c][2] * W[r][2];
          a.hbar_out[(6 * (br - 1) + v) * nq + q] = cb;
        }
      }
    }
    if (MODE == 1) a.hbar_out[12 * nq + q] = out12;
    if (MODE == 0) {
#pragma unroll
      for (int i = 0; i < 3; ++i) eb[i][i] += thbar;
      double Fb[3][3];  // ell = dF F^-1
#pragma unroll
      for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int k = 0; k < 3; ++k) Fb[r][k] = eb[r][0] * Fi[k][0] + eb[r][1] * Fi[k][1] + eb[r][2] * Fi[k][2];
      // parent-frame pseudo-integrands for the transposed basis (no weight)
#pragma unroll
      for (int f = 0; f < 3; ++f)
#pragma unroll
        for (int al = 0; al < 3; ++al)
          a.qa_out[(3 * f + al) * nq + q] =
              a.geo ? a.geo[(3 * al) * nq + q] * Fb[f][0] + a.geo[(3 * al + 1) * nq + q] * Fb[f][1] +
                          a.geo[(3 * al + 2) * nq + q] * Fb[f][2]
                    : a.geom.s[al] * Fb[f][al];
      a.qa_out[9 * nq + q] = (a.hbar ? a.hbar[14 * nq + q] : 0.0) + gp * gbar;
#pragma unroll
      for (int m = 10; m < 13; ++m) a.qa_out[m * nq + q] = 0.0;
    }
    if (status) atomicOr(a.status, status);
  }
  if (MODE == 1) {
    // parameter gradient: summed over the warp's lanes of one phase at a time
    unsigned left = __ballot_sync(0xffffffffu, pid >= 0);
    while (left) {
      const int k = __shfl_sync(0xffffffffu, pid, __ffs(left) - 1);
      left &= ~__ballot_sync(0xffffffffu, pid == k);
#pragma unroll
      for (int j = 0; j < 6; ++j) {
        double v = pid == k ? gpar[j] : 0.0;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0 && v != 0.0) atomicAdd(&red[k * 6 + j], v);
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < a.nphase * 6; i += blockDim.x)
      if (red[i] != 0.0) atomicAdd(a.gtheta + i, red[i]);
  }
}

cudaError_t launch_adjoint_point(const AdjArgs& a, cudaStream_t st) {
  if (a.nq == 0) return cudaSuccess;
  const unsigned nb = (unsigned)((a.nq + 127) / 128);
  if (a.mode == 0) k_adjoint_point<0><<<nb, 128, 0, st>>>(a);
  else k_adjoint_point<1><<<nb, 128, 0, st>>>(a);
  note_launch();
  return cudaGetLastError();
}

}  // namespace pff
