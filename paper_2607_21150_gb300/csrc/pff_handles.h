// Definitions of the opaque libpff handles, shared by the ABI and solver files.
#pragma once
#include <vector>

#include "../../include/pff.h"
#include "pff_internal.h"

using pff::PhaseDev;
using pff::GlobDev;
using pff::MeshDev;
using pff::Geom;
using pff::kMaxPhase;

struct pff_ctx {
  int nphase;
  PhaseDev phase[kMaxPhase];
  GlobDev glob;
};

struct pff_basis {
  int p, q;
  std::vector<double> xg, xq, wq, B, Dc, Dt;
};

struct pff_restr {
  pff_box box;
  int p;
  const int32_t* offsets;
  int64_t nn;
};

struct Tables {  // 1D matrices of a level: device copies for the assembled level (FP64) and the FP32 actions
  double *B64 = nullptr, *Dt64 = nullptr;
  float *B32 = nullptr, *Dc32 = nullptr;
  // B, D_t and D_c in FP32, each entry twice (kernel parameters)
  unsigned long long hB2[pff::kMaxQ * pff::kMaxQ] = {}, hD2[pff::kMaxQ * pff::kMaxQ] = {},
                     hDc2[pff::kMaxQ * pff::kMaxQ] = {};
  double hB[pff::kMaxQ * pff::kMaxQ] = {}, hDt[pff::kMaxQ * pff::kMaxQ] = {};
  pff::FixTab fix = {};  // the same for the FP64 kernels' fixed-point contractions
};

struct pff_op {
  pff_ctx* ctx;
  int p, Q;
  pff_box box;
  MeshDev mesh;
  long long nq, nel;
  Geom geom;
  Tables tab;
  double* hist_c = nullptr;
  double* hist_t = nullptr;
  uint8_t* phase = nullptr;
  uint8_t* flags = nullptr;
  double* lin64 = nullptr;
  float* lin32 = nullptr;     // FP32 copy (lin32_word layout)
  long long lin_len = 0;
  double* io = nullptr;
  uint8_t* mask = nullptr;
  uint8_t* emask = nullptr;   // [nel] elements with masked nodes (fine level), from pff_set_dirichlet
  double* dvals = nullptr;
  int* status = nullptr;
  int f32 = 0;
  int df = 0;                 // PFF_DF64 actions allowed (pff_op_enable_df)
  int det = 0;                // deterministic transpose (pff_op_set_deterministic)
  void* evec = nullptr;       // its element values, [nel][4][P^3] doubles of the fine order
  uint16_t* lin16 = nullptr;  // BF16 words (lin16_word layout), written by pff_residual when bf16 = 1
  long long lin16_len = 0;    // uint16 entries at lin16
  int bf16 = 0;
  double* geo = nullptr;      // mapped mesh: [10][nq] d xi / dX and w det J (null: the affine box)
  double* fint = nullptr;     // internal force work vector of pff_reaction (allocated on first use)
  double* sums = nullptr;     // 8 doubles (reaction sums, state summary)
};

namespace pff { struct HostIO; }

struct pff_level {
  pff::HostIO* hio = nullptr;  // device staging and streams of pff_jacobian_apply_host (created on first use)
  pff_op* op;
  int p;
  MeshDev mesh;
  Tables tab;
  uint8_t* mask = nullptr;   // owned copy (coarse levels) ; fine level uses op->mask
  uint8_t* emask = nullptr;  // [nel] elements with masked nodes (coarse levels; the fine level uses op->emask)
  bool is_fine = false;
  // prolongation table towards the finer level with order I_pf
  int I_pf = -1;
  double I1[pff::kMaxQ * pff::kMaxQ] = {};  // [I_pf + 1][p + 1]
};


namespace pff {
// Element blocks [blk0, blk0 + nblk) of a level action (nblk = 0: all), without
// the initialisation of y; prec PFF_F64, PFF_F32, PFF_DF64 or PFF_F32_BF16
// (pff_abi.cpp).
int apply_blocks(pff_level* L, int prec, const void* x, void* y, int transpose, int blk0, int nblk, cudaStream_t st);
// Chebyshev smoothing of J x = b or (transpose) J^T x = b on a level (Saad, Alg.
// 12.1); work: three level vectors.  from_zero: x is zero on entry and not read,
// and the first product is left out (pff_abi.cpp).
int smooth_level(pff_level* L, int prec, bool transpose, bool from_zero, int degree, double lmin, double lmax,
                 const void* diag, const void* b, void* x, void* work, cudaStream_t st);
// pff_prolong and pff_restrict with x_f += P x_c (add) and r_c = P^T (b - r_f)
// (b not null) (pff_abi.cpp).
int transfer_prolong(pff_level* c, pff_level* f, int prec, const void* xc, void* xf, bool add, cudaStream_t st);
int transfer_restrict(pff_level* c, pff_level* f, int prec, const void* rf, const void* b, void* rc, cudaStream_t st);
// The Dirichlet mask of a level's rows (pff_abi.cpp).
const uint8_t* level_rows_mask(const pff_level* L);
// Releases the staging buffers, streams and events of pff_jacobian_apply_host (pff_hostio.cpp).
void free_host_io(pff_level* L);
}  // namespace pff
