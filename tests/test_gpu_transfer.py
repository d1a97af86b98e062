"""p-transfers against the Kronecker product of the 1D prolongations, for every
pair of orders and boxes on both sides of the kernels' tiles (64 x 16 fine nodes,
32 x 16 in FP64), with arbitrary prescribed entries on both levels.

Tolerance: a restricted value sums at most 7^3 products of weights below one
whose absolute sum stays below 10 per direction's worst row, with round-off u per
stage of three: 1e-13 in FP64, 2e-6 in FP32 (relative 2-norm).
"""
import numpy as np
import pytest

from paper_2607_21150_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2607_21150_gb300 import pff  # noqa: E402


def matrix(n, pf, pc):
    xc, xf = inputs.gll_points(pc), inputs.gll_points(pf)
    P = np.zeros((pf * n + 1, pc * n + 1))
    for a, t in enumerate(xf):
        for b in range(pc + 1):
            w = np.prod([(t - xc[m]) / (xc[b] - xc[m]) for m in range(pc + 1) if m != b])
            P[pf * np.arange(n) + a, pc * np.arange(n) + b] = w
    return P


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("n", [(1, 1, 1), (2, 3, 2), (16, 4, 2), (17, 5, 3), (33, 9, 1), (11, 8, 4)])
@pytest.mark.parametrize("pf,pc", [(2, 1), (3, 1), (3, 2), (4, 1), (4, 2), (4, 3)])
def test_transfers(pf, pc, n, dtype):
    rng = np.random.default_rng(7)
    ctx = pff.pff_create_context(inputs.phase_vector(inputs.EX3_MATRIX)[None], 2, 1e-3, 1e-2, 0.01, 2.5e5)
    basis = pff.pff_create_basis(ctx, pf, pf + 1)
    nf = [4] + [pf * m + 1 for m in reversed(n)]
    nc = [4] + [pc * m + 1 for m in reversed(n)]
    restr = pff.pff_create_restriction(ctx, (*n, 0.1, 0.1, 0.1), pf, None, int(np.prod(nf[1:])))
    op = pff.pff_create_operator(ctx, basis, restr)
    fine, coarse = pff.pff_create_level(op, pf), pff.pff_create_level(op, pc)
    mf, mc = (rng.random(nf) < 0.1), (rng.random(nc) < 0.1)
    pff.pff_set_dirichlet(op, torch.from_numpy(mf.astype(np.uint8)).cuda(), None)
    pff.pff_level_set_mask(coarse, torch.from_numpy(mc.astype(np.uint8)).cuda())
    prec = pff.PFF_F64 if dtype == torch.float64 else pff.PFF_F32
    xc, rf = rng.uniform(-1, 1, nc), rng.uniform(-1, 1, nf)
    Px, Py, Pz = (matrix(m, pf, pc) for m in n)
    want_f = np.einsum("fcba,zc,yb,xa->fzyx", np.where(mc, 0.0, xc), Pz, Py, Px, optimize=True)
    want_c = np.einsum("fzyx,zc,yb,xa->fcba", np.where(mf, 0.0, rf), Pz, Py, Px, optimize=True)
    xf = torch.full(nf, float("nan"), dtype=dtype, device="cuda")
    rc = torch.full(nc, float("nan"), dtype=dtype, device="cuda")
    pff.pff_prolong(coarse, fine, prec, torch.from_numpy(xc).to("cuda", dtype), xf)
    pff.pff_restrict(coarse, fine, prec, torch.from_numpy(rf).to("cuda", dtype), rc)
    for got, want in ((xf, np.where(mf, 0.0, want_f)), (rc, np.where(mc, 0.0, want_c))):
        err = np.linalg.norm(got.double().cpu().numpy() - want) / np.linalg.norm(want)
        assert err <= (1e-13 if dtype == torch.float64 else 2e-6)
    for h in (coarse, fine):
        pff.pff_destroy_level(h)
    pff.pff_destroy_operator(op)
    pff.pff_destroy_restriction(restr)
    pff.pff_destroy_basis(basis)
    pff.pff_destroy_context(ctx)
