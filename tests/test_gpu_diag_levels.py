"""Diagonal of every level of every fine order, on boxes that fill the blocks of the
element kernels partly (the last block's lines belong to no element), box and
curved meshes, against the diagonal of the oracle's Galerkin operator P^T K P.

Tolerance: sums of at most 4 Q^3 positive and negative terms from words that err by
about 1e-13: 1e-12 in FP64 (the parity bar); 2e-5 in FP32 (words and products
rounded at 2^-24, as for the FP32 actions).
"""
import pytest

from paper_2607_21150_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2607_21150_gb300 import pff  # noqa: E402
from paper_2607_21150_gb300.session import Session  # noqa: E402
from test_gpu_solver import _box, np_, rel  # noqa: E402


@pytest.mark.parametrize("curved", [False, True])
@pytest.mark.parametrize("p,n", [(1, (5, 3, 5)), (2, (5, 3, 2)), (3, (3, 2, 3)), (4, (3, 2, 2))])
def test_diagonals(orc, p, n, curved):
    w = _box(*n, p, 5)
    if curved:
        w.X = inputs.mapped_coords(w.mesh, "smooth", amp=0.15, seed=5)
    s = Session(w, levels=range(1, p), f32=True)
    s.residual(torch.from_numpy(w.z.ravel()).cuda())
    K = orc.assemble(w)["K"]
    for l in range(p, 0, -1):
        want = K
        if l < p:
            mask = inputs.coarsen_mask(w.mesh, w.mask, l)
            want = orc.coarse_operator(K, orc.masked_prolongation(orc.prolongation(w.mesh, l), w.mask, mask), mask)
        assert rel(np_(s.diag(p=l)), want.diagonal()) <= 1e-12
        assert rel(np_(s.diag(p=l, prec=pff.PFF_F32)), want.diagonal()) <= 2e-5
    s.close()
