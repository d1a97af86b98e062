"""Assembled order-1 level: stencil products and h-multigrid cycles against the
oracle on grids whose node counts fall on either side of the kernels' tiles
(32 nodes per block), down to a single element.

Tolerances: FP64 sums of 108 products per row, 1e-12; cycles of fewer than
twenty products 1e-11; the FP32 stencil carries 2^-24 per product through the
same cycle, amplified by the Chebyshev recurrence (below a hundredfold): 1e-4.
"""
import numpy as np
import pytest

from paper_2607_21150_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2607_21150_gb300 import pff  # noqa: E402
from paper_2607_21150_gb300.session import Session  # noqa: E402
from test_gpu_solver import _box, np_, rel  # noqa: E402


@pytest.mark.parametrize("mixed", [0, 1])
@pytest.mark.parametrize("n", [(1, 1, 1), (3, 1, 2), (7, 3, 3), (5, 4, 3), (4, 4, 4), (8, 4, 12)])
def test_stencil_products_and_cycles(orc, n, mixed):
    w = _box(*n, 2, 21, state=False)
    s = Session(w, levels=(1,), f32=bool(mixed))
    s.residual(torch.from_numpy(w.z.ravel()).cuda())
    solver = s.solver([2, 1], mixed=mixed, coarse_solver=2)
    pff.pff_solver_setup(solver)
    mask = inputs.coarsen_mask(w.mesh, w.mask, 1)
    A = orc.coarse_operator(orc.assemble(w)["K"], orc.masked_prolongation(orc.prolongation(w.mesh, 1), w.mask, mask), mask)
    As, Ps, dims = [A], [], n
    for _ in range(1, pff.pff_solver_num_hlevels(solver)):
        dims = tuple(d // 2 for d in dims)
        coarse = orc.h_coarse_mask(mask, *dims)
        Ps.append(orc.masked_prolongation(orc.h_prolongation(*dims), mask, coarse))
        As.append(orc.coarse_operator(As[-1], Ps[-1], coarse))
        mask = coarse
    x = inputs.random_vector(A.shape[0], 30)
    y = torch.zeros(len(x), dtype=torch.float64, device="cuda")
    pff.pff_solver_coarse_apply(solver, torch.from_numpy(x).cuda(), y)
    assert rel(np_(y), A @ x) <= (1e-5 if mixed else 1e-12)
    pff.pff_solver_hcycle(solver, torch.from_numpy(x).cuda(), y)
    lams = [pff.pff_solver_hlevel_info(solver, l)[1] for l in range(len(As))]
    assert rel(np_(y), orc.vcycle(As, Ps, [K.diagonal() for K in As], lams, x)) <= (1e-4 if mixed else 1e-11)
    pff.pff_destroy_solver(solver)
