"""Right-hand sides at which a Krylov solve ends before its first iteration: zero,
and entries whose squares leave FP64 (||b|| infinite, which no residual can fall
below).  Both leave x = 0 after no iteration, a zero one without any work beyond
its norm; the coarse solve inside a V-cycle leaves its correction out likewise.
"""
import math

import pytest

from paper_2607_21150_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2607_21150_gb300 import pff  # noqa: E402
from paper_2607_21150_gb300.session import Session  # noqa: E402
from test_gpu_solver import _box  # noqa: E402


@pytest.fixture(scope="module")
def session():
    s = Session(_box(4, 4, 4, 2, 33), levels=(1,))
    s.residual(torch.from_numpy(s.w.z.ravel()).cuda())
    return s


@pytest.mark.parametrize("coarse_solver", [0, 1, 2])
def test_ends_before_the_first_iteration(session, coarse_solver):
    s = session
    solver = s.solver([2, 1], mixed=0, coarse_solver=coarse_solver)
    pff.pff_solver_setup(solver)
    b = torch.from_numpy(inputs.random_vector(s.w.mesh.ndof, 3)).cuda()
    x = torch.full_like(b, 7.0)
    before = pff.pff_kernel_launches()
    its, rel = pff.pff_solver_krylov(solver, torch.zeros_like(b), x, 1e-8, 50)
    assert pff.pff_kernel_launches() - before <= 2
    assert its == 0 and rel == 0.0 and torch.count_nonzero(x).item() == 0
    x.fill_(7.0)
    its, rel = pff.pff_solver_krylov(solver, b * 1e200, x, 1e-8, 50)
    assert its == 0 and math.isnan(rel) and torch.count_nonzero(x).item() == 0
    pff.pff_solver_vcycle(solver, torch.zeros_like(b), x)
    assert torch.count_nonzero(x).item() == 0
    pff.pff_solver_vcycle(solver, b * 1e200, x)
    assert torch.isfinite(x).all() and torch.count_nonzero(x).item() > 0
    pff.pff_destroy_solver(solver)
