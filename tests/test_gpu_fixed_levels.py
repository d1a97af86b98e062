"""Fixed-point contractions of the FP64 element kernels on every level of every
order: exponents at both ends, and non-finite entries that reach the nodes of their
own elements only (exact statements, see test_gpu_fixed.py)."""
import numpy as np
import pytest

from paper_2607_21150_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2607_21150_gb300 import pff  # noqa: E402
from paper_2607_21150_gb300.session import Session  # noqa: E402
from test_gpu_solver import _box  # noqa: E402

LEVELS = [(p, l) for p in (1, 2, 3, 4) for l in range(p, 0, -1)]


@pytest.fixture(scope="module")
def sessions():
    out = {}
    for p in (1, 2, 3, 4):
        w = _box(3, 5, 2, p, 5)
        out[p] = s = Session(w, levels=range(1, p))
        s.residual(torch.from_numpy(w.z.ravel()).cuda())
        pff.pff_op_set_deterministic(s.op, True)
    return out


@pytest.mark.parametrize("transpose", [False, True])
@pytest.mark.parametrize("p,l", LEVELS)
def test_powers_of_two_pass_through(sessions, p, l, transpose):
    s = sessions[p]
    x = torch.from_numpy(inputs.random_vector(4 * s.nn(l), 3)).cuda()
    y = s.apply(x, p=l, transpose=transpose)
    for shift in (-960, -300, -1, 40, 700):
        scale = torch.tensor(2.0, dtype=torch.float64).pow(shift).item()
        assert torch.equal(s.apply(x * scale, p=l, transpose=transpose), y * scale)


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("p,l", LEVELS)
def test_non_finite_entries_stay_in_their_elements(sessions, p, l, bad):
    s = sessions[p]
    m = s.w.mesh
    nx, ny, nz = (l * k + 1 for k in (m.nx, m.ny, m.nz))
    mask = s.w.mask if l == p else inputs.coarsen_mask(m, s.w.mask, l)
    free = torch.from_numpy(mask.reshape(4, -1) == 0).cuda()
    x = torch.from_numpy(inputs.random_vector(4 * s.nn(l), 7)).cuda()
    clean = s.apply(x, p=l).reshape(4, -1)
    # the vertex of the elements (0 and 1, 0 and 1, 0 and 1), which is free
    x[2 * s.nn(l) + l + nx * (l + ny * l)] = bad
    y = s.apply(x, p=l).reshape(4, -1)
    K, J, I = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    inside = torch.from_numpy(((I <= 2 * l) & (J <= 2 * l) & (K <= 2 * l)).ravel()).cuda()
    assert not torch.isfinite(y[2][inside & free[2]]).any()
    assert torch.equal(y[:, ~inside], clean[:, ~inside])
