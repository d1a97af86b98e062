"""Fixed-point contractions of the FP64 element kernels at the ends of what they
accept: entries of any exponent, fields that are zero or differ by many orders of
magnitude, subnormal and non-finite entries, every order and level.

Exact statements need no tolerance: a power of two passes through bit for bit
(both exponents shift together), and non-finite entries reach the nodes of their
own elements only.  Against K x the bound is that of the parity tests, 1e-12
(the stored words err by about 1e-13), per field where fields differ in size.
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
from test_gpu_solver import _box  # noqa: E402


@pytest.fixture(scope="module", params=[(2, (3, 2, 4)), (3, (3, 5, 2)), (4, (2, 3, 2))], ids=["Q2", "Q3", "Q4"])
def case(request, orc):
    p, n = request.param
    w = _box(*n, p, 5)
    s = Session(w, levels=(1,))
    s.residual(torch.from_numpy(w.z.ravel()).cuda())
    pff.pff_op_set_deterministic(s.op, True)
    return w, s, orc.assemble(w)["K"]


@pytest.mark.parametrize("shift", [-960, -300, -1, 40, 700])
def test_powers_of_two_pass_through(case, shift):
    w, s, _ = case
    for p in (w.mesh.p, 1):
        x = torch.from_numpy(inputs.random_vector(4 * s.nn(p), 3)).cuda()
        y = s.apply(x, p=p)
        scale = torch.tensor(2.0, dtype=torch.float64).pow(shift).item()
        assert torch.equal(s.apply(x * scale, p=p), y * scale)


def test_fields_of_different_size(case):
    w, s, K = case
    x = inputs.random_vector(w.mesh.ndof, 4).reshape(4, -1)
    for f in range(4):  # one field at a time, the others zero
        one = np.zeros_like(x)
        one[f] = x[f]
        y = s.apply(torch.from_numpy(one.ravel()).cuda()).cpu().numpy()
        ref = K @ one.ravel()
        assert np.linalg.norm(y - ref) <= 1e-12 * np.linalg.norm(ref)
    x *= np.array([1e-9, 1.0, 1e-4, 1e6])[:, None]
    for transpose in (False, True):
        y = s.apply(torch.from_numpy(x.ravel()).cuda(), transpose=transpose).cpu().numpy().reshape(4, -1)
        ref = ((K.T if transpose else K) @ x.ravel()).reshape(4, -1)
        for f in range(4):
            assert np.linalg.norm(y[f] - ref[f]) <= 1e-12 * np.linalg.norm(ref[f])


def test_zero_and_subnormal(case):
    w, s, _ = case
    x = torch.zeros(w.mesh.ndof, dtype=torch.float64, device="cuda")
    assert torch.equal(s.apply(x), x)
    tiny = torch.from_numpy(inputs.random_vector(w.mesh.ndof, 6)).cuda()
    assert torch.isfinite(s.apply(tiny * 2.0 ** -1060)).all()


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
def test_non_finite_entries_stay_in_their_elements(case, bad):
    w, s, _ = case
    m = w.mesh
    x = torch.from_numpy(inputs.random_vector(m.ndof, 7)).cuda()
    clean = s.apply(x)
    # a free node inside the first element
    node = 1 + m.nnx * (1 + m.nny * 1)
    x[2 * m.nn + node] = bad
    y = s.apply(x).reshape(4, -1)
    K, J, I = np.meshgrid(np.arange(m.nnz), np.arange(m.nny), np.arange(m.nnx), indexing="ij")
    inside = torch.from_numpy(((I <= m.p) & (J <= m.p) & (K <= m.p)).ravel()).cuda()
    free = torch.from_numpy(w.mask.astype(bool)).cuda().logical_not()
    assert not torch.isfinite(y[2][inside & free[2]]).any()
    assert torch.equal(y[:, ~inside], clean.reshape(4, -1)[:, ~inside])
