"""Chebyshev smoothing against the textbook recurrence written with level
actions and torch vectors, for every degree at which the fused updates differ
(1: none, 2: first and last in one, 3 and 5: all), caller vectors on and off
16-byte boundaries, with and without prescribed entries.

Tolerance: both sides carry the unit round-off of their type through at most six
products with D^-1 J of spectral radius below 10 on [0.35, 3.8] (amplification
below 1e4): 1e-11 in FP64, 5e-3 of the FP32 round-off scale, i.e. 1e-4, in FP32.
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


@pytest.fixture(scope="module", params=[True, False], ids=["dirichlet", "free"])
def session(request):
    w = _box(3, 2, 4, 2, 5, state=False)
    if not request.param:
        w.mask = w.dvals = None
    s = Session(w, f32=True, bf16=True)
    s.residual(torch.from_numpy(w.z.ravel()).cuda())
    return s


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("degree", [1, 2, 3, 5])
@pytest.mark.parametrize("prec", [pff.PFF_F64, pff.PFF_F32, pff.PFF_F32_BF16])
def test_smoothing_is_the_recurrence(session, prec, degree, offset):
    s = session
    dtype = torch.float64 if prec == pff.PFF_F64 else torch.float32
    n = s.w.mesh.ndof

    def vec(seed, lo=-1.0):
        v = torch.empty(n + 4, dtype=dtype, device="cuda")[offset:offset + n]
        return v.copy_(torch.from_numpy(np.random.default_rng(seed).uniform(lo, 1.0, n)).cuda())

    lmin, lmax = 0.35, 3.8
    diag, b, x = s.diag(prec=prec), vec(1), vec(2)
    scale = diag.abs().mean()
    b *= scale
    work = torch.full((3 * n + 4,), float("nan"), dtype=dtype, device="cuda")[offset:]
    theta, delta = 0.5 * (lmax + lmin), 0.5 * (lmax - lmin)
    rho = delta / theta
    ref = x.clone()
    r = (b - s.apply(ref, prec=prec)) / diag
    d = r / theta
    for k in range(degree):
        ref = ref + d
        if k + 1 < degree:
            r = r - s.apply(d.contiguous(), prec=prec) / diag
            rho, last = 1.0 / (2.0 * theta / delta - rho), rho
            d = rho * last * d + 2.0 * rho / delta * r
    pff.pff_chebyshev_smooth(s.levels[2], prec, degree, lmin, lmax, diag, b, x, work)
    err = float((x - ref).double().norm() / ref.double().norm())
    assert err <= (1e-11 if dtype == torch.float64 else 1e-4)
