"""FP32-arithmetic level actions at every order and level: masked faces and
masked entries scattered over the mesh, a last element block that is not full, more element blocks
than resident thread blocks, both directions, box and mapped meshes, the
structured and the explicit node map, and the deterministic mode.

The reference is the FP64 action of the same level (1e-12 against the oracle
elsewhere).  Bounds: FP32 words and about 200 FP32 operations behind one output
stay near 1e-6 of its size, 2e-5 is allowed; BF16 words err by 2^-9 each, 4e-3.
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
from test_gpu_parity import _mapped, _two_phase  # noqa: E402

MESHES = {4: (37, 13, 7), 3: (41, 13, 10), 2: (43, 21, 10), 1: (45, 31, 15)}


def _workload(p, mapped, scattered):
    w = _mapped(3, 2, 3, p, 5, "smooth") if mapped else _two_phase(*MESHES[p], p, 5)
    if scattered:  # one entry in 40, and every entry of one plane of nodes
        n = w.mesh.ndof
        mk = np.random.default_rng(p).random(n) < 0.025
        mk.reshape(4, -1)[:, : w.mesh.nnx * w.mesh.nny] = True
        w.mask, w.dvals = mk.astype(np.uint8), np.zeros(n)
    return w


@pytest.mark.parametrize("scattered", [False, True], ids=["faces", "scattered"])
@pytest.mark.parametrize("mapped", [False, True], ids=["box", "mapped"])
@pytest.mark.parametrize("p", [1, 2, 3, 4])
def test_level_actions_follow_fp64(p, mapped, scattered):
    w = _workload(p, mapped, scattered)
    # coarser levels take their mask from whole faces, edges and corners
    levels = () if scattered else tuple(range(p - 1, 0, -1))
    for offsets in (False, True) if scattered else (False,):  # an explicit map has no coarser levels
        s = Session(w, levels=levels, f32=True, bf16=True, offsets=offsets)
        s.residual(w.z)
        for det in (False,) if offsets else (False, True):  # deterministic: structured numbering only
            pff.pff_op_set_deterministic(s.op, det)
            for pl in (p, *levels):
                x = torch.from_numpy(inputs.random_vector(4 * s.nn(pl), 3)).cuda()
                for transpose in (False, True):
                    ref = s.apply(x, p=pl, transpose=transpose)
                    for prec, tol in ((pff.PFF_F32, 2e-5), (pff.PFF_F32_BF16, 4e-3)):
                        y = s.apply(x.float(), p=pl, prec=prec, transpose=transpose).double()
                        e = ((y - ref).norm() / ref.norm()).item()
                        assert e <= tol, (pl, transpose, prec, offsets, det, e)
        assert s.status() == 0
        s.close()


@pytest.mark.parametrize("offset", [0, 1, 2, 3])
@pytest.mark.parametrize("prec", ["f64", "f32", "bf16"])
def test_output_at_any_entry(prec, offset):
    """y may start at any entry of an allocation: masked rows are x bit for bit,
    the others the aligned action up to the order of the additions."""
    w = _workload(3, True, True)
    s = Session(w, f32=True, bf16=True)
    s.residual(w.z)
    code = {"f64": pff.PFF_F64, "f32": pff.PFF_F32, "bf16": pff.PFF_F32_BF16}[prec]
    dt = torch.float64 if prec == "f64" else torch.float32
    n = w.mesh.ndof
    x = torch.from_numpy(inputs.random_vector(n, 3)).cuda().to(dt)
    ref = s.apply(x, prec=code)
    buf = torch.full((n + 8,), 7.0, dtype=dt, device="cuda")
    y = buf[offset:offset + n]
    pff.pff_jacobian_apply(s.levels[3], code, x, y, s.stream)
    m = torch.from_numpy(w.mask.astype(bool)).cuda()
    assert torch.equal(y[m], x[m])
    # at most eight additions per row, in any order
    tol = 8 * torch.finfo(dt).eps
    assert ((y - ref).norm() <= tol * ref.norm()).item()
    assert (buf[:offset] == 7.0).all() and (buf[offset + n:] == 7.0).all()
    s.close()
