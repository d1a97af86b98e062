"""The deterministic mode across changes of the Dirichlet data: with the mask taken
away and set again the element values keep their buffer, the action is the
oracle's of the same data (the parity bar 1e-12) and reruns give the same bits."""
import pytest

from paper_2607_21150_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2607_21150_gb300 import pff  # noqa: E402
from paper_2607_21150_gb300.session import Session  # noqa: E402
from test_gpu_solver import _box, np_, rel  # noqa: E402


def test_mask_removed_and_set_again(orc):
    w = _box(3, 2, 4, 2, 5)
    s = Session(w)
    pff.pff_op_set_deterministic(s.op, True)
    s.residual(torch.from_numpy(w.z.ravel()).cuda())
    v = inputs.random_vector(w.mesh.ndof, 8)
    x = torch.from_numpy(v).cuda()
    for mask in (None, w.mask):
        if mask is None:
            pff.pff_set_dirichlet(s.op, None, None)
        else:
            pff.pff_set_dirichlet(s.op, s.mask, s.dvals)
        K = orc.assemble(w, mask=mask, dvals=None if mask is None else w.dvals)["K"]
        y = s.apply(x)
        assert torch.equal(s.apply(x), y)
        assert rel(np_(y), K @ v) <= 1e-12
    s.close()
