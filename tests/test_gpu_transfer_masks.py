"""p-transfers where most tiles have no prescribed node: no mask, one face, and a
single node on the tiles' edges, just inside and just outside the halo that a tile
looks at for flagged elements; and the V-cycle's forms x_f += P x_c and
r_c = P^T (b - r_f), against the Kronecker product of the 1D prolongations.

Tolerance as in test_gpu_transfer.py: 1e-13 in FP64, 2e-6 in FP32; adding to x_f or
subtracting from b rounds once more, below the same bounds.
"""
import ctypes
import itertools

import numpy as np
import pytest

from paper_2607_21150_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2607_21150_gb300 import pff  # noqa: E402
from test_gpu_transfer import matrix  # noqa: E402


class Levels:
    def __init__(self, pf, pc, n):
        self.ctx = pff.pff_create_context(inputs.phase_vector(inputs.EX3_MATRIX)[None], 2, 1e-3, 1e-2, 0.01, 2.5e5)
        self.basis = pff.pff_create_basis(self.ctx, pf, pf + 1)
        self.nf = [4] + [pf * m + 1 for m in reversed(n)]
        self.nc = [4] + [pc * m + 1 for m in reversed(n)]
        self.restr = pff.pff_create_restriction(self.ctx, (*n, 0.1, 0.1, 0.1), pf, None, int(np.prod(self.nf[1:])))
        self.op = pff.pff_create_operator(self.ctx, self.basis, self.restr)
        self.fine, self.coarse = pff.pff_create_level(self.op, pf), pff.pff_create_level(self.op, pc)
        self.P = [matrix(m, pf, pc) for m in n]

    def masks(self, mf, mc):
        dev = [None if m is None else torch.from_numpy(m.astype(np.uint8)).cuda() for m in (mf, mc)]
        pff.pff_set_dirichlet(self.op, dev[0], None)
        pff.pff_level_set_mask(self.coarse, dev[1])

    def prolong(self, xc):
        return np.einsum("fcba,zc,yb,xa->fzyx", xc, self.P[2], self.P[1], self.P[0], optimize=True)

    def restrict(self, rf):
        return np.einsum("fzyx,zc,yb,xa->fcba", rf, self.P[2], self.P[1], self.P[0], optimize=True)

    def close(self):
        for h in (self.coarse, self.fine):
            pff.pff_destroy_level(h)
        pff.pff_destroy_operator(self.op)
        pff.pff_destroy_restriction(self.restr)
        pff.pff_destroy_basis(self.basis)
        pff.pff_destroy_context(self.ctx)


def cleared(x, mask):
    return x if mask is None else np.where(mask, 0.0, x)


def dev(x, dtype):
    return torch.from_numpy(np.ascontiguousarray(x)).to("cuda", dtype)


def agree(got, want, dtype):
    err = np.linalg.norm(got.double().cpu().numpy() - want) / np.linalg.norm(want)
    assert err <= (1e-13 if dtype == torch.float64 else 2e-6)


def plain(L, rng, mf, mc, dtype):
    L.masks(mf, mc)
    prec = pff.PFF_F64 if dtype == torch.float64 else pff.PFF_F32
    xc, rf = rng.uniform(-1, 1, L.nc), rng.uniform(-1, 1, L.nf)
    if dtype == torch.float32:  # (the inputs exact in both types: a mask's slip must not hide in their rounding)
        xc, rf = xc.astype(np.float32).astype(np.float64), rf.astype(np.float32).astype(np.float64)
    xf = torch.full(L.nf, float("nan"), dtype=dtype, device="cuda")
    rc = torch.full(L.nc, float("nan"), dtype=dtype, device="cuda")
    pff.pff_prolong(L.coarse, L.fine, prec, dev(xc, dtype), xf)
    pff.pff_restrict(L.coarse, L.fine, prec, dev(rf, dtype), rc)
    agree(xf, cleared(L.prolong(cleared(xc, mc)), mf), dtype)
    agree(rc, cleared(L.restrict(cleared(rf, mf)), mc), dtype)
    for got, mask in ((xf, mf), (rc, mc)):
        if mask is not None:
            assert torch.count_nonzero(got[torch.from_numpy(mask).cuda()]).item() == 0


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("pf,pc", [(2, 1), (3, 1), (3, 2), (4, 1), (4, 2), (4, 3)])
def test_no_mask_and_single_faces(pf, pc, dtype):
    rng = np.random.default_rng(3)
    L = Levels(pf, pc, (35, 9, 3))
    plain(L, rng, None, None, dtype)
    for axis, end in itertools.product((1, 2, 3), (0, -1)):
        mf, mc = np.zeros(L.nf, bool), np.zeros(L.nc, bool)
        for m in (mf, mc):
            np.moveaxis(m, axis, 0)[end, (axis + 1) % 4] = True
        plain(L, rng, mf, mc, dtype)
    L.close()


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("pf,pc", [(2, 1), (3, 2), (4, 2)])
def test_one_node_at_a_tile_edge(pf, pc, dtype):
    rng = np.random.default_rng(4)
    tx = (32 if dtype == torch.float64 else 64) // pf
    L = Levels(pf, pc, (tx + 3, 9, 3))
    around = (-pf - 1, -pf, -1, 0, 1, pf, pf + 1)
    spots = [(pf * tx + d, pf * 4) for d in around] + [(pf * tx, pf * 4 + d) for d in around]
    for k, (i, j) in enumerate(spots + [(pf * tx, pf * 8), (pf * tx, pf * 8 + pf)]):
        mf = np.zeros(L.nf, bool)
        mf[k % 4, (pf * 2 - 1, pf, 0)[k % 3], j, i] = True
        plain(L, rng, mf, None, dtype)
    L.close()


@pytest.mark.parametrize("masked", [False, True])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("pf,pc", [(2, 1), (3, 1), (3, 2), (4, 1), (4, 2), (4, 3)])
def test_forms_of_the_cycle(pf, pc, dtype, masked):
    lib = pff.lib()
    prolong = lib["_ZN3pff16transfer_prolongEP9pff_levelS1_iPKvPvbP11CUstream_st"]
    restrict = lib["_ZN3pff17transfer_restrictEP9pff_levelS1_iPKvS3_PvP11CUstream_st"]
    vp, ci = ctypes.c_void_p, ctypes.c_int
    prolong.argtypes, restrict.argtypes = [vp, vp, ci, vp, vp, ctypes.c_bool, vp], [vp, vp, ci, vp, vp, vp, vp]
    rng = np.random.default_rng(6)
    L = Levels(pf, pc, (17, 5, 3))
    mf, mc = ((rng.random(L.nf) < 0.05), (rng.random(L.nc) < 0.05)) if masked else (None, None)
    L.masks(mf, mc)
    prec = pff.PFF_F64 if dtype == torch.float64 else pff.PFF_F32
    xc, x0, rf, b = (rng.uniform(-1, 1, n) for n in (L.nc, L.nf, L.nf, L.nf))
    d = [dev(v, dtype) for v in (xc, x0, rf, b)]
    rc = torch.full(L.nc, float("nan"), dtype=dtype, device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    assert prolong(L.coarse, L.fine, prec, d[0].data_ptr(), d[1].data_ptr(), True, st) == 0
    assert restrict(L.coarse, L.fine, prec, d[2].data_ptr(), d[3].data_ptr(), rc.data_ptr(), st) == 0
    agree(d[1], x0 + cleared(L.prolong(cleared(xc, mc)), mf), dtype)
    agree(rc, cleared(L.restrict(cleared(b - rf, mf)), mc), dtype)
    L.close()
