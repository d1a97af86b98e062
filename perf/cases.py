"""Timed cases of the framework: what a phase-field fracture simulation has it do.

A load step evaluates the residual (with its tangent), applies the Jacobian in
FP64, double-float, FP32 or with BF16 words, smooths, transfers and takes
diagonals on the p-multigrid levels, and wraps all of it into a Newton solve;
the reaction-curve gradient adds the reverse step.  Every kind is timed alone,
the last two as whole calls.  Meshes, materials, precisions and solver settings
are those of the repository's configurations (Table 2 of the paper), on boxes of
10 um elements with a two-phase microstructure drawn on the device.

`exact` restates the method in plain torch FP64: strains by power series of the
matrix logarithm, tangents by forward-mode (transposed: reverse-mode)
differentiation of the pointwise update, quadrature by dense einsums.
"""
import math

import numpy as np
import torch

from paper_2607_21150_gb300 import pff

GPA = 1.0e3
# Rows of pff_create_context: Gc, l0, E, nu, Maxwell (on, E, nu, eta_d), Prandtl
# (on, E, nu, sigma0), hardening (H_lin, sigma_inf, beta); matrix, then particle.
NO_LAW = (0.0, 0.0, 0.0)
MATERIALS = {
    # Example 2 (compression), Example 3 (tension), Example 3 with a hardening
    # matrix, and the two inelastic phases of the reaction-curve gradient
    "ex2": ((0.01, 0.01, 1 * GPA, 0.4, 1, 1 * GPA, 0.4, 0.1 * GPA, 0, 0, 0, 0, *NO_LAW),
            (0.1, 0.01, 10 * GPA, 0.3, 0, 0, 0, 0, 0, 0, 0, 0, *NO_LAW)),
    "ex3": ((0.8, 0.005, 1 * GPA, 0.3, 1, 1 * GPA, 0.3, 0.01 * GPA, 1, 198 * GPA, 0.3, 500.0, 0.0, 500.0, 0.0),
            (8.0, 0.005, 400 * GPA, 0.25, 0, 0, 0, 0, 0, 0, 0, 0, *NO_LAW)),
    "ex3h": ((0.8, 0.005, 1 * GPA, 0.3, 1, 1 * GPA, 0.3, 0.01 * GPA, 1, 198 * GPA, 0.3, 500.0, 2 * GPA, 800.0, 40.0),
             (8.0, 0.005, 400 * GPA, 0.25, 0, 0, 0, 0, 0, 0, 0, 0, *NO_LAW)),
    "adj": ((0.8, 0.005, 1 * GPA, 0.3, 1, 1 * GPA, 0.3, 0.01 * GPA, 1, 198 * GPA, 0.3, 500.0, 0.0, 500.0, 0.0),
            (8.0, 0.005, 400 * GPA, 0.25, 1, 400 * GPA, 0.25, 1 * GPA, 1, 400 * GPA, 0.25, 5000.0, 0.0, 5000.0, 0.0)),
}
PRECS = {"f64": pff.PFF_F64, "f32": pff.PFF_F32, "df64": pff.PFF_DF64, "bf16": pff.PFF_F32_BF16}
LEVELS = {2: (2, 1), 3: (3, 1), 4: (4, 2, 1)}  # p-multigrid orders of a load step
H = 0.01  # element size, mm
SMOOTH_DEGREE, SMOOTH_LO, SMOOTH_HI = 3, 0.35, 3.8  # the solver's degree; [0.1, 1.1] of a typical lambda_max
HOST_CHUNKS = 8


def _case(kind, p, nx, ny, nz, material, at=2, **more):
    return {"kind": kind, "p": p, "nx": nx, "ny": ny, "nz": nz, "material": material, "at": at, **more}


def listed():
    def named(name, *args, **more):
        return {"name": name, **_case(*args, **more)}

    return [
        # the unit-cube example: the smallest call, all latency and launches
        named("action f64 Q2 4^3", "action", 2, 4, 4, 4, "ex3", prec="f64", transpose=False, mapped=False, bc="none"),
        # the headline: one Krylov product of the 64^3 compression test
        named("action f64 Q4 64^3", "action", 4, 64, 64, 64, "ex2", prec="f64", transpose=False, mapped=False, bc="compression"),
        # the outer product of the mixed solver, on a ragged specimen
        named("action df64 Q4 41x37x29", "action", 4, 41, 37, 29, "ex2", prec="df64", transpose=False, mapped=False, bc="compression"),
        # a level product of the adjoint solve on a curved specimen
        named("action f32 Q3 mapped transposed", "action", 3, 33, 27, 35, "ex3", prec="f32", transpose=True, mapped=True, bc="tension"),
        # the Krylov product for a caller whose vectors live in host memory
        named("host action f64 Q4 40^3", "host", 4, 40, 40, 40, "ex2", prec="f64", bc="compression"),
        # pre- or post-smoothing of the mixed solver's finest level
        named("smooth bf16 Q4 40^3", "smooth", 4, 40, 40, 40, "ex2", prec="bf16", level=4, mapped=False, bc="compression"),
        # the transfers of one V-cycle between its two finest levels
        named("transfer f32 Q4-Q2 48^3", "transfer", 4, 48, 48, 48, "ex2", prec="f32", level=2, bc="compression"),
        # the smoother's diagonal on the bar of the notched test, each Newton iteration
        named("diagonal f32 Q3 24x24x72", "diagonal", 3, 24, 24, 72, "ex3", prec="f32", level=3, mapped=False, bc="tension"),
        # residual and tangent of a load step, with the copies that the mixed solver reads
        named("residual Q4 32^3", "residual", 4, 32, 32, 32, "ex2", copies=True, mapped=False, bc="compression"),
        # the same with all three branches, hardening and yielding on a curved specimen
        named("residual Q2 24^3 hardening mapped", "residual", 2, 24, 24, 24, "ex3h", copies=True, mapped=True, bc="tension"),
        # a whole load step: the first of the 16^3 tension test, with the fastest solver settings
        named("newton Q4 16^3", "newton", 4, 16, 16, 16, "ex3", at=1, bc="tension"),
        # a whole reverse step of the reaction-curve gradient
        named("adjoint Q2 24^3", "adjoint", 2, 24, 24, 24, "adj", bc="tension"),
    ]


# Elements per direction (lowest, highest) from which a kind's drawn boxes come.
RANGES = {"action": (3, 60), "host": (6, 36), "smooth": (4, 44), "transfer": (4, 48), "diagonal": (4, 36),
          "residual": (4, 36), "newton": (5, 15), "adjoint": (6, 24)}


def draw(rng):
    kind = rng.choice(("action", "action", "action", "host", "smooth", "transfer", "diagonal", "residual", "residual",
                       "newton", "adjoint"))
    lo, hi = RANGES[kind]
    mean = rng.uniform(math.log(lo), math.log(hi))
    n = [round(math.exp(rng.uniform(max(math.log(lo), mean - 0.35), min(math.log(hi), mean + 0.35)))) for _ in range(3)]
    material, bc = rng.choice((("ex2", "compression"), ("ex3", "tension")))
    p = rng.choice((2, 3, 4))
    if kind == "action":
        return _case(kind, p, *n, material, prec=rng.choice(tuple(PRECS)), transpose=rng.random() < 0.25,
                     mapped=rng.random() < 0.25, bc=bc)
    if kind == "host":
        return _case(kind, p, *n, material, prec=rng.choice(("f64", "df64", "f32")), bc=bc)
    if kind == "smooth":
        return _case(kind, p, *n, material, prec=rng.choice(("f64", "f32", "bf16")), level=rng.choice(LEVELS[p][:2]),
                     mapped=rng.random() < 0.25, bc=bc)
    if kind == "transfer":
        return _case(kind, p, *n, material, prec=rng.choice(("f64", "f32", "f32")), level=LEVELS[p][1], bc=bc)
    if kind == "diagonal":
        return _case(kind, p, *n, material, prec=rng.choice(("f64", "f32", "f32")), level=rng.choice(LEVELS[p][:2]),
                     mapped=rng.random() < 0.25, bc=bc)
    if kind == "residual":
        return _case(kind, p, *n, rng.choice((material, "ex3h")), copies=rng.random() < 0.75, mapped=rng.random() < 0.25,
                     bc=bc)
    if kind == "newton":
        return _case(kind, p, *n, "ex3", at=1, bc="tension")
    return _case(kind, 2, *n, "adj", bc="tension")


# ---------------------------------------------------------------- inputs
class Data:
    """What a case's caller has in hand, as device tensors; the same for the same seed."""

    def __init__(self, case, seed, device):
        self.case, self.dev = case, torch.device(device)
        self.gen = torch.Generator(device=self.dev).manual_seed(1000003 * seed + 17)
        self.p, self.Q = case["p"], case["p"] + 1
        self.n = (case["nx"], case["ny"], case["nz"])
        self.L = tuple(H * m for m in self.n)
        self.nel = self.n[0] * self.n[1] * self.n[2]
        self.nq = self.nel * self.Q ** 3
        self.rows = np.array(MATERIALS[case["material"]])
        ex2 = case["material"] == "ex2"
        c0 = 8.0 / 3.0 if case["at"] == 1 else 2.0
        self.eta, self.zeta, self.dt = (1e-2 if ex2 else 1e-3), 1e-2, (0.02 if ex2 else 0.005)
        self.s_phi = self.rows[0, 2] * c0 / (2.0 * self.rows[0, 1] * self.rows[0, 0])
        self.strain = float(self.rand(()) * 0.004 + 0.002) * (-1.0 if case["bc"] == "compression" else 1.0)

    def rand(self, shape, lo=0.0, hi=1.0, dtype=torch.float64):
        return torch.rand(shape, generator=self.gen, device=self.dev, dtype=dtype) * (hi - lo) + lo

    def nodes(self, p=None):
        p = self.p if p is None else p
        return tuple(p * m + 1 for m in reversed(self.n))  # z, y, x

    def ndof(self, p=None):
        return 4 * math.prod(self.nodes(p))

    def axes(self):
        """Node coordinates per direction (x, y, z)."""
        g = torch.tensor((gll(self.p) + 1.0) * 0.5 * H, device=self.dev)[:-1]
        out = []
        for m in self.n:
            e = torch.arange(m, device=self.dev, dtype=torch.float64) * H
            out.append(torch.cat([(e[:, None] + g[None, :]).reshape(-1), e.new_tensor([m * H])]))
        return out

    def phases(self):
        """Phase per quadrature point: one sphere per cell of a jittered lattice, about 0.6 of the volume."""
        cells = [max(1, round(m / 6.4)) for m in self.n]
        centre = self.rand((3, *cells), 0.4, 0.6)
        radius = self.rand(tuple(cells), 0.48, 0.60)
        g = torch.tensor((np.polynomial.legendre.leggauss(self.Q)[0] + 1.0) * 0.5, device=self.dev)
        idx, frac = [], []
        for d in range(3):
            m = self.n[d]
            u = (torch.arange(m, device=self.dev, dtype=torch.float64)[:, None] + g[None, :]) * (cells[d] / m)
            i = u.floor().clamp(max=cells[d] - 1)
            shape = [1] * 6
            shape[2 - d], shape[5 - d] = m, self.Q  # ez, ey, ex, k, j, i
            idx.append(i.long().reshape(shape))
            frac.append((u - i).float().reshape(shape))
        centre = centre.float()
        out = torch.empty((self.n[2], self.n[1], self.n[0], self.Q, self.Q, self.Q), dtype=torch.uint8, device=self.dev)
        for z in range(0, self.n[2], 8):  # slabs bound the temporaries
            s = slice(z, z + 8)
            at = (idx[0], idx[1], idx[2][s])
            r2 = sum((([frac[0], frac[1], frac[2][s]][d]) - centre[d][at]) ** 2 for d in range(3))
            out[s] = (r2 < radius.float()[at] ** 2).to(torch.uint8)
        return out.reshape(-1)

    def mask(self, p=None):
        """Prescribed DoFs: clamped ends (tension) or frictionless platens and symmetry planes."""
        bc = self.case["bc"]
        if bc == "none":
            return None
        m = torch.zeros((4, *self.nodes(p)), dtype=torch.uint8, device=self.dev)
        if bc == "tension":
            m[0:3, 0] = 1
            m[0:3, -1] = 1
        else:
            m[2, 0] = 1
            m[2, -1] = 1
            m[0, :, :, 0] = 1
            m[1, :, 0, :] = 1
        return m.reshape(-1)

    def top(self):
        m = torch.zeros((4, *self.nodes()), dtype=torch.uint8, device=self.dev)
        m[2, -1] = 1
        return m.reshape(-1)

    def stretch(self, strain):
        """Nodal state of a homogeneous uniaxial strain."""
        z = torch.zeros((4, *self.nodes()), dtype=torch.float64, device=self.dev)
        z[2] = strain * self.axes()[2][:, None, None]
        return z

    def state(self):
        """A nodal state within a load step: uniaxial strain, fluctuations, damage up to 0.3."""
        z = self.stretch(self.strain)
        amp = 1e-3 * H / self.p
        z[:3] += self.rand((3, *self.nodes()), -amp, amp)
        z[3] = self.rand(self.nodes(), 0.0, 0.3)
        if self.case["bc"] != "none":
            fixed = self.mask().reshape(z.shape).bool()
            z[fixed] = self.stretch(self.strain)[fixed]
        return z.reshape(-1)

    def virgin(self, phase):
        """Committed history of an unloaded specimen; AT1 starts from the threshold 3 Gc / (16 l0)."""
        h = torch.zeros((15, self.nq), dtype=torch.float64, device=self.dev)
        h[0:3] = 1.0
        h[6:9] = 1.0
        if self.case["at"] == 1:
            psi_c = torch.tensor(3.0 * self.rows[:, 0] / (16.0 * self.rows[:, 1]), device=self.dev)
            h[13] = psi_c[phase.long()]
        return h

    def loaded(self, phase):
        """Committed history within a test: isochoric inelastic strains of about 0.2 %, some plastic strain,
        crack-driving energies of the order of the stored ones, earlier damage."""
        h = self.virgin(phase)
        for off in (0, 6):
            s = self.rand((6, self.nq), -2e-3, 2e-3)
            s[:3] -= s[:3].mean(0)
            h[off:off + 6] += s + 0.5 * sym_mul(s, s)
        h[12] = self.rand((self.nq,), 0.0, 0.01)
        h[13] = self.rand((self.nq,), 0.0, 0.02 if self.case["material"] == "ex2" else 3.0)
        h[14] = self.rand((self.nq,), 0.0, 0.3)
        return h

    def coords(self):
        """Nodal coordinates [3][N_n] of the smoothly curved specimen."""
        x = self.axes()
        Z, Y, X = torch.meshgrid(x[2], x[1], x[0], indexing="ij")
        X = (X, Y, Z)
        out = []
        for d in range(3):
            a, b = (d + 1) % 3, (d + 2) % 3
            out.append(X[d] + 0.15 * H * torch.sin(2 * math.pi * X[a] / self.L[a]) * torch.sin(math.pi * X[b] / self.L[b]))
        return torch.stack(out).reshape(-1)

    def vector(self, p=None, dtype=torch.float64):
        return self.rand((self.ndof(p),), -1.0, 1.0, dtype)


def sym_mul(a, b):
    """Product of symmetric matrices that commute, Voigt order 11, 22, 33, 23, 13, 12."""
    return torch.stack([a[0] * b[0] + a[5] * b[5] + a[4] * b[4], a[5] * b[5] + a[1] * b[1] + a[3] * b[3],
                        a[4] * b[4] + a[3] * b[3] + a[2] * b[2], a[5] * b[4] + a[1] * b[3] + a[3] * b[2],
                        a[0] * b[4] + a[5] * b[3] + a[4] * b[2], a[0] * b[5] + a[5] * b[1] + a[4] * b[3]])


def inputs_of(case, seed, device):
    """The Data of a case with the tensors that its kind needs."""
    d = Data(case, seed, device)
    kind = case["kind"]
    d.phase = d.phases()
    d.X = d.coords() if case.get("mapped") else None
    if kind == "newton":
        step = 0.002 * float(d.rand((), 0.7, 1.1))
        d.hist, d.z = d.virgin(d.phase), d.stretch(step).reshape(-1)
        d.dt = step / 0.4
        return d
    d.hist, d.z = d.loaded(d.phase), d.state()
    single = torch.float32 if case.get("prec") in ("f32", "bf16") else torch.float64
    if kind in ("action", "host"):
        d.x = d.vector(dtype=single)
    elif kind == "residual":
        d.x = d.vector()
    elif kind == "smooth":
        d.b, d.x0 = d.vector(case["level"], single) * 1e-2, d.vector(case["level"], single) * 1e-6
    elif kind == "transfer":
        d.xc, d.rf = d.vector(case["level"], single), d.vector(dtype=single)
    elif kind == "adjoint":
        d.hbar = d.rand((15, d.nq), -1e-3, 1e-3)
    return d


# ---------------------------------------------------------------- the framework's side
class State:
    """Handles and device buffers that a program keeps between the timed calls."""

    def __init__(self, case, seed):
        self.case = case
        d = self.d = inputs_of(case, seed, "cuda")
        kind, prec = case["kind"], case.get("prec")
        solve = kind == "newton"
        self.levels, self.solver = {}, None
        self.ctx = pff.pff_create_context(d.rows, case["at"], d.eta, d.zeta, d.dt, d.s_phi)
        self.basis = pff.pff_create_basis(self.ctx, d.p, d.Q)
        self.restr = pff.pff_create_restriction(self.ctx, (*d.n, H, H, H), d.p, None, d.ndof() // 4)
        self.op = pff.pff_create_operator(self.ctx, self.basis, self.restr)
        if d.X is not None:
            pff.pff_op_set_geometry(self.op, d.X)
        copies = solve or case.get("copies", False)
        if copies or prec == "f32" or kind in ("smooth", "diagonal"):
            pff.pff_op_enable_f32(self.op, True)
        if copies or prec == "df64" or kind == "residual":
            pff.pff_op_enable_df(self.op, True)
        if copies or prec == "bf16":
            pff.pff_op_enable_bf16(self.op, True)
        pff.pff_set_qpoint_state(self.op, d.phase, d.hist)
        mask = d.mask()
        if mask is not None:
            pff.pff_set_dirichlet(self.op, mask, d.z)
        orders = LEVELS[d.p] if kind in ("newton", "adjoint") else {d.p, case.get("level", d.p)}
        for p in orders:
            self.levels[p] = pff.pff_create_level(self.op, p)
            if p != d.p and mask is not None:
                pff.pff_level_set_mask(self.levels[p], d.mask(p))
        self.fine = self.levels[d.p]
        self.r = torch.zeros(d.ndof(), dtype=torch.float64, device="cuda")
        if kind in ("newton", "adjoint"):
            prm = pff.pff_solver_default_params(mixed=int(solve), outer_prec=pff.PFF_DF64 if solve else pff.PFF_F64,
                                                level_words=16 if solve else 32, newton_rtol=1e-9)
            self.solver = pff.pff_create_solver(self.op, [self.levels[p] for p in LEVELS[d.p]], prm)
            self.top = d.top()
            self.z = d.z.clone()
            self.hbar_prev = torch.zeros_like(d.hist)
        elif kind != "residual":
            pff.pff_residual(self.op, d.z, self.r)
        if kind in ("action", "host", "residual"):
            self.y = torch.empty_like(d.x)
        if kind == "residual":
            self.hist, self.flags = torch.empty_like(d.hist), torch.empty_like(d.phase)
        if kind == "host":
            self.xh, self.yh = d.x.cpu().pin_memory(), torch.empty(d.x.shape, dtype=d.x.dtype).pin_memory()
        if kind in ("smooth", "diagonal"):
            self.level = self.levels[case["level"]]
            single = torch.float32 if prec in ("f32", "bf16") else torch.float64
            self.diag = torch.empty(d.ndof(case["level"]), dtype=single, device="cuda")
        if kind == "smooth":
            pff.pff_assemble_diagonal(self.level, PRECS[prec], self.diag)
            self.x, self.work = d.x0.clone(), torch.empty(3 * d.x0.numel(), dtype=d.x0.dtype, device="cuda")
        if kind == "transfer":
            self.xf, self.rc = torch.empty_like(d.rf), torch.empty_like(d.xc)
        torch.cuda.synchronize()
        d.hist = d.phase = d.X = None  # the operator holds its own copies
        if kind == "adjoint":
            self.hist_prev = torch.empty((15, d.nq), dtype=torch.float64, device="cuda")
            pff.pff_get_history(self.op, 0, self.hist_prev)

    def __del__(self):
        try:
            if self.solver is not None:
                pff.pff_destroy_solver(self.solver)
            for level in self.levels.values():
                pff.pff_destroy_level(level)
            pff.pff_destroy_operator(self.op)
            pff.pff_destroy_restriction(self.restr)
            pff.pff_destroy_basis(self.basis)
            pff.pff_destroy_context(self.ctx)
        except Exception:  # a state that was never finished, or the interpreter's end
            pass


def prepare(case, seed):
    return State(case, seed)


def run(s):
    kind, d, prec = s.case["kind"], s.d, PRECS.get(s.case.get("prec"))
    if kind == "action":
        apply = pff.pff_jacobian_transpose_apply if s.case["transpose"] else pff.pff_jacobian_apply
        apply(s.fine, prec, d.x, s.y)
        return s.y
    if kind == "host":
        pff.pff_jacobian_apply_host(s.fine, prec, s.xh, s.yh, HOST_CHUNKS)
        return s.yh
    if kind == "smooth":
        s.x.copy_(d.x0)
        pff.pff_chebyshev_smooth(s.level, prec, SMOOTH_DEGREE, SMOOTH_LO, SMOOTH_HI, s.diag, d.b, s.x, s.work)
        return s.x
    if kind == "transfer":
        coarse = s.levels[s.case["level"]]
        pff.pff_restrict(coarse, s.fine, prec, d.rf, s.rc)
        pff.pff_prolong(coarse, s.fine, prec, d.xc, s.xf)
        return [s.rc, s.xf]
    if kind == "diagonal":
        pff.pff_assemble_diagonal(s.level, prec, s.diag)
        return s.diag
    if kind == "residual":  # what a line search takes from it, and the first product with its tangent
        pff.pff_residual(s.op, d.z, s.r)
        pff.pff_get_history(s.op, 1, s.hist)
        pff.pff_get_flags(s.op, s.flags)
        pff.pff_jacobian_apply(s.fine, pff.PFF_DF64, d.x, s.y)
        return [s.r, s.hist, s.flags, s.y]
    if kind == "newton":
        s.z.copy_(d.z)
        pff.pff_newton_solve(s.solver, s.z)
        return [s.z, pff.pff_reaction(s.op, s.top)[2]]
    grad = np.zeros(6 * len(d.rows))
    pff.pff_adjoint_step(s.solver, s.z, s.hist_prev, s.top, 1.0, d.hbar, s.hbar_prev, grad, rtol=1e-11)
    return [s.hbar_prev, grad]


# ---------------------------------------------------------------- work
def _sizes(case, level=None):
    p = case["p"] if level is None else level
    n = (case["nx"], case["ny"], case["nz"])
    nel = n[0] * n[1] * n[2]
    return nel, nel * (case["p"] + 1) ** 3, 4 * (p * n[0] + 1) * (p * n[1] + 1) * (p * n[2] + 1)


def _action(case, prec, level=None):
    """Bytes and flops of one product: the stored words, both vectors; the sum-factorised contractions
    (interpolation, three derivatives, their transposes) and the pointwise map."""
    nel, nq, ndof = _sizes(case, level)
    P, Q = (case["p"] if level is None else level) + 1, case["p"] + 1
    words = 70 if case.get("mapped") else 67
    word, entry = {"f64": (8, 8), "df64": (8, 8), "f32": (4, 4), "bf16": (2, 4)}[prec]
    basis = 2 * (P ** 3 * Q + P ** 2 * Q ** 2 + P * Q ** 3) + 6 * Q ** 4
    return nq * words * word + 2 * ndof * entry, nel * 2 * (4 * basis + 103 * Q ** 3)


def work(case):
    kind = case["kind"]
    nel, nq, ndof = _sizes(case)
    if kind in ("action", "host"):
        b, f = _action(case, case["prec"])
    elif kind == "smooth":  # degree products, and the vectors of the recurrence
        b, f = _action(case, case["prec"], case["level"])
        n, e = _sizes(case, case["level"])[2], 8 if case["prec"] == "f64" else 4
        b, f = SMOOTH_DEGREE * b + 4 * n * e, SMOOTH_DEGREE * (f + 8 * n)
    elif kind == "transfer":
        e, nc = 8 if case["prec"] == "f64" else 4, _sizes(case, case["level"])[2]
        P, Pc = case["p"] + 1, case["level"] + 1
        b, f = 2 * e * (ndof + nc), 2 * nel * 4 * 2 * (Pc ** 3 * P + Pc ** 2 * P ** 2 + Pc * P ** 3)
    elif kind == "diagonal":
        e, n = 8 if case["prec"] == "f64" else 4, _sizes(case, case["level"])[2]
        P, Q, terms = case["level"] + 1, case["p"] + 1, 25 if case.get("mapped") else 22
        b, f = e * (terms * nq + n), nel * terms * 2 * (P * Q ** 3 + P ** 2 * Q ** 2 + P ** 3 * Q)
    elif kind == "residual":
        # history in and out, the words and their copies out, state in and residual out, then one product;
        # the pointwise update and its tangent are about 6000 operations per point
        ab, af = _action(case, "df64")
        b = nq * (2 * 15 * 8 + 2 + 67 * (18 if case["copies"] else 16)) + 2 * 8 * ndof + ab
        f = 6000 * nq + af * 2
    else:
        # nominal counts of the whole calls: 5 residuals and 40 preconditioned products of a load step,
        # one residual and 20 of a reverse step, with 8 level products on each p-level per cycle
        ab, af = _action(case, "df64" if kind == "newton" else "f64")
        lb, lf = (sum(v) for v in zip(*(_action(case, "bf16" if kind == "newton" else "f64", p)
                                        for p in LEVELS[case["p"]][:-1])))
        res, its = (5, 40) if kind == "newton" else (1, 20)
        b, f = res * nq * 1500 + its * (ab + 8 * lb), res * 6000 * nq + its * (af + 8 * lf)
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------- the method in 64 bits
def gll(p):
    if p == 1:
        return np.array([-1.0, 1.0])
    inner = np.polynomial.legendre.Legendre.basis(p).deriv().roots()
    return np.concatenate([[-1.0], np.sort(inner.real), [1.0]])


def lagrange(nodes, x):
    """Values and derivatives [len(x)][len(nodes)] of the Lagrange basis."""
    n = len(nodes)
    B, D = np.ones((len(x), n)), np.zeros((len(x), n))
    for a in range(n):
        others = [m for m in range(n) if m != a]
        den = np.prod([nodes[a] - nodes[m] for m in others])
        for q, t in enumerate(x):
            B[q, a] = np.prod([t - nodes[m] for m in others]) / den
            D[q, a] = sum(np.prod([t - nodes[m] for m in others if m != k]) for k in others) / den
    return B, D


def mul(A, B):
    return [[A[r][0] * B[0][c] + A[r][1] * B[1][c] + A[r][2] * B[2][c] for c in range(3)] for r in range(3)]


def transposed(A):
    return [[A[c][r] for c in range(3)] for r in range(3)]


def inverse(A):
    cof = [[A[(r + 1) % 3][(c + 1) % 3] * A[(r + 2) % 3][(c + 2) % 3] - A[(r + 1) % 3][(c + 2) % 3] * A[(r + 2) % 3][(c + 1) % 3]
            for c in range(3)] for r in range(3)]
    det = A[0][0] * cof[0][0] + A[0][1] * cof[0][1] + A[0][2] * cof[0][2]
    return [[cof[c][r] / det for c in range(3)] for r in range(3)], det


def voigt(A):
    return torch.stack([A[0][0], A[1][1], A[2][2], A[1][2], A[0][2], A[0][1]])


def from_voigt(v):
    return [[v[0], v[5], v[4]], [v[5], v[1], v[3]], [v[4], v[3], v[2]]]


ONE = torch.tensor([1.0, 1.0, 1.0, 0.0, 0.0, 0.0], dtype=torch.float64)


def half_log1p(X):
    """log(I + X) / 2 of symmetric X (Voigt) by its power series, for |X| up to about 0.15."""
    one = ONE.to(X.device)[:, None]
    terms = 20
    s = one * ((-1.0) ** (terms - 1) / terms) + 0.0 * X
    for k in range(terms - 1, 0, -1):
        s = sym_mul(s, X) + one * ((-1.0) ** (k - 1) / k)
    return 0.5 * sym_mul(s, X)


def exp_sym(S):
    one = ONE.to(S.device)[:, None]
    out = one + 0.0 * S
    for k in range(14, 0, -1):
        out = sym_mul(out, S) / k + one
    return out


class Exact:
    """Residual, trial history, Jacobian products, diagonal and transfers of a case in torch FP64."""

    POINTS = 1 << 20  # quadrature points handled at a time

    def __init__(self, d):
        self.d = d
        dev = d.dev
        self.xq, self.wq = np.polynomial.legendre.leggauss(d.Q)
        self.t = {}
        for p in {d.p, d.case.get("level", d.p)}:
            B, D = lagrange(gll(p), self.xq)
            self.t[p] = torch.tensor(B, device=dev), torch.tensor(D, device=dev)
        self.table = torch.tensor(d.rows, device=dev)
        layer = d.n[0] * d.n[1] * d.Q ** 3
        self.step = max(1, self.POINTS // layer)

    def grid(self, nz):
        d = self.d
        return (nz, d.n[1], d.n[0], d.Q, d.Q, d.Q)

    def slabs(self):
        """Ranges of element layers, and the quadrature points of each."""
        d = self.d
        layer = d.n[0] * d.n[1] * d.Q ** 3
        for z in range(0, d.n[2], self.step):
            e = min(d.n[2], z + self.step)
            yield z, e, slice(z * layer, e * layer)

    def points(self, x, p, z, e):
        """Values and parent gradients [fields][points], [3][fields][points] of a nodal field on element layers."""
        d = self.d
        B, D = self.t[p]
        v = x.reshape(-1, *d.nodes(p))[:, p * z:p * e + 1].unfold(1, p + 1, p).unfold(2, p + 1, p).unfold(3, p + 1, p)

        def tensor(Tz, Ty, Tx):
            w = torch.einsum("fzyxcba,ia->fzyxcbi", v, Tx)
            w = torch.einsum("fzyxcbi,jb->fzyxcji", w, Ty)
            return torch.einsum("fzyxcji,kc->fzyxkji", w, Tz).reshape(x.numel() // math.prod(d.nodes(p)), -1)

        return tensor(B, B, B), torch.stack([tensor(B, B, D), tensor(B, D, B), tensor(D, B, B)])

    def scatter(self, out, val, grad, p, z, e):
        """The transposed of points(), added to out."""
        d = self.d
        B, D = self.t[p]
        o = out.reshape(4, *d.nodes(p))

        def tensor(v, Tz, Ty, Tx):
            v = v.reshape(4, *self.grid(e - z))
            v = torch.einsum("fzyxkji,kc->fzyxcji", v, Tz)
            v = torch.einsum("fzyxcji,jb->fzyxcbi", v, Ty)
            return torch.einsum("fzyxcbi,ia->fzyxcba", v, Tx)

        v = tensor(val, B, B, B) + tensor(grad[0], B, B, D) + tensor(grad[1], B, D, B) + tensor(grad[2], D, B, B)
        self.add_nodes(o, v, p, z, e)

    def add_nodes(self, o, v, p, z, e):
        d = self.d
        for c in range(p + 1):
            for b in range(p + 1):
                for a in range(p + 1):
                    o[:, p * z + c:p * (e - 1) + c + 1:p, b:p * (d.n[1] - 1) + b + 1:p,
                      a:p * (d.n[0] - 1) + a + 1:p] += v[..., c, b, a]

    def geometry(self, z, e):
        """d xi / dX [3][3] and w det J of the slab's points."""
        d = self.d
        w = torch.tensor(np.einsum("k,j,i->kji", self.wq, self.wq, self.wq), device=d.dev).expand(self.grid(e - z)).reshape(-1)
        if d.X is None:
            return None, w * (H / 2) ** 3
        _, g = self.points(d.X, d.p, z, e)  # [al][f]
        G, det = inverse([[g[al][f] for al in range(3)] for f in range(3)])
        return G, w * det

    def physical(self, G, g):
        if G is None:
            return g * (2.0 / H)
        return torch.stack([sum(G[al][A] * g[al] for al in range(3)) for A in range(3)])

    def parent(self, G, g):
        if G is None:
            return g * (2.0 / H)
        return torch.stack([sum(G[al][A] * g[A] for A in range(3)) for al in range(3)])

    def update(self, q, gu, phi, gphi, want_history=False):
        """Box 1 of the paper in series with the fracture element at the points q: stress P [9], s_phi L,
        phase-field flux [3]; with want_history the trial history too."""
        d = self.d
        rows = self.table[d.phase[q].long()].T
        h = d.hist[:, q]
        Gc, l0 = rows[0], rows[1]
        c0 = 8.0 / 3.0 if d.case["at"] == 1 else 2.0
        g, gp = (1.0 - phi) ** 2 + d.eta, -2.0 * (1.0 - phi)
        F = [[gu[3 * r + c] + (1.0 if r == c else 0.0) for c in range(3)] for r in range(3)]
        U = [[gu[3 * r + c] for c in range(3)] for r in range(3)]
        Fi, _ = inverse(F)
        tr = U[0][0] + U[1][1] + U[2][2]
        UU = mul(U, U)
        cof = U[0][0] * (U[1][1] * U[2][2] - U[1][2] * U[2][1]) - U[0][1] * (U[1][0] * U[2][2] - U[1][2] * U[2][0]) \
            + U[0][2] * (U[1][0] * U[2][1] - U[1][1] * U[2][0])
        theta = torch.log1p(tr + 0.5 * (tr * tr - UU[0][0] - UU[1][1] - UU[2][2]) + cof)
        GG = voigt([[U[r][c] + U[c][r] + U[r][0] * U[c][0] + U[r][1] * U[c][1] + U[r][2] * U[c][2] for c in range(3)]
                    for r in range(3)])
        tau, psi, kappa = 0.0, 0.0, 0.0
        one = ONE.to(d.dev)[:, None]
        new, gained = [h[0:6], h[6:12]], torch.zeros_like(phi)
        for br, off in ((0, 2), (1, 5), (2, 9)):
            on = torch.ones_like(phi) if br == 0 else rows[off - 1]
            E, nu = torch.where(on > 0, rows[off], 1.0), torch.where(on > 0, rows[off + 1], 0.0)
            mu = on * E / (2.0 * (1.0 + nu))
            kappa = kappa + on * E / (3.0 * (1.0 - 2.0 * nu))
            X = GG
            if br:
                C = from_voigt(h[6 * (br - 1):6 * br] - one)
                X = X + voigt(mul(mul(F, C), transposed(F)))
            ed = half_log1p(X)
            ed = ed - one * ((ed[0] + ed[1] + ed[2]) / 3.0)
            s2 = (ed[:3] ** 2).sum(0) + 2.0 * (ed[3:] ** 2).sum(0)
            a = torch.ones_like(phi)
            if br == 1:
                a = 1.0 / (1.0 + torch.where(on > 0, mu * d.dt / torch.where(on > 0, rows[7], 1.0), 0.0) * g)
            elif br == 2:
                sig0, Hl, sinf, beta = rows[11], rows[12], rows[13], rows[14]
                mu1 = torch.where(on > 0, mu, 1.0)
                qtr = 2.0 * mu1 * torch.sqrt(1.5 * s2)
                ep = h[12]

                def sig(e):
                    return sig0 + Hl * e + (sinf - sig0) * (1.0 - torch.exp(-beta * e))

                def slope(e):
                    return Hl + (sinf - sig0) * beta * torch.exp(-beta * e)

                yields = (g * qtr - sig(ep) > 0.0) & (on > 0)
                dg = torch.zeros_like(phi)
                for _ in range(8):
                    dg = dg + (g * qtr - 3.0 * g * mu1 * dg - sig(ep + dg)) / (3.0 * g * mu1 + slope(ep + dg))
                gained = torch.where(yields, dg, 0.0)
                a = torch.where(yields, 1.0 - 3.0 * mu1 * dg / qtr, 1.0)
            tau = tau + 2.0 * mu * a * ed
            psi = psi + mu * a * a * s2
            if br and want_history:
                b = from_voigt(exp_sym(2.0 * (a * ed + one * (theta / 3.0))))
                c = voigt(mul(mul(Fi, b), transposed(Fi)))
                new[br - 1] = torch.where(on > 0, c, new[br - 1])
        tens = theta >= 0.0
        tv = kappa * theta
        T = from_voigt(g * tau + one * torch.where(tens, g * tv, tv))
        psi = torch.where(tens, psi + 0.5 * kappa * theta * theta, psi)
        Hh = torch.where(psi > h[13], psi, h[13])
        dalpha = 1.0 if d.case["at"] == 1 else 2.0 * phi
        Lphi = gp * Hh + Gc / (c0 * l0) * dalpha + d.zeta * (phi - h[14]) / d.dt
        P = mul(T, transposed(Fi))
        flux = d.s_phi * 2.0 * Gc * l0 / c0 * gphi
        out = (torch.stack([P[r][c] for r in range(3) for c in range(3)]), d.s_phi * Lphi, flux)
        if want_history:
            return (*out, torch.cat([new[0], new[1], (h[12] + gained)[None], Hh[None], phi[None]]))
        return out

    def at(self, x, z, e, G, p):
        """grad u [9], phi, grad phi [3] of a nodal field at the slab's points."""
        v, g = self.points(x, p, z, e)
        g = self.physical(G, g)
        return torch.stack([g[A][r] for r in range(3) for A in range(3)]), v[3], torch.stack([g[A][3] for A in range(3)])

    def back(self, out, P, Lphi, flux, z, e, G, w, p):
        g = torch.stack([torch.stack([P[3 * r + A] for r in range(3)] + [flux[A]]) for A in range(3)])
        v = torch.zeros_like(g[0])
        v[3] = w * Lphi
        self.scatter(out, v, self.parent(G, g) * w, p, z, e)

    def residual(self):
        d = self.d
        r, hist = torch.zeros(d.ndof(), dtype=torch.float64, device=d.dev), []
        for z, e, q in self.slabs():
            G, w = self.geometry(z, e)
            *f, h = self.update(q, *self.at(d.z, z, e, G, d.p), want_history=True)
            self.back(r, *f, z, e, G, w, d.p)
            hist.append(h)
        fixed = d.mask()
        return torch.where(fixed.bool(), 0.0, r) if fixed is not None else r, torch.cat(hist, 1)

    def product(self, x, p, transpose=False):
        """J x or J^T x on the level of order p, prescribed rows and columns those of the identity."""
        d = self.d
        x = x.double()
        fixed = d.mask(p)
        free = x if fixed is None else torch.where(fixed.bool(), 0.0, x)
        y = torch.zeros_like(x)
        for z, e, q in self.slabs():
            G, w = self.geometry(z, e)
            base, dx = self.at(d.z, z, e, G, d.p), self.at(free, z, e, G, p)
            if transpose:
                f = torch.func.vjp(lambda *a: self.update(q, *a), *base)[1](dx)
            else:
                f = torch.func.jvp(lambda *a: self.update(q, *a), base, dx)[1]
            self.back(y, *f, z, e, G, w, p)
        return y if fixed is None else torch.where(fixed.bool(), x, y)

    def diagonal(self, p):
        d = self.d
        B, D = self.t[p]
        out = torch.zeros((4, *d.nodes(p)), dtype=torch.float64, device=d.dev)
        for z, e, q in self.slabs():
            G, w = self.geometry(z, e)
            base = self.at(d.z, z, e, G, d.p)
            n = base[1].numel()
            A = torch.zeros((4, 3, 3, n), dtype=torch.float64, device=d.dev)
            for f in range(4):
                for be in range(3):
                    t = [torch.zeros_like(b) for b in base]
                    t[0 if f < 3 else 2][3 * f + be if f < 3 else be] = 1.0
                    o = torch.func.jvp(lambda *a: self.update(q, *a), base, tuple(t))[1]
                    A[f, :, be] = o[0][3 * f:3 * f + 3] if f < 3 else o[2]
            t = (torch.zeros_like(base[0]), torch.ones_like(base[1]), torch.zeros_like(base[2]))
            value = torch.func.jvp(lambda *a: self.update(q, *a), base, t)[1][1]
            if G is None:
                A = A * (2.0 / H) ** 2
            else:
                g = torch.stack([torch.stack(r) for r in G])
                A = torch.einsum("aAn,fABn,bBn->fabn", g, A, g)
            A = (A * w).reshape(4, 3, 3, *self.grid(e - z))
            v = torch.zeros((4, e - z, d.n[1], d.n[0], p + 1, p + 1, p + 1), dtype=torch.float64, device=d.dev)
            for al in range(3):
                for be in range(3):
                    M = [(D if al == k else B) * (D if be == k else B) for k in range(3)]
                    v += torch.einsum("fzyxkji,kc,jb,ia->fzyxcba", A[:, al, be], M[2], M[1], M[0])
            v[3] += torch.einsum("zyxkji,kc,jb,ia->zyxcba", (w * value).reshape(self.grid(e - z)), B * B, B * B, B * B)
            self.add_nodes(out, v, p, z, e)
        fixed = d.mask(p)
        out = out.reshape(-1)
        return out if fixed is None else torch.where(fixed.bool(), 1.0, out)

    def smooth(self, p):
        """Saad, Algorithm 12.1, preconditioned by the diagonal."""
        d = self.d
        diag, b, x = self.diagonal(p), d.b.double(), d.x0.double()
        theta, delta = 0.5 * (SMOOTH_HI + SMOOTH_LO), 0.5 * (SMOOTH_HI - SMOOTH_LO)
        sigma = theta / delta
        rho = 1.0 / sigma
        r = (b - self.product(x, p)) / diag
        dx = r / theta
        for _ in range(SMOOTH_DEGREE - 1):
            x = x + dx
            r = r - self.product(dx, p) / diag
            rho, last = 1.0 / (2.0 * sigma - rho), rho
            dx = rho * last * dx + 2.0 * rho / delta * r
        return x + dx

    def transfer(self, pc):
        d = self.d
        I1 = torch.tensor(lagrange(gll(pc), gll(d.p))[0], device=d.dev)
        P = []
        for m in d.n:  # 1D prolongation of the whole direction
            T = torch.zeros((d.p * m + 1, pc * m + 1), dtype=torch.float64, device=d.dev)
            for e in range(m):
                T[d.p * e:d.p * e + d.p + 1, pc * e:pc * e + pc + 1] = I1
            P.append(T)
        mf, mc = d.mask(), d.mask(pc)
        xc, rf = d.xc.double(), d.rf.double()
        if mf is not None:
            xc, rf = torch.where(mc.bool(), 0.0, xc), torch.where(mf.bool(), 0.0, rf)
        xf = torch.einsum("fcba,zc,yb,xa->fzyx", xc.reshape(4, *d.nodes(pc)), P[2], P[1], P[0]).reshape(-1)
        rc = torch.einsum("fzyx,zc,yb,xa->fcba", rf.reshape(4, *d.nodes()), P[2], P[1], P[0]).reshape(-1)
        if mf is not None:
            xf, rc = torch.where(mf.bool(), 0.0, xf), torch.where(mc.bool(), 0.0, rc)
        return [rc, xf]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("newton", "adjoint"):
        return None
    d = inputs_of(case, seed, "cuda" if torch.cuda.is_available() else "cpu")
    if kind == "transfer":
        return Exact(d).transfer(case["level"])
    if kind == "action" and d.nq > 16_000_000 and case["transpose"]:
        return None
    if kind in ("smooth", "diagonal") and d.nq > 9_000_000:
        return None
    x = Exact(d)
    if kind in ("action", "host"):
        return x.product(d.x, d.p, case.get("transpose", False))
    if kind == "smooth":
        return x.smooth(case["level"])
    if kind == "diagonal":
        return x.diagonal(case["level"])
    r, hist = x.residual()
    return [r, hist, None, x.product(d.x, d.p)]
