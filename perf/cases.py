"""The workloads that this library is timed on: single solves from a few
thousand to eight million cells (FP64 and mixed, DIC and diagonal, natural and
random cell numbering), the differentiable solve, batched solves, GAMG, PBiCG,
the coefficient assembly with its reverse mode, the finite-volume operators
around the solve, and the matrix-vector product.

Inputs follow the recipe of the synthetic hex blocks (jittered points, random
cell renumbering, faces in upper-triangular order, log-normal or unit
diffusivity, one Dirichlet patch), generated here on the GPU so that a new
state takes milliseconds.  Solves run to residuals at which x is determined to
better than the rounding of its last iterations, so that two correct FP64
programs agree on it.
"""
import math

import torch

from paper_2512_22215_gb300 import (F64, MIXED, PRECOND_DIAGONAL, PRECOND_DIC, PRECOND_DILU, BatchSolve, GamgSolver,
                                    LduMesh, SolverControls, assemble_laplacian, pressure_solve)

PRECOND = {"diagonal": PRECOND_DIAGONAL, "dic": PRECOND_DIC, "dilu": PRECOND_DILU}
PRECISION = {"f64": F64, "mixed": MIXED}


def _case(name, kind, nx, ny=None, nz=None, permute=True, **kw):
    return dict(name=name, kind=kind, nx=nx, ny=ny or nx, nz=nz or nx, permute=permute, **kw)


def listed():
    return [
        # a small pressure system in natural cell order (the 16^3 configuration)
        _case("solve_16_f64_dic", "solve", 16, permute=False, jitter=0.0, lognormal=False, precision="f64",
              precond="dic", tol=1e-10),
        # learning a diffusivity: assembly, solve, loss and the gradients back to it (the 64^3 adjoint configuration)
        _case("adjoint_64", "adjoint", 64, tol=1e-12),
        # the 2.1M-cell FP64 configuration with its two preconditioners
        _case("solve_128_f64_dic", "solve", 128, precision="f64", precond="dic", tol=1e-11),
        _case("solve_128_f64_diagonal", "solve", 128, precision="f64", precond="diagonal", tol=1e-11),
        # the 8M-cell production solve (mixed precision)
        _case("solve_200_mixed_dic", "solve", 200, precision="mixed", precond="dic", tol=1e-11),
        # many small independent systems of uneven sizes in one launch
        dict(name="batch_32_f64_dic", kind="batch", n_sys=32, cells_lo=1e4, cells_hi=5e5, sizes_seed=5,
             precision="f64", precond="dic", tol=1e-11),
        # new coefficients every outer iteration, and their reverse mode
        _case("assembly_200", "assembly", 200),
        # weights, gradient, right-hand side, flux and divergence of a pressure correction
        _case("pressure_ops_150x131x113", "pressure_ops", 150, 131, 113),
        # lduMatrix::Amul on the caller's arrays (a caller's own Krylov loop)
        _case("amul_200_f64", "amul", 200, dtype="f64"),
        # the multigrid pressure solver: face-area pairing with Richardson, coefficient pairing with Gauss-Seidel
        _case("gamg_64_richardson", "gamg", 64, smoother=0, weights="area", tol=1e-11),
        _case("gamg_128_gauss_seidel", "gamg", 128, smoother=1, weights="coefficient", tol=1e-11),
        # a momentum-like asymmetric system (upwind convection-diffusion)
        _case("pbicg_128_dilu", "pbicg", 128, precond="dilu", tol=1e-11),
    ]


def _side(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _box(rng, lo, hi):
    """Three sides near a common one, ragged."""
    n = _side(rng, lo, hi)
    return [max(2, min(hi, int(round(n * rng.uniform(0.8, 1.25))))) for _ in range(3)]


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "adjoint", "batch", "assembly", "pressure_ops", "amul", "gamg", "pbicg"])
    if kind == "batch":
        lo = _side(rng, 4e3, 4e4)
        return dict(kind=kind, n_sys=rng.randint(6, 32), cells_lo=float(lo), cells_hi=float(rng.randint(lo, 500000)),
                    sizes_seed=rng.randint(0, 1 << 20), precision=rng.choice(["f64", "mixed"]), precond="dic", tol=1e-11)
    hi = {"solve": 160, "adjoint": 80, "assembly": 200, "pressure_ops": 160, "amul": 200, "gamg": 112, "pbicg": 128}[kind]
    nx, ny, nz = _box(rng, 12, hi)
    c = dict(kind=kind, nx=nx, ny=ny, nz=nz, permute=rng.random() < 0.75)
    if kind == "solve":
        # in natural order the number of DIC levels grows with the side, so those stay smaller
        if not c["permute"]:
            c.update(nx=min(nx, 72), ny=min(ny, 72), nz=min(nz, 72))
        c.update(precision=rng.choice(["f64", "mixed"]), precond=rng.choice(["dic", "dic", "diagonal"]), tol=1e-11)
    elif kind == "adjoint":
        if not c["permute"]:
            c.update(nx=min(nx, 48), ny=min(ny, 48), nz=min(nz, 48))
        c.update(tol=1e-12)
    elif kind == "amul":
        c.update(dtype=rng.choice(["f64", "f32"]))
    elif kind == "gamg":
        c.update(rng.choice([dict(smoother=0, weights="area"), dict(smoother=1, weights="coefficient")]), tol=1e-11)
    elif kind == "pbicg":
        c.update(precond=rng.choice(["dilu", "diagonal"]), tol=1e-11)
    return c


# ------------------------------------------------------------- the meshes ---
def _dot(a, b):
    return (a * b).sum(-1)


def _quads(p0, p1, p2, p3):
    """Area vectors and centres of quads, triangulated about their mean point."""
    mid = (p0 + p1 + p2 + p3) * 0.25
    corners = (p0, p1, p2, p3)
    s, wsum, csum = 0.0, 0.0, 0.0
    for k in range(4):
        a, b = corners[k], corners[(k + 1) % 4]
        at = 0.5 * torch.cross(b - a, mid - a, dim=-1)
        mag = at.norm(dim=-1, keepdim=True)
        s, wsum, csum = s + at, wsum + mag, csum + mag * (a + b + mid) / 3.0
    return s, csum / wsum


class _Block:
    """A jittered hex block on the GPU: LDU addressing, geometry, diffusivity,
    and (for the solves) the matrix of the pressure equation."""

    def __init__(self, nx, ny, nz, permute, seed, jitter=0.2, lognormal=True):
        g = torch.Generator(device="cuda").manual_seed(seed)
        kw = dict(dtype=torch.float64, device="cuda")
        lin = [torch.linspace(0.0, 1.0, n + 1, **kw) for n in (nz, ny, nx)]
        P = torch.stack(torch.meshgrid(*lin, indexing="ij")[::-1], dim=-1)      # [k, j, i, xyz]
        if jitter > 0.0 and min(nx, ny, nz) > 1:
            h = torch.tensor([1.0 / nx, 1.0 / ny, 1.0 / nz], **kw)
            d = torch.rand(nz - 1, ny - 1, nx - 1, 3, generator=g, **kw)
            P[1:-1, 1:-1, 1:-1] += (2.0 * d - 1.0) * jitter * h
        S, C = [None] * 3, [None] * 3                                            # faces normal to x, y, z
        S[0], C[0] = _quads(P[:-1, :-1], P[:-1, 1:], P[1:, 1:], P[1:, :-1])
        S[1], C[1] = _quads(P[:-1, :, :-1], P[1:, :, :-1], P[1:, :, 1:], P[:-1, :, 1:])
        S[2], C[2] = _quads(P[:, :-1, :-1], P[:, :-1, 1:], P[:, 1:, 1:], P[:, 1:, :-1])
        ax = (2, 1, 0)                                                           # array axis of x, y, z
        n_of = (nx, ny, nz)

        def cut(t, d, a, b):
            return t.narrow(ax[d], a, b - a)

        sides = [(sg, cut(S[d], d, o, o + n_of[d]), cut(C[d], d, o, o + n_of[d]))
                 for d in range(3) for sg, o in ((-1.0, 0), (1.0, 1))]
        mid = sum(c for _, _, c in sides) / 6.0
        vol, cen = 0.0, 0.0
        for sg, s, c in sides:
            v = sg * _dot(s, c - mid) / 3.0
            vol, cen = vol + v, cen + v[..., None] * (0.75 * c + 0.25 * mid)
        cen = cen / vol[..., None]
        N = nx * ny * nz
        ids = torch.randperm(N, generator=g, device="cuda") if permute else torch.arange(N, device="cuda")
        ids3 = ids.view(nz, ny, nx)
        lo, up, sf, cf, a_, b_ = [], [], [], [], [], []
        for d in range(3):
            m = n_of[d] - 1
            a, b = cut(ids3, d, 0, m).reshape(-1), cut(ids3, d, 1, m + 1).reshape(-1)
            lo.append(torch.minimum(a, b))
            up.append(torch.maximum(a, b))
            sg = torch.where(a < b, 1.0, -1.0).to(torch.float64)[:, None]
            sf.append(cut(S[d], d, 1, m + 1).reshape(-1, 3) * sg)
            cf.append(cut(C[d], d, 1, m + 1).reshape(-1, 3))
        lo, up = torch.cat(lo), torch.cat(up)
        order = torch.argsort(lo * N + up)
        self.order = order
        self.n = N
        self.lower, self.upper_addr = lo[order].int(), up[order].int()
        self.sf, self.cf = torch.cat(sf)[order], torch.cat(cf)[order]
        self.c = torch.empty(N, 3, **kw)
        self.c[ids] = cen.reshape(-1, 3)
        self.v = torch.empty(N, **kw)
        self.v[ids] = vol.reshape(-1)
        bc, bs, bf, bt = [], [], [], []
        for d in range(3):
            for o, sg in ((0, -1.0), (n_of[d], 1.0)):
                cell = cut(ids3, d, 0, 1) if o == 0 else cut(ids3, d, o - 1, o)
                bc.append(cell.reshape(-1))
                bs.append(sg * cut(S[d], d, o, o + 1).reshape(-1, 3))
                bf.append(cut(C[d], d, o, o + 1).reshape(-1, 3))
                bt.append(torch.full((cell.numel(),), 1 if d == 0 and o else 0, dtype=torch.int8, device="cuda"))
        self.bcell, self.btype = torch.cat(bc).int(), torch.cat(bt)
        self.bsf, self.bcf = torch.cat(bs).contiguous(), torch.cat(bf).contiguous()
        F, B = self.lower.numel(), self.bcell.numel()
        if lognormal:
            self.gamma = torch.randn(F, generator=g, **kw).exp()
            self.bgamma = torch.randn(B, generator=g, **kw).exp()
        else:
            self.gamma, self.bgamma = torch.ones(F, **kw), torch.ones(B, **kw)
        self.b = torch.randn(N, generator=g, **kw)
        self.gen, self.ids, self.shape, self.kw = g, ids, (nz, ny, nx), kw
        self.splits = [cut(ids3, d, 0, n_of[d] - 1).shape for d in range(3)]

    def coeffs(self):
        """|S|/max(n.d, 0.05 |d|) of the internal faces and the Dirichlet ones (0 elsewhere)."""
        d = self.c[self.upper_addr.long()] - self.c[self.lower.long()]
        bd = self.bcf - self.c[self.bcell.long()]
        f = lambda s, d: s.norm(dim=1) / torch.maximum(_dot(s, d) / s.norm(dim=1), 0.05 * d.norm(dim=1))  # noqa: E731
        return f(self.sf, d), torch.where(self.btype == 1, f(self.bsf, bd), torch.zeros_like(self.bgamma))

    def structured(self, face):
        """A face array back in the block's directions (x, y, z faces as 3-D arrays)."""
        t = torch.empty_like(face)
        t[self.order] = face
        return [v.view(s) for v, s in zip(t.split([math.prod(s) for s in self.splits]), self.splits)]

    def cell_sum(self, low, high, bval):
        """Per-cell sums in a fixed order: low/high, what a face adds to the cell below and above it."""
        t = torch.zeros(self.shape, **self.kw)
        for d, (lo, hi) in enumerate(zip(low, high)):
            n = t.shape[2 - d]
            t.narrow(2 - d, 0, n - 1).add_(lo)
            t.narrow(2 - d, 1, n - 1).add_(hi)
        r = torch.empty(self.n, **self.kw)
        r[self.ids] = t.reshape(-1)
        fixed = self.btype == 1                     # one patch: one such face a cell
        cell = self.bcell[fixed].long()
        r[cell] = r[cell] + bval[fixed]
        return r

    def matrix(self):
        """(diag, upper) of the pressure equation."""
        k, kb = self.coeffs()
        a = self.gamma * k
        s = self.structured(a)
        return self.cell_sum(s, s, self.bgamma * kb), -a

    def convection(self, pe=2.0):
        """(diag, lower, upper): the laplacian with first-order upwind convection of a random flux, the diagonal
        raised to the row sums over the relaxation factor 0.7."""
        k, kb = self.coeffs()
        a = self.gamma * k
        phi = pe * torch.randn(a.numel(), generator=self.gen, **self.kw) * a.mean()
        lower, upper = -a - phi.clamp(min=0.0), -a - (-phi).clamp(min=0.0)
        diag = torch.zeros(self.n, **self.kw)
        # the cell below a face in its direction is its owner or its neighbour: pick that side's coefficient
        sg = []
        ids3 = self.ids.view(self.shape)
        for d in range(3):
            n = ids3.shape[2 - d]
            sg.append(ids3.narrow(2 - d, 0, n - 1) < ids3.narrow(2 - d, 1, n - 1))
        ls, us = self.structured(-lower), self.structured(-upper)
        low = [torch.where(o, u, l) for o, l, u in zip(sg, ls, us)]
        high = [torch.where(o, l, u) for o, l, u in zip(sg, ls, us)]
        diag = self.cell_sum(low, high, self.bgamma * kb) / 0.7
        return diag, lower, upper

    def handle(self, asymmetric=False):
        return LduMesh(self.lower, self.upper_addr, self.n, centres=self.c, asymmetric=asymmetric)


def _block(case, seed):
    return _Block(case["nx"], case["ny"], case["nz"], case["permute"], seed, case.get("jitter", 0.2),
                  case.get("lognormal", True))


def _batch_blocks(case, seed):
    g = torch.Generator().manual_seed(case["sizes_seed"])
    lo, hi = math.log(case["cells_lo"]), math.log(case["cells_hi"])
    cells = torch.exp(lo + (hi - lo) * torch.rand(case["n_sys"], generator=g, dtype=torch.float64)).tolist()
    sides = [max(2, round(v ** (1.0 / 3.0))) for v in cells]
    return [_Block(n, n, n, True, 1000 * seed + k) for k, n in enumerate(sides)]


# ---------------------------------------------------------- prepare and run ---
def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if "precond" in case:
        st["ctl"] = SolverControls(precond=PRECOND[case["precond"]], precision=PRECISION[case.get("precision", "f64")],
                                   tolerance=case["tol"])
    if kind == "batch":
        blocks = _batch_blocks(case, seed)
        meshes = [B.handle() for B in blocks]
        mats = [B.matrix() for B in blocks]
        st["x"] = [torch.zeros_like(B.b) for B in blocks]
        st["batch"] = BatchSolve(meshes, [d for d, _ in mats], [u for _, u in mats], [B.b for B in blocks], st["x"],
                                 st["ctl"], autotune=False)
        return st
    B = _block(case, seed)
    st["B"], st["mesh"] = B, B.handle(asymmetric=kind == "pbicg")
    if kind == "solve":
        st["diag"], st["upper"] = B.matrix()
    elif kind == "pbicg":
        st["diag"], st["lower"], st["upper"] = B.convection()
    elif kind == "gamg":
        st["diag"], st["upper"] = B.matrix()
        weight = B.sf.norm(dim=1) if case["weights"] == "area" else st["upper"].abs()
        st["gamg"] = GamgSolver(st["mesh"], weight, smoother=case["smoother"])
        st["ctl"] = SolverControls(tolerance=case["tol"], max_iter=1000)
    elif kind == "amul":
        st["diag"], st["upper"] = B.matrix()
        st["x"] = B.b
        if case["dtype"] == "f32":
            st["diag"], st["upper"], st["x"] = st["diag"].float(), st["upper"].float(), B.b.float()
        st["y"] = torch.empty_like(st["x"])
    elif kind == "pressure_ops":
        st["diag"], st["upper"] = B.matrix()
        st["phi"] = torch.randn(B.lower.numel(), generator=B.gen, **B.kw) * B.sf.norm(dim=1)
        st["bphi"] = torch.randn(B.bcell.numel(), generator=B.gen, **B.kw) * B.bsf.norm(dim=1)
        st["p"] = torch.randn(B.n, generator=B.gen, **B.kw)
    elif kind == "assembly":
        st["gu"] = torch.randn(B.lower.numel(), generator=B.gen, **B.kw)
        st["gd"] = torch.randn(B.n, generator=B.gen, **B.kw)
        B.gamma.requires_grad_(True)
        B.bgamma.requires_grad_(True)
    elif kind == "adjoint":
        st["xt"] = torch.randn(B.n, generator=B.gen, **B.kw)
        for t in (B.gamma, B.bgamma, B.b):
            t.requires_grad_(True)
        st["ctl"] = SolverControls(tolerance=case["tol"])
    B.order = B.ids = None                          # the generator's own
    return st


def run(st):
    kind = st["case"]["kind"]
    if kind == "batch":
        torch._foreach_zero_(st["x"])
        st["batch"].run()
        return st["x"]
    B, M = st["B"], st["mesh"]
    if kind == "solve":
        x, p = M.solve(st["diag"], st["upper"], B.b, None, st["ctl"])
        return {"x": x, "converged": p["converged"]}
    if kind == "pbicg":
        x, p = M.pbicg_solve(st["diag"], st["lower"], st["upper"], B.b, None, st["ctl"])
        return {"x": x, "converged": p["converged"]}
    if kind == "gamg":
        x, p = st["gamg"].solve(st["diag"], st["upper"], B.b, None, st["ctl"])
        return {"x": x, "converged": p["converged"]}
    if kind == "amul":
        return M.amul(st["diag"], st["upper"], st["x"], st["y"])
    if kind == "pressure_ops":
        w = M.fv_weights(B.sf, B.cf, B.c)
        grad = M.fv_grad(B.sf, w, B.v, st["p"], B.bcell, B.bsf, B.btype)
        corr, b = M.pressure_rhs(B.sf, B.c, w, B.gamma, grad, st["phi"], B.bcell, st["bphi"])
        phi, bphi = M.pressure_flux(st["upper"], corr, st["p"], st["phi"], B.c, B.bcell, B.bsf, B.bcf, B.bgamma,
                                    B.btype, st["bphi"])
        div = M.fv_div(phi, B.bcell, bphi)
        return {"w": w, "grad": grad, "corr": corr, "b": b, "phi": phi, "bphi": bphi, "div": div}
    upper, diag = assemble_laplacian(M, B.gamma, B.bgamma, B.sf, B.c, B.bcell, B.bsf, B.bcf, B.btype)
    if kind == "assembly":
        gg, gb = torch.autograd.grad([upper, diag], [B.gamma, B.bgamma], [st["gu"], st["gd"]])
        return {"upper": upper.detach(), "diag": diag.detach(), "dgamma": gg, "dbgamma": gb}
    x = pressure_solve(M, upper, diag, B.b, st["ctl"])
    loss = 0.5 * ((x - st["xt"]) ** 2).sum()
    gg, gb, g = torch.autograd.grad(loss, [B.gamma, B.bgamma, B.b])
    return {"x": x.detach(), "dgamma": gg, "dbgamma": gb, "db": g}


# ------------------------------------------------------------------- work ---
def _counts(nx, ny, nz):
    n = nx * ny * nz
    return n, 3 * n - nx * ny - ny * nz - nx * nz, 2 * (nx * ny + ny * nz + nx * nz)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        w = {"bytes": 0.0, "flops": 0.0}
        g = torch.Generator().manual_seed(case["sizes_seed"])
        lo, hi = math.log(case["cells_lo"]), math.log(case["cells_hi"])
        for v in torch.exp(lo + (hi - lo) * torch.rand(case["n_sys"], generator=g, dtype=torch.float64)).tolist():
            s = max(2, round(v ** (1.0 / 3.0)))
            one = work(dict(kind="solve", nx=s, ny=s, nz=s, precond="dic"))
            w = {k: w[k] + one[k] for k in w}
        return w
    N, F, Bf = _counts(case["nx"], case["ny"], case["nz"])
    if kind in ("solve", "pbicg", "gamg", "adjoint"):
        # addressing, coefficients, b in, x out; the operations of as many iterations as the side needs
        # (it grows with the side), each one Amul, one preconditioning and the vector updates
        side = max(case["nx"], case["ny"], case["nz"])
        its = {"solve": 5.0 * side, "adjoint": 10.0 * side, "pbicg": 12.0, "gamg": 40.0}[kind]
        per = (8 * F + 13 * N) * (2 if kind == "pbicg" else 1)
        return {"bytes": 16.0 * F + 24.0 * N, "flops": its * per}
    if kind == "amul":
        return {"bytes": 16.0 * F + 24.0 * N if case["dtype"] == "f64" else 12.0 * F + 12.0 * N,
                "flops": 4.0 * F + N}
    if kind == "assembly":
        # forward: S, gamma, addressing, centres in, upper, diag out; reverse: their gradients in, dgamma out
        return {"bytes": 64.0 * F + 48.0 * N + 80.0 * Bf, "flops": 40.0 * F + 6.0 * N}
    # S, C_f, gamma, phi, upper, addressing, centres, volumes, p in; w, grad, corr, b, phi, div out
    return {"bytes": 8.0 * (3 + 3 + 1 + 1 + 1 + 1 + 3) * F + 8.0 * (3 + 1 + 1 + 3 + 1 + 1) * N + 90.0 * Bf,
            "flops": 95.0 * F + 15.0 * N}


# ------------------------------------------------- the same in plain torch ---
def _mv(B, diag, lower, upper, x):
    l, u = B.lower.long(), B.upper_addr.long()
    y = diag * x
    y.index_add_(0, u, lower * x[l])
    y.index_add_(0, l, upper * x[u])
    return y


def _csr(B, diag, lower, upper):
    l, u = B.lower.long(), B.upper_addr.long()
    i = torch.arange(B.n, device="cuda")
    rows, cols = torch.cat([i, u, l]), torch.cat([i, l, u])
    order = torch.argsort(rows * B.n + cols)
    crow = torch.zeros(B.n + 1, dtype=torch.int64, device="cuda")
    crow[1:] = torch.bincount(rows, minlength=B.n).cumsum(0)
    return torch.sparse_csr_tensor(crow, cols[order], torch.cat([diag, lower, upper])[order], (B.n, B.n))


def _cg(A, diag, b, tol=1e-15):
    """Jacobi-preconditioned CG, then the same on the remaining residual."""
    x = torch.zeros_like(b)
    for _ in range(2):
        r = b - A @ x
        z = r / diag
        p, rho = z.clone(), torch.dot(r, z)
        d, stop = torch.zeros_like(b), tol * b.norm()
        for k in range(20000):
            q = A @ p
            alpha = rho / torch.dot(p, q)
            d += alpha * p
            r -= alpha * q
            if k % 25 == 24 and float(r.norm()) < stop:
                break
            z = r / diag
            rho, old = torch.dot(r, z), rho
            p = z + (rho / old) * p
        x = x + d
    return x


def _bicgstab(A, diag, b, tol=1e-15):
    x = torch.zeros_like(b)
    for _ in range(2):
        r = b - A @ x
        r0, d = r.clone(), torch.zeros_like(b)
        rho = alpha = om = torch.ones((), dtype=torch.float64, device="cuda")
        v, p = torch.zeros_like(b), torch.zeros_like(b)
        stop = tol * b.norm()
        for _ in range(400):
            rn = torch.dot(r0, r)
            p = r + (rn / rho) * (alpha / om) * (p - om * v)
            y = p / diag
            v = A @ y
            alpha = rn / torch.dot(r0, v)
            s = r - alpha * v
            z = s / diag
            t = A @ z
            om = torch.dot(t, s) / torch.dot(t, t)
            d += alpha * y + om * z
            r = s - om * t
            rho = rn
            if float(r.norm()) < stop:
                break
        x = x + d
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for B in _batch_blocks(case, seed):
            diag, upper = B.matrix()
            out.append(_cg(_csr(B, diag, upper, upper), diag, B.b))
        return out
    B = _block(case, seed)
    l, u = B.lower.long(), B.upper_addr.long()
    if kind in ("solve", "gamg"):
        diag, upper = B.matrix()
        return {"x": _cg(_csr(B, diag, upper, upper), diag, B.b), "converged": None}
    if kind == "pbicg":
        diag, lower, upper = B.convection()
        return {"x": _bicgstab(_csr(B, diag, lower, upper), diag, B.b), "converged": None}
    if kind == "amul":
        diag, upper = B.matrix()
        ops = (diag, upper, B.b)
        if case["dtype"] == "f32":
            ops = tuple(t.float().double() for t in ops)
        return _mv(B, ops[0], ops[1], ops[1], ops[2])
    k, kb = B.coeffs()
    if kind == "assembly":
        gu = torch.randn(B.lower.numel(), generator=B.gen, **B.kw)
        gd = torch.randn(B.n, generator=B.gen, **B.kw)
        diag, upper = B.matrix()
        return {"upper": upper, "diag": diag, "dgamma": (gd[l] + gd[u] - gu) * k, "dbgamma": gd[B.bcell.long()] * kb}
    if kind == "adjoint":
        xt = torch.randn(B.n, generator=B.gen, **B.kw)
        diag, upper = B.matrix()
        A = _csr(B, diag, upper, upper)
        x = _cg(A, diag, B.b)
        lam = _cg(A, diag, x - xt)
        du, dd = -(lam[l] * x[u] + lam[u] * x[l]), -lam * x
        return {"x": x, "dgamma": (dd[l] + dd[u] - du) * k, "dbgamma": dd[B.bcell.long()] * kb, "db": lam}
    # the finite-volume operators
    diag, upper = B.matrix()
    phi = torch.randn(B.lower.numel(), generator=B.gen, **B.kw) * B.sf.norm(dim=1)
    bphi = torch.randn(B.bcell.numel(), generator=B.gen, **B.kw) * B.bsf.norm(dim=1)
    p = torch.randn(B.n, generator=B.gen, **B.kw)
    own, nei = _dot(B.sf, B.cf - B.c[l]).abs(), _dot(B.sf, B.c[u] - B.cf).abs()
    w = nei / (own + nei)
    bc = B.bcell.long()
    sp = B.sf * (w * p[l] + (1.0 - w) * p[u])[:, None]
    grad = torch.zeros(B.n, 3, **B.kw)
    grad.index_add_(0, l, sp).index_add_(0, u, -sp)
    grad.index_add_(0, bc, B.bsf * torch.where(B.btype == 1, torch.zeros_like(p[bc]), p[bc])[:, None])
    grad = grad / B.v[:, None]
    d, mag = B.c[u] - B.c[l], B.sf.norm(dim=1)
    delta = 1.0 / torch.maximum(_dot(B.sf, d) / mag, 0.05 * d.norm(dim=1))
    kk = B.sf / mag[:, None] - d * delta[:, None]
    corr = B.gamma * mag * _dot(kk, w[:, None] * grad[l] + (1.0 - w)[:, None] * grad[u])
    b = torch.zeros(B.n, **B.kw)
    b.index_add_(0, l, corr - phi).index_add_(0, u, phi - corr).index_add_(0, bc, -bphi)
    out = phi - (-upper * (p[u] - p[l]) + corr)
    bout = bphi + B.bgamma * kb * p[bc]
    div = torch.zeros(B.n, **B.kw)
    div.index_add_(0, l, out).index_add_(0, u, -out).index_add_(0, bc, bout)
    return {"w": w, "grad": grad, "corr": corr, "b": b, "phi": out, "bphi": bout, "div": div}
