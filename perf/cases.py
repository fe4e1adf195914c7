"""Timed cases of the real-space RPA hot path, through the package's public entry points.

A case names an entry point (op), the model system (grid, spacing, wells, orbitals, boundary
conditions) and the sizes of the call:

  coulomb      Context.coulomb_apply: nu^power on a block of grid functions
  sternheimer  Context.sternheimer_solve: a list of Sternheimer systems, one per right-hand side
  chi0         Context.apply_nuchi0: nu^1/2 chi0(i omega) nu^1/2 on a block of trial vectors
  batch        apply_nuchi0_batch: the same for several independent systems of different sizes
  ec           Context.ec: the subspace iteration over the frequencies, Ritz values and E_c
  grad         Context.ec_gradient: the same and dE_c/dV_loc

The systems are Gaussian wells in a box (or a periodic cell) with their exact lowest orbitals.  A
program has the ground state in hand (the method reads it from files), so a case's ground state is
computed once and kept in this module; the seed picks one of its eight mirror images, and the
blocks of vectors.  Options are the library's defaults but for the precision, the COCG tolerance,
the boundary conditions and the counts of frequencies and iterations.  The tolerance is 1e-11, the
one of the parity tests: what the calls return in 64 bits is then determined well below what a
change of rounding within a converged solve can move.
"""
import functools
import math

import numpy as np
import torch

import paper_2504_01816_gb300 as rpa

RADIUS = 6


def _case(name, op, grid, n_s, n_r, prec="mixed", h=0.4, omega=0.3, periodic=False, **more):
    c = dict(op=op, nx=grid[0], ny=grid[1], nz=grid[2], h=h, n_s=n_s, n_r=n_r, prec=prec, omega=omega,
             periodic=periodic, tol=1e-11)
    if name:
        c["name"] = name
    c.update(more)
    return c


def listed():
    return [
        # one right-hand side per orbital of a small molecule: latency and launches count
        _case("sternheimer_24", "sternheimer", (24, 24, 24), 4, 4, h=0.45),
        # the tiny isolated system in the plain FP64 form: one application of the operator
        _case("chi0_15_fp64", "chi0", (15, 15, 15), 4, 8, prec="fp64", h=0.5),
        # the Coulomb half-apply of a whole block of trial vectors, FP64
        _case("coulomb_40", "coulomb", (40, 40, 40), 1, 64, power=0.5),
        # independent molecules of different sizes in one call
        _case("batch_24_32", "batch", (24, 24, 24), 4, 6, h=0.45, omega=0.7,
              systems="24x24x24/4/6,28x26x30/6/5,32x32x32/8/4"),
        # the benchmark system: one application to its whole block of trial vectors
        _case("chi0_40", "chi0", (40, 40, 40), 16, 64),
        # a bulk cell at the benchmark's sizes
        _case("chi0_bulk40", "chi0", (40, 40, 40), 16, 16, periodic=True),
        # odd sizes: an odd number of points along every axis, ragged counts of orbitals and vectors
        _case("chi0_odd", "chi0", (37, 43, 29), 7, 11, omega=1.1),
        # the largest molecule of the uneven batch: planes past one block of the fused kernel
        _case("chi0_56", "chi0", (56, 56, 56), 32, 8, omega=0.7),
        # the LiH-shaped cell: 128 electrons
        _case("chi0_lih72", "chi0", (72, 72, 72), 64, 4, h=0.3, omega=0.7),
        # the plain FP64 form at an ordinary size
        _case("chi0_32_fp64", "chi0", (32, 32, 32), 8, 16, prec="fp64", h=0.45),
        # a whole E_c evaluation: two iterations at each of two frequencies
        _case("ec_32", "ec", (32, 32, 32), 8, 32, h=0.45, n_omega=2, iters=2),
        # E_c and its gradient by the adjoint, as an optimisation of the potential calls it
        _case("grad_32", "grad", (32, 32, 32), 8, 16, h=0.45, n_omega=2, iters=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["coulomb", "sternheimer", "chi0", "chi0", "chi0", "chi0", "batch", "ec", "grad"])
    periodic = rng.random() < 0.2
    omega = round(math.exp(rng.uniform(math.log(0.1), math.log(4.0))), 3)
    base = rng.randint(15, 56)
    grid = [base if rng.random() < 0.4 else max(13, min(60, base + rng.randint(-7, 7))) for _ in range(3)]
    nd = grid[0] * grid[1] * grid[2]
    h = rng.choice([0.4, 0.45, 0.5])
    if op == "coulomb":
        return _case(None, op, grid, 1, max(1, min(_log_int(rng, 1, 128), 8_000_000 // nd)), h=h, periodic=periodic,
                     power=rng.choice([0.5, 1.0]))
    if op == "batch":
        parts = []
        for _ in range(rng.randint(2, 5)):
            g = [rng.randint(20, 36) for _ in range(3)]
            parts.append("%dx%dx%d/%d/%d" % (*g, rng.randint(3, 9), rng.randint(2, 8)))
        return _case(None, op, [int(v) for v in parts[0].split("/")[0].split("x")], 4, 4, h=0.45, omega=omega,
                     systems=",".join(parts))
    prec = "fp64" if rng.random() < 0.2 and nd < 40_000 else "mixed"
    n_s = rng.randint(3, 8) if nd < 20_000 else rng.randint(6, 24)
    solves = max(4.0, min(1024.0, 3.0e7 / nd)) / (8.0 if prec == "fp64" else 1.0)
    if op == "sternheimer":
        return _case(None, op, grid, n_s, max(1, min(_log_int(rng, 1, 64), int(solves))), prec, h, omega, periodic)
    if op in ("ec", "grad"):
        n_r = max(2, min(_log_int(rng, 4, 64), int(solves / n_s / 2)))
        return _case(None, op, grid, n_s, n_r, prec, h, 0.0, periodic, n_omega=rng.randint(1, 2),
                     iters=rng.randint(1, 2) if op == "ec" else 1)
    return _case(None, op, grid, n_s, max(1, min(_log_int(rng, 2, 64), int(solves / n_s))), prec, h, omega, periodic)


# ------------------------------------------------------------------------- model systems
def _second_difference(n, h, periodic):
    """-d2/dx2 on n points, 12th-order centred differences."""
    f = math.factorial
    w = [0.0] + [2.0 * (-1) ** (k + 1) * f(RADIUS) ** 2 / (k * k * f(RADIUS - k) * f(RADIUS + k))
                 for k in range(1, RADIUS + 1)]
    w[0] = -2.0 * sum(1.0 / k ** 2 for k in range(1, RADIUS + 1))
    d = np.zeros((n, n))
    for i in range(n):
        for o in range(-RADIUS, RADIUS + 1):
            j = i + o
            if periodic:
                d[i, j % n] -= w[abs(o)] / h ** 2
            elif 0 <= j < n:
                d[i, j] -= w[abs(o)] / h ** 2
    return torch.as_tensor(d, device="cuda")


class _Operator:
    """H = -1/2 L_h + V on rows of grid functions (plain torch, per-axis matrix products)."""

    def __init__(self, grid, h, v, periodic):
        self.nx, self.ny, self.nz = grid
        self.d = [_second_difference(n, h, periodic) for n in grid]
        self.v = v
        self.top = 0.5 * sum(float(torch.linalg.eigvalsh(d)[-1]) for d in self.d) + max(0.0, float(v.max()))

    def to(self, dtype):
        o = object.__new__(_Operator)
        o.nx, o.ny, o.nz, o.top = self.nx, self.ny, self.nz, self.top
        o.d = [d.to(dtype) for d in self.d]
        o.v = self.v.to(dtype)
        return o

    def __call__(self, x):
        k = x.shape[0]
        if x.is_complex():
            r = torch.view_as_real(x).movedim(-1, 1).reshape(2 * k, -1)
            return torch.view_as_complex(self(r).view(k, 2, -1).movedim(1, -1).contiguous())
        dx, dy, dz = self.d
        a = x.reshape(-1, self.nx) @ dx
        a = a.view(k * self.nz, self.ny, self.nx) + torch.matmul(dy, x.reshape(k * self.nz, self.ny, self.nx))
        a = a.view(k, self.nz, -1) + torch.matmul(dz, x.reshape(k, self.nz, -1))
        return 0.5 * a.reshape(k, -1) + self.v * x


def _orthonormal(x):
    for _ in range(2):
        c = torch.linalg.cholesky(x.double() @ x.double().T)
        x = torch.linalg.solve_triangular(c, x.double(), upper=False).to(x.dtype)
    return x


@functools.lru_cache(maxsize=16)
def _ground_state(grid, h, n_s, periodic):
    """V_loc of n_s Gaussian wells (at least 4) and the n_s lowest orbitals of its Hamiltonian, by
    Chebyshev-filtered subspace iteration: in FP32 first, then in FP64 to a residual of 1e-11."""
    rng = np.random.default_rng([*grid, n_s, int(periodic), int(1000 * h)])
    wells = max(4, n_s)
    box = [n * h if periodic else (n + 1) * h for n in grid]
    axes = [np.arange(n) * h if periodic else (np.arange(n) + 1.0) * h for n in grid]
    v = np.zeros(grid[::-1])
    for _ in range(wells):
        depth, width = rng.uniform(1.0, 3.0), rng.uniform(0.8, 1.5)
        g = []
        for t, b in zip(axes, box):
            m = 0.0 if periodic else min(2.0 * width, 0.3 * b)
            c = rng.uniform(m, b - m)
            g.append(sum(np.exp(-((t - c - k * b) ** 2) / (2 * width ** 2)) for k in ((-1, 0, 1) if periodic else (0,))))
        v -= depth * g[2][:, None, None] * g[1][None, :, None] * g[0][None, None, :]
    vloc = torch.as_tensor(v.reshape(-1), device="cuda")
    op = _Operator(grid, h, vloc, periodic)
    m = n_s + max(8, n_s // 2)
    gen = torch.Generator(device="cuda").manual_seed(7)
    x = torch.randn(m, vloc.numel(), dtype=torch.float32, device="cuda", generator=gen)
    for dtype, tol, outer in ((torch.float32, 3e-4, 30), (torch.float64, 1e-11, 60)):
        f = op.to(dtype)
        x = _orthonormal(x.to(dtype))
        for _ in range(outer):
            hx = f(x)
            theta, q = torch.linalg.eigh((x @ hx.T).double())
            x, hx = q.T.to(dtype) @ x, q.T.to(dtype) @ hx
            if float(torch.linalg.norm(hx - theta.to(dtype)[:, None] * x, dim=1)[:n_s].max()) < tol:
                break
            lo, cut = float(theta[0]), float(theta[-1])
            e, c = (1.02 * op.top - cut) / 2, (1.02 * op.top + cut) / 2
            s = e / (lo - c)
            tau = 2.0 / s
            y0, y = x, (hx - c * x) * (s / e)
            for _k in range(47):
                s1 = 1.0 / (tau - s)
                y0, y, s = y, (f(y) - c * y) * (2.0 * s1 / e) - (s * s1) * y0, s1
            x = _orthonormal(y)
    eps = theta[:n_s].cpu().numpy()
    return vloc, x[:n_s].contiguous(), eps


def _system(case, seed, grid=None, n_s=None):
    """The case's ground state, mirrored along the axes that the seed picks."""
    grid = grid or (case["nx"], case["ny"], case["nz"])
    n_s = n_s or case["n_s"]
    vloc, psi, eps = _ground_state(tuple(grid), case["h"], n_s, case["periodic"])
    flips = [a + 1 for a in range(3) if (seed >> a) & 1]
    shape = (-1, grid[2], grid[1], grid[0])

    def mirror(t):
        return torch.flip(t.view(shape), flips).reshape(t.shape).contiguous() if flips else t.clone()

    return tuple(grid), mirror(vloc), mirror(psi), eps


def _block(seed, k, n, part=0):
    gen = torch.Generator(device="cuda").manual_seed(1000003 * (seed + 1) + part)
    return torch.randn(k, n, dtype=torch.float64, device="cuda", generator=gen)


def _parts(case):
    for t in case["systems"].split(","):
        g, n_s, n_r = t.split("/")
        yield tuple(int(v) for v in g.split("x")), int(n_s), int(n_r)


def _options(case):
    o = rpa.default_options()
    o.prec = rpa.RPA_MIXED if case["prec"] == "mixed" else rpa.RPA_FP64
    o.tol = case["tol"]
    o.periodic = int(case["periodic"])
    if case["op"] in ("ec", "grad"):
        o.n_omega = case["n_omega"]
        o.fixed_subspace_iters = case["iters"]
    return o


def _orbitals(case):
    return [k * case["n_s"] // case["n_r"] if case["n_r"] > case["n_s"] else k for k in range(case["n_r"])]


def prepare(case, seed):
    systems = [(g, n_s, n_r) for g, n_s, n_r in _parts(case)] if case["op"] == "batch" else \
        [((case["nx"], case["ny"], case["nz"]), case["n_s"], case["n_r"])]
    contexts, blocks = [], []
    for i, (grid, n_s, n_r) in enumerate(systems):
        _, vloc, psi, eps = _system(case, seed, grid, n_s)
        contexts.append(rpa.Context(*grid, case["h"], vloc, psi, eps, _options(case)))
        blocks.append(_block(seed, n_r, vloc.numel(), i))
    return {"case": case, "contexts": contexts, "blocks": blocks}


def run(state):
    case, ctx, x = state["case"], state["contexts"][0], state["blocks"][0]
    op = case["op"]
    if op == "coulomb":
        return ctx.coulomb_apply(case["power"], x)
    if op == "sternheimer":
        # the iteration counts say how the solutions were found and are left out
        sol, _, status, code = ctx.sternheimer_solve(case["omega"], _orbitals(case), x)
        return {"x": sol, "status": status, "code": code}
    if op == "chi0":
        r, code = ctx.apply_nuchi0(case["omega"], x)
        return {"r": r, "code": code}
    if op == "batch":
        rs, code = rpa.rpa.apply_nuchi0_batch(state["contexts"], case["omega"], state["blocks"])
        return {"r": rs, "code": code}
    if op == "ec":
        res = ctx.ec(x)
        return {"lambdas": res.lambdas, "e_c": res.e_c, "e_c_per_omega": res.e_c_per_omega, "code": res.status}
    res, g, v = ctx.ec_gradient(x, want_subspace=True)
    return {"lambdas": res.lambdas, "e_c": res.e_c, "e_c_per_omega": res.e_c_per_omega, "grad": g, "subspace": v,
            "code": res.status}


# ------------------------------------------------------------------------- 64-bit values
def _coulomb(op, x, power, h):
    """(4 pi)^p (-L_h)^-p through the per-axis eigenvectors; the zero mode of a periodic cell drops out."""
    lam, q = zip(*(torch.linalg.eigh(d) for d in op.d))
    k = x.shape[0]
    t = x.view(k, op.nz, op.ny, op.nx)
    t = torch.einsum("kzyx,xa,yb,zc->kcba", t, q[0], q[1], q[2])
    s = lam[2][:, None, None] + lam[1][None, :, None] + lam[0][None, None, :]
    ok = s > 1e-9 * float(s.max())
    f = torch.where(ok, (4.0 * math.pi / torch.where(ok, s, torch.ones_like(s))) ** power, torch.zeros_like(s))
    return torch.einsum("kcba,xa,yb,zc->kzyx", t * f, q[0], q[1], q[2]).reshape(k, -1)


def _solve(op, psi, sigma, b, project):
    """(H + sigma_k) x_k = b_k by COCG in FP64, in the complement of psi when project is set."""
    if project:
        b = b - (b @ psi.T) @ psi
    sigma = sigma[:, None]
    x = torch.zeros(b.shape, dtype=torch.complex128, device=b.device)
    r = b.to(torch.complex128)
    p = r.clone()
    rho = (r * r).sum(1, keepdim=True)
    stop = 1e-13 * torch.linalg.norm(b, dim=1, keepdim=True)
    for it in range(3000):
        live = torch.linalg.norm(r, dim=1, keepdim=True) > stop
        if it % 8 == 0 and not bool(live.any()):
            break
        q = op(p) + sigma * p
        alpha = torch.where(live, rho / (p * q).sum(1, keepdim=True), torch.zeros_like(rho))
        x += alpha * p
        r -= alpha * q
        new = (r * r).sum(1, keepdim=True)
        p = torch.where(live, r + (new / rho) * p, p)
        rho = torch.where(live, new, rho)
    if project:
        x -= torch.complex((x.real @ psi.T) @ psi, (x.imag @ psi.T) @ psi)
    return x


def _solutions(op, psi, eps, omega, dv):
    """For every orbital n the solutions of (H - eps_n + i omega) x = -P_c(u_n dv_j), j over the rows."""
    for n in range(psi.shape[0]):
        sigma = torch.full((dv.shape[0],), complex(-float(eps[n]), omega), dtype=torch.complex128, device=dv.device)
        yield n, _solve(op, psi, sigma, -psi[n] * dv, True)


def _chi(op, psi, eps, h, omega, v):
    dv = _coulomb(op, v, 0.5, h)
    rho = torch.zeros_like(dv)
    for n, x in _solutions(op, psi, eps, omega, dv):
        rho += (4.0 / h ** 3) * psi[n] * x.real
    return _coulomb(op, rho, 0.5, h)


def _rows(x):
    c = torch.linalg.cholesky(x @ x.T)
    return torch.linalg.solve_triangular(c, x, upper=False)


def exact(case, seed):
    n_all = case["nx"] * case["ny"] * case["nz"] * case["n_s"] * case["n_r"] * case.get("n_omega", 1) * \
        case.get("iters", 1)
    if case["op"] in ("chi0", "ec", "grad") and n_all > 8.0e7:
        return None
    h, omega = case["h"], case["omega"]
    if case["op"] == "batch":
        out = []
        for i, (grid, n_s, n_r) in enumerate(_parts(case)):
            _, vloc, psi, eps = _system(case, seed, grid, n_s)
            op = _Operator(grid, h, vloc, case["periodic"])
            out.append(_chi(op, psi, eps, h, omega, _block(seed, n_r, vloc.numel(), i)))
        return {"r": out, "code": None}
    grid, vloc, psi, eps = _system(case, seed)
    op = _Operator(grid, h, vloc, case["periodic"])
    x = _block(seed, case["n_r"], vloc.numel())
    if case["op"] == "coulomb":
        return _coulomb(op, x, case["power"], h)
    if case["op"] == "sternheimer":
        sigma = torch.as_tensor([complex(-eps[n], omega) for n in _orbitals(case)], device="cuda")
        return {"x": _solve(op, psi, sigma, x, True), "status": None, "code": None}
    if case["op"] == "chi0":
        return {"r": _chi(op, psi, eps, h, omega, x), "code": None}
    nodes, weights = np.polynomial.legendre.leggauss(case["n_omega"])
    om, wt = (1.0 + nodes) / (1.0 - nodes), 2.0 * weights / (1.0 - nodes) ** 2
    v = _rows(x)
    lambdas = np.zeros((case["n_omega"], case["n_r"]))
    per = np.zeros(case["n_omega"])
    grad = torch.zeros_like(vloc)
    for m in reversed(range(case["n_omega"])):
        for _ in range(case["iters"]):
            last, r = v, _chi(op, psi, eps, h, om[m], v)
            c = v @ r.T
            lam, q = torch.linalg.eigh(0.5 * (c + c.T))
            v = _rows(r)
        lambdas[m] = lam.cpu().numpy()
        per[m] = wt[m] / (2 * math.pi) * float((torch.log1p(-lam) + lam).sum())
        if case["op"] == "grad":
            dv = _coulomb(op, q.T @ last, 0.5, h)
            coef = wt[m] / (2 * math.pi) * (-lam / (1.0 - lam)) * (4.0 / h ** 3)
            for _, y in _solutions(op, psi, eps, om[m], dv):
                grad += (coef[:, None] * (y * y).real).sum(0)
    out = {"lambdas": lambdas, "e_c": float(per.sum()), "e_c_per_omega": per, "code": None}
    if case["op"] == "grad":
        out.update(grad=grad, subspace=v)
    return out


# ------------------------------------------------------------------------- work
def work(case):
    size = 8.0 if case["prec"] == "mixed" else 16.0
    bytes_, flops = 0.0, 0.0
    systems = list(_parts(case)) if case["op"] == "batch" else \
        [((case["nx"], case["ny"], case["nz"]), case["n_s"], case["n_r"])]
    for grid, n_s, n_r in systems:
        nd = grid[0] * grid[1] * grid[2]
        coulomb_flops = 4.0 * nd * sum(grid)
        if case["op"] == "coulomb":
            bytes_ += 16.0 * nd * n_r
            flops += coulomb_flops * n_r
            continue
        passes = case.get("n_omega", 1) * case.get("iters", 1) + \
            (case.get("n_omega", 1) if case["op"] == "grad" else 0)
        count = (n_r if case["op"] == "sternheimer" else n_s * n_r) * passes
        # what the call cannot do without: the block in and out, and the orbitals once per pass
        bytes_ += passes * 8.0 * nd * (2 * n_r + n_s) + (2 * size * nd * n_r if case["op"] == "sternheimer" else 0.0)
        # about 100 iterations to the tolerance at these spacings and frequencies: the 37-point stencil
        # and the vector updates and products of COCG on a complex block
        flops += count * nd * 100.0 * (2 * 37 + 2 * 20) + (2 * coulomb_flops * n_r * passes if case["op"] != "sternheimer" else 0.0)
    return {"bytes": bytes_, "flops": flops}
