"""The Lanczos kernels of the Sternheimer solves (csrc/lanczos.cu) against the oracle's COCG.

Grids at the edges of its tiling: rows that are not a multiple of the 16-byte units, an odd number of
rows, slabs of unequal height, slabs thinner than the stencil's reach (halos over several blocks),
one system and more systems than resident clusters.  Tolerance: two solvers that both meet
||b - A x|| <= tol ||b|| differ by at most 2 tol cond(A) in x; |A^-1| <= 1 / omega and |A| is bounded by
the stencil's symbol and the potential, so cond(A) <= top / omega, of which the residuals of a converged
solve use a part: the test asks for 2 tol top / omega.
"""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rpa():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2504_01816_gb300 as m
    return m


def solve_and_check(rpa, grid, prec, periodic, nsys, h=0.5, omega=0.4, tol=1e-11, project=False, orbital=None,
                    kernel="k_lanczos<"):
    s = synth.small_system(grid, h=h, n_s=2, n_wells=2, seed=29, periodic=periodic)
    g = oracle.Grid(s.nx, s.ny, s.nz, s.h, periodic=periodic) if periodic else oracle.Grid(s.nx, s.ny, s.nz, s.h)
    b = np.random.default_rng(8).standard_normal((nsys, s.n_d))
    orbs = np.arange(nsys) % s.n_s if orbital is None else np.full(nsys, orbital)
    o = rpa.default_options()
    o.tol, o.prec = tol, rpa.RPA_MIXED if prec == "mixed" else rpa.RPA_FP64
    with rpa.Context.from_system(s, o) as ctx:
        x, it, st, code = ctx.sternheimer_solve(omega, orbs, torch.as_tensor(b, device="cuda"), project=project)
        o2 = rpa.Options(**{**o.__dict__, "profile": 1, "n_omega": 1, "fixed_subspace_iters": 1})
        ctx.set_options(rpa.Options(**{**o2.__dict__, "periodic": int(periodic)}))
        res = ctx.ec(torch.as_tensor(synth.trial_vectors(3, 2, s.n_d), device="cuda"))
    assert any(k["name"].startswith(kernel) for k in res.stats["kernels"]), res.stats["kernels"]
    assert code == rpa.RPA_OK and np.all(st.cpu().numpy() == 0)
    x, it = x.cpu().numpy(), it.cpu().numpy()
    sig = -s.eps[orbs] + 1j * omega
    bp = b - (b @ s.psi.T) @ s.psi if project else b
    w = synth.fornberg_second_derivative(6)
    top = 1.5 * (abs(w[0]) + 2.0 * np.abs(w[1:]).sum()) / h ** 2 + float(np.abs(s.vloc).max()) + float(np.abs(sig).max())
    check = np.unique(np.linspace(0, nsys - 1, min(nsys, 6)).astype(int))
    ref, rit, rst = oracle.cocg(g, s.vloc, sig[check], bp[check].astype(complex), tol, 100000)
    assert np.all(rst == 0)
    for k, i in enumerate(check):
        r = bp[i] - oracle.apply_h(g, s.vloc, x[i], sig[i])
        assert np.linalg.norm(r) <= 1.5 * tol * np.linalg.norm(bp[i])
        assert np.linalg.norm(x[i] - ref[k]) <= 2 * tol * top / omega * np.linalg.norm(ref[k])
    return it, rit


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("grid,periodic,nsys", [
    ((6, 6, 8), False, 1),          # the smallest grid the kernel takes; one system
    ((13, 11, 17), False, 3),       # odd along every axis, slabs of unequal height
    ((16, 14, 9), False, 200),      # more systems than clusters of the larger sizes
    ((21, 9, 31), False, 2),        # rows of 5 units and one point
    ((12, 10, 8), True, 1),         # periodic: images inside 16-byte units
    ((15, 7, 11), True, 4),         # periodic with odd rows: images by single points
    ((14, 13, 24), True, 2),        # periodic, rows not a multiple of the unit, an odd number of rows
])
def test_lanczos_matches_oracle(rpa, prec, grid, periodic, nsys):
    solve_and_check(rpa, grid, prec, periodic, nsys)


@pytest.mark.parametrize("project", [False, True])
def test_lanczos_past_its_history(rpa, project):
    """A fine grid: more steps than the history holds (128), so that the solution is formed in parts and
    the COCG direction handed over between them."""
    it, rit = solve_and_check(rpa, (14, 13, 15), "fp64", False, 2, h=0.12, omega=0.3, tol=1e-11, project=project,
                              orbital=1)
    assert np.all(it > 140), it
    assert np.all(np.abs(it - rit) <= np.maximum(3, 0.1 * rit)), (it, rit)


@pytest.mark.parametrize("prec,grid,nsys", [
    ("mixed", (20, 17, 16), 700),   # several solves a cluster, short: the solution warps keep up
    ("mixed", (33, 31, 30), 160),   # large blocks: the other warps take part in what they leave
    ("fp64", (17, 15, 16), 320),
])
def test_lanczos_solutions_formed_beside_the_next_solve(rpa, prec, grid, nsys):
    """Every solution of a queue is its own system's, and the same whichever warps formed its points."""
    s = synth.small_system(grid, h=0.5, n_s=2, n_wells=2, seed=29)
    g = oracle.Grid(s.nx, s.ny, s.nz, s.h)
    b = np.random.default_rng(9).standard_normal((nsys, s.n_d))
    orbs = np.arange(nsys) % s.n_s
    o = rpa.default_options()
    o.tol, o.prec = 1e-10, rpa.RPA_MIXED if prec == "mixed" else rpa.RPA_FP64
    with rpa.Context.from_system(s, o) as ctx:
        bt = torch.as_tensor(b, device="cuda")
        runs = [ctx.sternheimer_solve(0.4, orbs, bt, project=False) for _ in range(3)]
        xs = [r[0].cpu().numpy() for r in runs]
    assert all(r[3] == rpa.RPA_OK for r in runs)
    assert np.array_equal(xs[0], xs[1]) and np.array_equal(xs[0], xs[2])
    for i in range(nsys):
        r = b[i] - oracle.apply_h(g, s.vloc, xs[0][i], -s.eps[orbs[i]] + 0.4j)
        assert np.linalg.norm(r) <= 1.5 * 1e-10 * np.linalg.norm(b[i]), i


@pytest.mark.parametrize("grid,nsys", [
    ((57, 61, 10), 3),              # rows of 14 units and one point, odd rows, bands of unequal height
    ((90, 90, 8), 2),               # wide planes: several bands, the fewest planes the kernel takes
    ((72, 70, 20), 90),             # more systems than resident clusters
])
@pytest.mark.parametrize("h,tol", [(0.5, 1e-11), (0.12, 1e-10)])
def test_streaming_lanczos_matches_oracle(rpa, grid, nsys, h, tol):
    """Grids that do not fit on chip; at h = 0.12 the solves take more steps than the history holds."""
    if h < 0.2 and nsys > 3:
        pytest.skip("the oracle's time")
    solve_and_check(rpa, grid, "mixed", False, nsys, h=h, tol=tol, kernel="k_lanczos_stream")


def test_on_chip_and_streaming_solutions_agree(rpa):
    """Grids of more than four blocks a system: few systems are solved on chip, many by the streaming kernel."""
    s = synth.small_system((46, 45, 44), h=0.5, n_s=1, n_wells=1, seed=5)
    b = torch.as_tensor(np.random.default_rng(6).standard_normal((200, s.n_d)), device="cuda")
    o = rpa.default_options()
    o.tol, o.prec = 1e-10, rpa.RPA_MIXED
    with rpa.Context.from_system(s, o) as ctx:
        few = ctx.sternheimer_solve(0.4, np.zeros(3, int), b[:3], project=False)
        many = ctx.sternheimer_solve(0.4, np.zeros(200, int), b, project=False)
    assert few[3] == rpa.RPA_OK and many[3] == rpa.RPA_OK
    x, y = few[0].cpu().numpy(), many[0][:3].cpu().numpy()
    w = synth.fornberg_second_derivative(6)
    top = 1.5 * (abs(w[0]) + 2.0 * np.abs(w[1:]).sum()) / 0.25 + float(np.abs(s.vloc).max()) + abs(-s.eps[0] + 0.4j)
    assert np.linalg.norm(x - y) <= 2 * 1e-10 * top / 0.4 * np.linalg.norm(x)


@pytest.mark.parametrize("grid,nsys", [
    ((57, 61, 10), 2),              # rows of 14 units and one point, odd rows, bands of unequal height
    ((64, 62, 9), 70),              # several solves a cluster
    ((90, 70, 8), 1),               # images in whole units, the fewest planes
])
def test_periodic_streaming_lanczos_matches_oracle(rpa, grid, nsys):
    """Periodic grids that do not fit on chip: images along every axis."""
    solve_and_check(rpa, grid, "mixed", True, nsys, h=0.5, tol=1e-11, kernel="k_lanczos_stream")
