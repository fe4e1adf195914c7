"""Forms of the Lanczos kernels that a solve's sizes choose, each with the kernel that ran asserted.

Solves of more steps than the history holds (128): the solution is formed in parts and the COCG direction handed over,
on chip in FP32 and FP64 and streaming, in a box and in a periodic cell; and the same systems solved on chip (few)
and streaming (many).  The systems are empty boxes and cells, their orbitals products of 1D eigenvectors.  The
kernel is read from the profile of a call with the same number of systems (the plan depends on that
number, the grid and the options alone).  Tolerances: residuals formed by the oracle at 1.5 tol; two solves that
meet tol differ by at most 2 tol cond(A), cond(A) <= top / omega.
"""
import dataclasses

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


def empty(grid, h, periodic, n_s):
    """Orbitals (n_s, n_d) and energies of the grid without a potential, and a bound on the spectrum."""
    w = synth.fornberg_second_derivative(6)
    axes = []
    for n in grid:
        d = np.zeros((n, n))
        for i in range(n):
            for o in range(-6, 7):
                if periodic:
                    d[i, (i + o) % n] -= 0.5 * w[abs(o)] / h ** 2
                elif 0 <= i + o < n:
                    d[i, i + o] -= 0.5 * w[abs(o)] / h ** 2
        axes.append(np.linalg.eigh(d))
    pick = sorted((axes[0][0][a] + axes[1][0][b] + axes[2][0][c], a, b, c)
                  for a in range(3) for b in range(3) for c in range(3))[:n_s]
    psi = np.stack([np.einsum("z,y,x->zyx", axes[2][1][:, c], axes[1][1][:, b], axes[0][1][:, a]).reshape(-1)
                    for _, a, b, c in pick])
    return psi, np.array([p[0] for p in pick]), sum(a[0][-1] for a in axes)


def run(rpa, grid, h, periodic, nsys, omega, n_s=1, **options):
    psi, eps, top = empty(grid, h, periodic, n_s)
    n_d = psi.shape[1]
    o = dataclasses.replace(rpa.default_options(), periodic=int(periodic), **options)
    b = np.random.default_rng(4).standard_normal((nsys, n_d))
    orbs = np.arange(nsys) % n_s
    with rpa.Context(*grid, h, torch.zeros(n_d, dtype=torch.float64, device="cuda"), torch.as_tensor(psi, device="cuda"), eps,
                     o) as ctx:
        x, it, st, code = ctx.sternheimer_solve(omega, orbs, torch.as_tensor(b, device="cuda"), project=False)
        assert nsys % n_s == 0
        ctx.set_options(dataclasses.replace(o, profile=1, n_omega=1, fixed_subspace_iters=1))
        names = [k["name"] for k in ctx.ec(torch.as_tensor(synth.trial_vectors(3, nsys // n_s, n_d), device="cuda")).stats["kernels"]]
    assert code == rpa.RPA_OK and np.all(st.cpu().numpy() == 0)
    g = oracle.Grid(*grid, h, periodic=True) if periodic else oracle.Grid(*grid, h)
    x = x.cpu().numpy()
    for i in sorted({0, nsys - 1}):
        r = b[i] - oracle.apply_h(g, np.zeros(n_d), x[i], -eps[orbs[i]] + 1j * omega)
        assert np.linalg.norm(r) <= 1.5 * options["tol"] * np.linalg.norm(b[i])
    return x, it.cpu().numpy(), names, top


@pytest.mark.parametrize("kernel,prec,grid,periodic", [
    ("k_lanczos<f32>", "mixed", (30, 28, 26), False),
    ("k_lanczos<f32>", "mixed", (31, 29, 28), True),
    ("k_lanczos<f64>", "fp64", (18, 17, 16), False),
    ("k_lanczos<f64>", "fp64", (22, 21, 20), True),
    ("k_lanczos_stream<f32>", "mixed", (72, 70, 12), False),
    ("k_lanczos_stream<f32>", "mixed", (57, 61, 10), True),
])
def test_solves_past_the_history(rpa, kernel, prec, grid, periodic):
    """One inner solve each (the mixed form's tolerance is that of one), of more than 128 steps."""
    mixed = prec == "mixed"
    _, it, names, _ = run(rpa, grid, 0.1, periodic, 2, 0.05, prec=rpa.RPA_MIXED if mixed else rpa.RPA_FP64,
                          tol=1e-4 if mixed else 1e-11, inner_tol=1e-5)
    assert any(n.startswith(kernel) for n in names), names
    assert np.all(it > 135), it


def test_on_chip_and_streaming_solutions_of_the_same_systems(rpa):
    grid, h, omega, tol = (46, 45, 44), 0.5, 0.4, 1e-10
    few, _, n_few, top = run(rpa, grid, h, False, 3, omega, prec=rpa.RPA_MIXED, tol=tol)
    many, _, n_many, _ = run(rpa, grid, h, False, 200, omega, prec=rpa.RPA_MIXED, tol=tol)
    assert any(n.startswith("k_lanczos<") for n in n_few), n_few
    assert any(n.startswith("k_lanczos_stream<") for n in n_many), n_many
    assert np.linalg.norm(few - many[:3]) <= 2 * tol * top / omega * np.linalg.norm(few)


@pytest.mark.parametrize("prec,grid,periodic,nsys", [
    ("mixed", (6, 6, 8), False, 1), ("fp64", (16, 14, 9), False, 200), ("mixed", (21, 9, 31), False, 2),
    ("fp64", (15, 7, 11), True, 4), ("mixed", (14, 13, 24), True, 2)])
def test_kernel_of_small_and_odd_grids(rpa, prec, grid, periodic, nsys):
    _, _, names, _ = run(rpa, grid, 0.5, periodic, nsys, 0.4, prec=rpa.RPA_MIXED if prec == "mixed" else rpa.RPA_FP64, tol=1e-10)
    assert any(n.startswith("k_lanczos<") for n in names), names
