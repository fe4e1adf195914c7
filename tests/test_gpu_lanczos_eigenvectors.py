"""Sternheimer solves whose right-hand side is an eigenvector, or a few of them, and a little noise.

The Krylov space of such a right-hand side is nearly invariant after one step (a few), and the norm of the next
Lanczos vector is a small difference of large sums.  The solution has to meet ||b - A x|| <= tol ||b||; the
residual is formed by the oracle's operator in FP64, whose own rounding (eps |A| |x| / |b|, with
|A| < 100 and |x| <= |b| / omega) lies below 1e-13: the asserted 1.5 tol leaves room for a recursive residual's
drift, as in the other solver tests.
"""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("grid,periodic", [((13, 13, 13), False), ((14, 12, 9), True)])
@pytest.mark.parametrize("mixed_of", [1, 3])
@pytest.mark.parametrize("noise", [0.0, 1e-12, 1e-11, 1e-10, 1e-9, 1e-7])
def test_solves_next_to_eigenvectors(prec, grid, periodic, mixed_of, noise):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2504_01816_gb300 as rpa
    s = synth.small_system(grid, h=0.5, n_s=12, n_wells=4, seed=29, periodic=periodic)
    g = oracle.Grid(s.nx, s.ny, s.nz, s.h, periodic=periodic) if periodic else oracle.Grid(s.nx, s.ny, s.nz, s.h)
    rng = np.random.default_rng(17)
    unit = lambda v: v / np.linalg.norm(v, axis=-1, keepdims=True)  # noqa: E731
    if mixed_of == 1:
        b = s.psi.copy()
    else:
        b = rng.standard_normal((12, mixed_of)) @ s.psi[:mixed_of]
    b = unit(b) + noise * unit(rng.standard_normal((12, s.n_d)))
    orbs, tol, omega = np.arange(12) % 4, 1e-11, 0.4
    o = rpa.default_options()
    o.tol, o.prec, o.periodic = tol, rpa.RPA_MIXED if prec == "mixed" else rpa.RPA_FP64, int(periodic)
    with rpa.Context.from_system(s, o) as ctx:
        x, _, st, code = ctx.sternheimer_solve(omega, orbs, torch.as_tensor(b, device="cuda"), project=False)
    assert code == rpa.RPA_OK and np.all(st.cpu().numpy() == 0)
    x = x.cpu().numpy()
    worst = max(np.linalg.norm(b[i] - oracle.apply_h(g, s.vloc, x[i], -s.eps[orbs[i]] + 1j * omega)) /
                np.linalg.norm(b[i]) for i in range(12))
    assert worst <= 1.5 * tol
