"""Sternheimer solves without P_c at frequencies next to zero.

The right-hand side has the orbital whose energy is the shift, so the system is singular at omega = 0 and its solution
grows as 1 / omega.  Asserted: RPA_OK comes with a residual of 1.5 tol, formed by the oracle; at omega = 0
the call does not say that it converged.  In FP64 the residual that a recursion carries parts from the true one
by eps top / omega (2e-10 at omega = 1e-6, top = 48), which sets the tolerances here.
"""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,omega,tol", [
    ("fp64", 0.0, 1e-8), ("mixed", 0.0, 1e-8), ("fp64", 1e-6, 1e-8), ("fp64", 1e-4, 1e-10), ("mixed", 1e-4, 1e-8),
    ("mixed", 1e-2, 1e-10)])
def test_frequencies_next_to_zero(prec, omega, tol):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2504_01816_gb300 as rpa
    s = synth.small_system((20, 17, 16), h=0.5, n_s=4, n_wells=4, seed=29)
    g = oracle.Grid(s.nx, s.ny, s.nz, s.h)
    b = np.random.default_rng(8).standard_normal((4, s.n_d))
    orbs = np.arange(4)
    o = rpa.default_options()
    o.tol, o.prec = tol, rpa.RPA_MIXED if prec == "mixed" else rpa.RPA_FP64
    with rpa.Context.from_system(s, o) as ctx:
        x, _, st, code = ctx.sternheimer_solve(omega, orbs, torch.as_tensor(b, device="cuda"), project=False)
    if omega == 0.0:
        assert code in (rpa.RPA_ERR_NOT_CONVERGED, rpa.RPA_ERR_BREAKDOWN)
        return
    assert code == rpa.RPA_OK
    x = x.cpu().numpy()
    for i in range(4):
        r = b[i] - oracle.apply_h(g, s.vloc, x[i], -s.eps[orbs[i]] + 1j * omega)
        assert np.linalg.norm(r) <= 1.5 * tol * np.linalg.norm(b[i])
