"""rpa_ec_gradient returns the same values whether or not the final subspace is asked for (one choice of kernels)."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,prec,periodic", [
    ((16, 14, 12), "mixed", False), ((15, 13, 11), "fp64", False), ((24, 23, 12), "fp64", True), ((25, 19, 12), "mixed", True)])
def test_values_do_not_depend_on_the_outputs_asked_for(grid, prec, periodic):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2504_01816_gb300 as rpa
    s = synth.small_system(grid, h=0.5, n_s=3, n_wells=3, seed=12, periodic=periodic)
    v0 = torch.as_tensor(synth.trial_vectors(12, 6, s.n_d), device="cuda")
    o = rpa.default_options()
    o.tol, o.prec, o.periodic = 1e-10, rpa.RPA_MIXED if prec == "mixed" else rpa.RPA_FP64, int(periodic)
    o.n_omega, o.fixed_subspace_iters = 2, 2
    with rpa.Context.from_system(s, o) as ctx:
        a, ga, va = ctx.ec_gradient(v0, want_subspace=True)
        b, gb = ctx.ec_gradient(v0)[:2]
        c = ctx.ec(v0)
    assert a.status == b.status == c.status == rpa.RPA_OK
    assert np.array_equal(a.lambdas, b.lambdas) and a.e_c == b.e_c and np.array_equal(a.e_c_per_omega, b.e_c_per_omega)
    assert torch.equal(ga, gb)
    # rpa_ec solves the same systems by its own kernels: Ritz values to 2 tol cond(A) of their size
    assert np.allclose(a.lambdas, c.lambdas, rtol=1e-6, atol=1e-10)
