"""The P_c coefficients of chi0's pair systems in FP64 (k_gram_pairs): one contraction for all orbital pairs.

Tiles are 32 pairs by 32 columns, chunks a multiple of 32 points: one pair and one column, a pair count just
above a tile with a ragged column tile, and a grid whose last chunk is partly filled.  Coefficients that miss a
pair or a point leave an occupied component in the right-hand sides, far above the tolerance: two
solvers that meet tol = 1e-11 differ by at most 2 tol cond(A) (cond(A) <= top / omega < 1e3 here).
"""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,n_s,ncols", [((8, 7, 9), 1, 1), ((9, 8, 8), 8, 33), ((13, 11, 7), 3, 5)])
def test_pair_coefficients(grid, n_s, ncols):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2504_01816_gb300 as rpa
    s = synth.small_system(grid, h=0.5, n_s=n_s, n_wells=n_s, seed=11)
    v = synth.random_block(2, ncols, s.n_d)
    o = rpa.default_options()
    o.tol, o.prec = 1e-11, rpa.RPA_FP64
    with rpa.Context.from_system(s, o) as ctx:
        r, code = ctx.apply_nuchi0(0.5, torch.as_tensor(v, device="cuda"), symmetric=False)
    assert code == rpa.RPA_OK
    ref = oracle.Oracle.from_system(s).nu_chi0(v, 0.5, 1e-11)
    assert np.max(np.abs(r.cpu().numpy() - ref)) <= 2e-8 * np.max(np.abs(ref))
