"""The split COCG kernels on periodic grids that their xy tiles do not divide.

The last tile along an axis reaches past the grid there; what it holds past the edge has to be the images of the
first columns.  Grids: two tiles of rows with one row too many, the same across x (tiles of up to 64 columns),
both, and z chunks.  Asserted: the oracle's residual at 1.5 tol.
"""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,shape,z_chunks,precondition", [
    ("fp64", 1, 1, 0), ("mixed", 1, 1, 0), ("mixed", 2, 1, 0), ("mixed", 1, 2, 0), ("mixed", 1, 1, 1)])
@pytest.mark.parametrize("grid", [(24, 23, 12), (28, 27, 9), (71, 11, 8), (67, 19, 8)])
def test_tiles_past_the_edge(prec, shape, z_chunks, precondition, grid):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2504_01816_gb300 as rpa
    s = synth.small_system(grid, h=0.5, n_s=2, n_wells=2, seed=31, periodic=True)
    g = oracle.Grid(s.nx, s.ny, s.nz, s.h, periodic=True)
    b = np.random.default_rng(5).standard_normal((3, s.n_d))
    orbs, omega, tol = np.arange(3) % 2, 0.4, 1e-10
    o = rpa.default_options()
    o.tol, o.prec, o.periodic = tol, rpa.RPA_MIXED if prec == "mixed" else rpa.RPA_FP64, 1
    o.stencil_shape, o.z_chunks, o.precondition = shape, z_chunks, precondition
    with rpa.Context.from_system(s, o) as ctx:
        x, _, st, code = ctx.sternheimer_solve(omega, orbs, torch.as_tensor(b, device="cuda"), project=False)
    assert code == rpa.RPA_OK and np.all(st.cpu().numpy() == 0)
    x = x.cpu().numpy()
    for i in range(3):
        r = b[i] - oracle.apply_h(g, s.vloc, x[i], -s.eps[orbs[i]] + 1j * omega)
        assert np.linalg.norm(r) <= 1.5 * tol * np.linalg.norm(b[i])
