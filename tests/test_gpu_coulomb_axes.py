"""The Coulomb operator's axis transforms by parity (csrc/coulomb.cu) against the oracle's operator.

Axes of odd and even length, shorter than a tile's eight warps and longer than its 32 lines, lines that do
not fill the last tile, and a periodic grid, whose degenerate eigenvectors have no parity.  Tolerance: the
sums have at most max(n) terms and the factors lie within a few units of rounding of orthogonal ones, six
products: 6 n eps cond, cond = (lam_max / lam_min)^p below 1e3 here for p <= 1: 1e-10 for n <= 70; the
asserted 1e-11 leaves the rounding errors their random signs.
"""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,ncols,periodic", [
    ((8, 9, 10), 1, False),
    ((13, 7, 70), 3, False),
    ((65, 8, 7), 5, False),
    ((32, 33, 8), 2, False),
    ((14, 13, 16), 3, True),
])
def test_axis_transforms(grid, ncols, periodic):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2504_01816_gb300 as rpa
    s = synth.small_system(grid, h=0.5, n_s=1, n_wells=1, seed=3, periodic=periodic)
    op = oracle.Oracle.from_system(s).coulomb
    x = np.random.default_rng(4).standard_normal((ncols, s.n_d))
    o = rpa.default_options()
    o.prec = rpa.RPA_FP64
    with rpa.Context.from_system(s, o) as ctx:
        for p in (0.5, 1.0):
            got = ctx.coulomb_apply(p, torch.as_tensor(x, device="cuda")).cpu().numpy()
            ref = op.apply(x, p)
            assert np.linalg.norm(got - ref) <= 1e-11 * np.linalg.norm(ref), p
