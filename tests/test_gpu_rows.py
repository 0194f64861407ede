"""The density and collision kernels over rows of 128 cells (lattices that tiles of 32 x 4 cover badly) against
the same kernels over tiles of 64 x 2 (option lbm_block_x), which never take rows.

The arithmetic of a cell is the same, so one step differs at most by how the compiler contracts products:
a few units in the last place of FP64 (1e-13) and FP32 (1e-5), and the rounding of binary16 storage (2e-2).
"""
import numpy as np
import pytest

from paper_1902_10432_gb300 import cbl, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-13), ("fp32", 1e-5), ("fp16dev", 2e-2)])
@pytest.mark.parametrize("size", [(4, 4, 4), (5, 7, 4), (33, 9, 6), (40, 36, 44), (48, 5, 9), (72, 41, 30)])
@pytest.mark.parametrize("q", [19, 27])
def test_rows_against_tiles(q, size, prec, tol):
    import __graft_entry__

    __graft_entry__.build()
    nx, ny, nz = size
    out = []
    for bx in (32, 64):
        s = cbl.Sim(nx, ny, nz, prec=prec, q=q, tau=1.1, ext_force=(1e-4, -2e-4, 5e-5))
        s.set_option("lbm_variant", 0)
        s.set_option("lbm_block_x", bx)
        if min(size) > 20:
            s.add_body("sphere", center=(nx / 2 + 0.3, ny / 2, nz / 2), radius=6.0, fixed=True)
        rng = np.random.default_rng(5)
        mask = rng.random((nz, ny, nx)) > 0.55
        s.init_fluid(1.888, 0.1194, mask)
        s.step(2)
        out.append((s.populations(), s.fields()[0], s.total_mass()))
    (fa, ra, ma), (fb, rb, mb) = out
    assert np.abs(fa - fb).max() < tol * np.abs(fb).max()
    assert np.abs(ra - rb).max() < tol * np.abs(rb).max()
    assert abs(ma - mb) < 1e-2 * tol * mb + 1e-13 * mb
