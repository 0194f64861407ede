"""The no-allocation step over its range of sizes: two kernels, mass summed by the last block.

Populations against the regular step on the split pass (the same formulas; FP32 within 2e-5 of the largest),
mass against the 64-bit sum of the input (nothing leaves a periodic lattice; a density is a sum of 19
floats, so 19 x 6e-8 at most), in repeated calls (the slots and the count of blocks start anew), with
and without the sum.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [(4, 4, 4), (5, 4, 7), (33, 5, 6), (31, 9, 4), (32, 4, 8), (97, 6, 5), (128, 128, 64)])
def test_sizes_against_the_regular_step(size):
    import torch

    import __graft_entry__

    __graft_entry__.build()
    from paper_1902_10432_gb300 import cbl

    nx, ny, nz = size
    rng = np.random.default_rng(nx)
    rho = 0.12 + 1.77 * (rng.random((nz, ny, nx)) > 0.55)
    u = 0.01 * rng.standard_normal((nz, ny, nx, 3))
    ext = (1e-4, -2e-4, 5e-5)
    sim = cbl.Sim(nx, ny, nz, prec="fp32", tau=1.1, ext_force=ext)
    sim.set_option("lbm_variant", 0)
    sim.init_fluid_fields(rho, u)
    a = torch.tensor(sim.populations().reshape(-1), dtype=torch.float32, device="cuda")
    b = torch.empty_like(a)
    mass = torch.zeros(1, dtype=torch.float64, device="cuda")
    for k in range(3):
        total = float(a.double().sum())
        cbl.lbm_step_noalloc(a, b, nx, ny, nz, tau=1.1, ext_force=ext, mass_out=None if k == 1 else mass)
        torch.cuda.synchronize()
        sim.step(1)
        ref = sim.populations().reshape(-1)
        assert np.abs(b.double().cpu().numpy() - ref).max() < 2e-5 * np.abs(ref).max()
        if k != 1:
            assert abs(mass.item() - total) < 19 * 6e-8 * total
        a, b = b, a
