"""Batches at the limits of a launch's grid."""
import numpy as np
import pytest

from paper_1902_10432_gb300 import cbl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


def test_more_bodies_than_a_grid_numbers():
    # nine instances of 7300 spheres each (tiles of 9 x 8 x 8 cells side by side): 65700 bodies in all, beyond the
    # 65535 blocks that a grid has along z
    nb, step = 7300, 9

    def sim():
        s = cbl.Sim(step * nb, 8, 8, prec="fp32", eta=1.0, tau=0.9, mpf_kinetics=1)
        s.set_option("tile_tail", 0.0)
        for k in range(nb):
            s.add_body("sphere", center=(step * k + 4.0 + 0.3 * (k % 3), 4.0, 4.2), radius=0.9)
        mask = np.zeros((8, 8, step * nb), np.uint8)
        mask[5:] = 1
        s.init_fluid(1.9, 0.12, mask)
        return s

    sims, alone = [sim() for _ in range(9)], sim()
    b = cbl.Batch(sims)
    b.step(2)
    b.sync()
    alone.step(2)
    F = alone.body_forces()[0]
    assert np.abs(F).max() > 0
    for s in (sims[0], sims[8]):
        assert np.array_equal(s.flags()[1], alone.flags()[1])
        assert np.allclose(s.body_forces()[0], F, rtol=1e-9, atol=1e-12)
        assert np.abs(s.fields()[0] - alone.fields()[0]).max() < 2e-5
    b.close()


def test_work_items_follow_the_passes():
    # the instances change from the moment to the split pass: the items are those of the split pass alone
    def sims(variant):
        out = []
        for _ in range(2):
            s = cbl.Sim(96, 64, 96, prec="fp32")
            s.set_option("lbm_variant", variant)
            s.init_fluid(1.9, 0.12)
            out.append(s)
        return out

    split, mom = cbl.Batch(sims(0)), sims(3)
    changed = cbl.Batch(mom)
    assert changed.info() != split.info()
    for s in mom:
        s.set_option("lbm_variant", 0)
    changed.set_option("tile", 1)
    assert changed.info() == split.info()
    changed.step(3)
    changed.sync()
    for b in (changed, split):
        b.close()
