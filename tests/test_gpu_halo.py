"""The device error's bit 0 (a phase field in the outer two layers of its tile) for bodies at rest."""
import numpy as np
import pytest

from paper_1902_10432_gb300 import cbl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("mpf", [0, 1])
@pytest.mark.parametrize("fixed", [True, False])
def test_turned_box_that_outgrows_its_tile_is_reported(mpf, fixed):
    # a long box turned by a right angle: its tile was sized along x, the field now reaches its edge along y
    s = cbl.Sim(44, 40, 36, prec="fp64", mpf_kinetics=mpf)
    s.add_body("box", center=(22.0, 20.0, 18.0), half=(10.0, 3.0, 3.0), fixed=fixed)
    s.init_fluid(1.9, 0.12)
    s.step(2)
    assert s.info()["device_error"] == 0
    c = np.sqrt(0.5)
    s.move_bodies(s.bodies()["X"], Q=np.array([[c, 0.0, 0.0, c]]), V=np.zeros((1, 3)), W=np.zeros((1, 3)))
    s.step(1)
    assert s.info()["device_error"] & 1
