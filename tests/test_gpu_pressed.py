"""Bodies pressed into each other within a third one's rim: the sum of the phases is above 1 where a third field
vanishes (the kinetics leaves values around 0 on every rim), so that clamping, rescaling and the ownership
of a cell meet. FP64 against the oracle within 1e-9 (the bound of the chain's tests)."""
import numpy as np
import pytest

from paper_1902_10432_gb300 import workloads

pytestmark = pytest.mark.gpu

from _pair import compare, make_pair  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("mpf", [1, 0])
@pytest.mark.parametrize("side", [9.0, 11.0, 13.5])  # of the triangle of centres; R = 6, rims of 2.5 cells
def test_three_pressed_bodies_follow_the_oracle(side, mpf):
    w = workloads.small_spheres(nx=36, ny=34, nz=38, R=6.0, gap=1.0, mpf=mpf, mobility=2e-3)
    proto = w.bodies[0]
    h = side * np.sqrt(3.0) / 2.0
    # (not symmetric about the axes, so that no two phases tie)
    centres = [(10.3, 11.2, 18.1), (10.3 + side, 11.4, 18.9), (10.1 + side / 2, 11.3 + h, 19.2),
               (10.2 + side / 2, 11.1 + h / 3, 18.3 + 0.8 * side)]
    w.bodies = [dict(proto, center=c) for c in centres]
    w.mask[:] = 0
    w.mask[26:32] = 1
    g, o = make_pair(w, options=dict(tile_tail=30.0))
    for _ in range(3):
        g.step(2)
        o.step(2)
        for k in range(4):
            assert np.abs(g.phi(k) - o.phi(k)).max() < 1e-9
        e = compare(g, o)
        assert e["flag_mismatch"] == 0 and e["rho"] < 1e-9 and e["force"] < 1e-8, e
    phi = np.array([o.phi(k) for k in range(4)])
    assert ((phi > 1e-9).sum(0) >= 3).sum() > 10  # cells where three fields meet
