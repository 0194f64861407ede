"""A body's centre given many lattice lengths outside is its periodic image's."""
import numpy as np
import pytest

from paper_1902_10432_gb300 import workloads

pytestmark = pytest.mark.gpu

from _pair import make_pair  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("lengths", [(0, 0, 0), (-1, 1, 2), (5, -7, 3), (-400, 900, -3000)])
def test_centre_far_outside(lengths):
    # against the oracle, whose dense fields know no tiles, with the bodies where they are
    w = workloads.small_spheres(prec="fp64")
    _, o = make_pair(w)
    far = workloads.small_spheres(prec="fp64")
    for b in far.bodies:
        b["center"] = tuple(c + k * n for c, k, n in zip(b["center"], lengths, (w.nx, w.ny, w.nz)))
    f, _ = make_pair(far)
    for s in (f, o):
        s.step(5)
    assert f.info()["device_error"] == 0
    assert np.array_equal(f.flags()[1], o.flags()[1])
    # (an offset of the centre of 1e5 cells leaves its place 1e-11 of a cell)
    assert np.abs(f.phi(0) - o.phi(0)).max() < 1e-9
    assert np.abs(f.fields()[0] - o.fields()[0]).max() < 1e-9 * np.abs(o.fields()[0]).max()
    assert np.abs(f.bodies()["X"] - o.bodies()["X"]).max() < 1e-9
