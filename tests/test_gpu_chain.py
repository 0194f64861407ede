"""The bodies' chain over tiles: planes per block, tile lists, flag changes and batches of different instances.

FP64 against the oracle within 1e-9 (sums in another order, the bound of the moving spheres' parity test):
few bodies (a plane per block) and many (four, with tiles whose planes and rows are no multiple of a
block), moving by cells so that cells are covered and uncovered, bodies at rest, kinetics on and off, and
thresholds on both sides of 1/2. A batch of unlike instances against each of them alone: the same kernels, so
the FP32 fields differ by the order of FP64 sums only (2e-5 of the largest, the bound of the moment pass).
"""
import numpy as np
import pytest

from paper_1902_10432_gb300 import cbl, workloads

pytestmark = pytest.mark.gpu

from _pair import compare, make_pair  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    import torch

    __graft_entry__.build()
    assert torch.cuda.is_available()


def _velocities(n):
    rng = np.random.default_rng(3)
    return rng.uniform(-0.2, 0.2, size=(n, 3)), rng.uniform(-4e-3, 4e-3, size=(n, 3))


@pytest.mark.parametrize("mpf,solid,member,still", [(1, 0.05, 0.5, False), (0, 0.05, 0.5, False), (1, 0.05, 0.5, True),
                                                    (0, 0.05, 0.5, True), (1, 0.9, 0.2, False), (1, 0.3, 0.8, False)])
@pytest.mark.parametrize("many", [False, True])
def test_chain_follows_the_oracle(many, mpf, solid, member, still):
    if many:
        w, _, _ = workloads.packing(seed=1, n_spheres=14, L=62, Rmin=5.0, Rmax=8.0, prec="fp64", mpf=mpf)
    else:
        w = workloads.small_spheres(nx=41, ny=37, nz=59, R=7.0, mpf=mpf)
    for b in w.bodies:
        b["fixed"] = still
    # with kinetics the tiles span the lattice, so that the tiled field equals the oracle's dense one
    g, o = make_pair(w, options=dict(tile_tail=30.0) if mpf else None, solid_threshold=solid, member_threshold=member)
    if not still:
        V, W = _velocities(len(w.bodies))
        g.set_body_velocities(V=V, W=W)
        for k in range(len(w.bodies)):
            o.set_body_velocity(k, V[k], W[k])
    s0 = o.flags()[0]
    for _ in range(2):
        g.step(7)
        o.step(7)
        e = compare(g, o)
        assert e["flag_mismatch"] == 0
        assert e["rho"] < 1e-9 and e["vel"] < 1e-9 and e["force"] < 1e-8, e
        for k in range(len(w.bodies)):
            assert np.abs(g.phi(k) - o.phi(k)).max() < 1e-9
    assert still or (o.flags()[0] != s0).sum() > 10
    # (bit 0: a thrown body's smeared front reaches the edge of a tile of the default size, as it should report)
    assert g.info()["device_error"] & ~1 == 0


@pytest.mark.parametrize("n,gap,member,rc", [(2, -1.0, 0.5, 3.0), (12, -3.0, 0.5, 3.0), (12, -3.0, 0.2, 4.5), (9, 0.5, 0.9, 2.0)])
def test_repulsion_of_touching_spheres(n, gap, member, rc):
    # pairs in reach of a contact, several neighbours at once, tables of one to four offsets per lane
    w, _, _ = workloads.packing(seed=4, n_spheres=n, L=41, Rmin=5.0, Rmax=8.0, min_gap=gap, prec="fp64")
    g, o = make_pair(w, options=dict(tile_tail=30.0), member_threshold=member, rc=rc)
    for _ in range(2):
        g.step(1)
        o.step(1)
        rep_g, rep_o = g.body_forces()[2][:, 2, :], o.body_forces()[2][:, 2, :]
        scale = max(np.abs(rep_o).max(), 1e-300)
        assert np.abs(rep_g - rep_o).max() < 1e-9 * scale
        assert compare(g, o)["force"] < 1e-8
    assert gap > 0 or np.abs(rep_o).max() > 0


def _unlike():
    ws = [workloads.small_spheres(prec="fp32", nx=41, ny=37, nz=59, R=7.0),
          workloads.spheres2(seed=2, prec="fp32", nx=64, ny=64, nz=128, R=14.0),  # 2^19 cells: moment pass
          workloads.small_spheres(prec="fp32", nx=40, ny=36, nz=64, R=8.0, mpf=0),
          workloads.spheres2(seed=3, prec="fp32", nx=40, ny=44, nz=60, R=9.0),
          workloads.spheres2(seed=4, prec="fp32", nx=97, ny=67, nz=93, R=15.0, mpf=0)]  # ragged, moment pass
    ws[3].bodies = []
    for b in ws[2].bodies:
        b["fixed"] = True
    return ws


@pytest.mark.parametrize("copies", [1, 2])  # chains on branches (below eight instances), one launch per kernel
def test_unlike_instances_of_a_batch_step_as_alone(copies):
    def sims():
        out = []
        for w in _unlike() * copies:
            s = cbl.Sim(w.nx, w.ny, w.nz, **w.params)
            workloads.build(s, w)
            out.append(s)
        return out

    alone, many = sims(), sims()
    assert [s.get_option("lbm_variant") == 3 for s in alone] == [False, True, False, False, True] * copies
    b = cbl.Batch(many)
    b.step(20)
    b.sync()
    for a, m in zip(alone, many):
        a.step(20)
        assert np.array_equal(a.flags()[0], m.flags()[0]) and np.array_equal(a.flags()[1], m.flags()[1])
        (ra, va, _), (rm, vm, _) = a.fields(), m.fields()
        assert np.abs(rm - ra).max() < 2e-5 * np.abs(ra).max()
        assert np.abs(vm - va).max() < 4e-4 * np.abs(va).max()
        fa, fm = a.populations(), m.populations()
        assert np.abs(fm - fa).max() < 2e-5 * np.abs(fa).max()
        assert abs(a.total_mass() - m.total_mass()) < 1e-6 * a.total_mass()
        assert a.info()["device_error"] == m.info()["device_error"]
    b.close()
