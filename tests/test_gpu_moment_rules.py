"""Where the moment pass runs by default, and what a state on it gives to its readers right after a step."""
import numpy as np
import pytest

from paper_1902_10432_gb300 import autotune, cbl, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    import torch

    __graft_entry__.build()
    assert torch.cuda.is_available()


def _sim(w, variant=None, **kw):
    s = cbl.Sim(w.nx, w.ny, w.nz, **dict(w.params, **kw))
    if variant is not None:
        s.set_option("lbm_variant", variant)
    workloads.build(s, w)
    return s


def test_binary16_default_gives_the_bits_of_the_other_passes():
    # 2^19 cells, held bodies (no order of FP64 sums in the result); the first rounding that differs is carried on
    # by the flow, so 60 steps and equality
    w = workloads.spheres2(seed=2, prec="fp16dev", nx=64, ny=64, nz=128, R=14.0)
    for b in w.bodies:
        b["fixed"] = True
    a, b = _sim(w), _sim(w, 0)
    assert a.get_option("lbm_variant") == 0
    batch = cbl.Batch([_sim(w) for _ in range(2)])
    for s in (a, b, batch):
        s.step(60)
    batch.sync()
    for s in [a] + batch.sims:
        assert np.array_equal(s.populations(), b.populations())
        assert np.array_equal(s.fields()[1], b.fields()[1])
    batch.close()
    assert all(c["lbm_variant"] != 3 for c in autotune.candidates("fp16dev"))
    assert _sim(workloads.spheres2(seed=2, prec="fp32", nx=64, ny=64, nz=128, R=14.0)).get_option("lbm_variant") == 3


@pytest.mark.parametrize("copies", [1, 3])  # chains on branches (below eight instances), one launch per kernel
def test_instances_without_bodies_beside_those_with(copies):
    # a fluid without bodies on each pass beside pairs of spheres: every instance ends its step once
    def sims():
        ws = []
        for k in range(copies):
            ws += [workloads.spheres2(seed=2, prec="fp32", nx=64, ny=64, nz=128, R=14.0),
                   workloads.spheres2(seed=3, prec="fp32", nx=64, ny=64, nz=128, R=14.0),
                   workloads.small_spheres(prec="fp32")]
            ws[-2].bodies = []
            if k == 1:
                ws[-1].bodies = []
        return [_sim(w) for w in ws]

    alone, many = sims(), sims()
    assert {(s.nb == 0, s.get_option("lbm_variant")) for s in alone} >= {(True, 3), (False, 3), (False, 0)}
    b = cbl.Batch(many)
    b.step(7)
    b.step(4)
    b.sync()
    for a, m in zip(alone, many):
        a.step(11)
        # the same kernels: equal up to the order of FP64 sums (the bounds of the batch of unlike instances)
        for x, y in zip(a.fields()[:2], m.fields()[:2]):
            assert np.abs(x - y).max() < 4e-4 * np.abs(x).max()
        assert np.abs(a.populations() - m.populations()).max() < 2e-5 * np.abs(a.populations()).max()
        assert abs(a.total_mass() - m.total_mass()) < 1e-6 * a.total_mass()
    b.close()


def _rel(a, b):
    fine = np.isfinite(b)  # a cell that a thrown body uncovers starts empty: its velocity may overflow, on both sides alike
    assert np.array_equal(fine, np.isfinite(a))
    return float(np.abs(a[fine] - b[fine]).max() / np.abs(b[fine]).max())


@pytest.mark.parametrize("batch", [False, True])
def test_populations_right_after_a_body_has_jumped(batch, tmp_path):
    # seven cells in one step: the step writes all populations before the refill and no brick says so. What a
    # reader gets right after it is the split pass's, with the refill in it, and reading, saving and loading
    # change nothing of what follows. (1e-4: the bound of the thrown sphere's test, which takes as many steps
    # after it: the cells that it uncovers start empty and blow up on every pass. 1e-9: the order of FP64 sums.)
    w = workloads.small_spheres(prec="fp32", mobility=2e-3)
    split, read, quiet = (_sim(w, v) for v in (0, 3, 3))
    fill = [_sim(w, 3) for _ in range(7)] if batch else []

    def step(s, n):
        b = cbl.Batch([s] + fill) if batch and s is not split else s
        b.step(n)
        if b is not s:
            b.sync()
            b.close()

    for s in (split, read, quiet):
        step(s, 3)
        s.set_body_velocities(V=np.array([[0.0, 0.0, -7.0], [0.0, 0.0, 0.0]]), W=np.zeros((2, 3)))
        step(s, 1)
    f = read.populations()
    assert _rel(f, split.populations()) < 1e-4
    assert abs(f.sum() - split.populations().sum()) < 1e-6 * f.sum()  # the refill hands over what was covered
    path = str(tmp_path / "jumped.ckpt")
    read.save(path)
    loaded = cbl.Sim(w.nx, w.ny, w.nz, **w.params)
    loaded.set_option("lbm_variant", 3)
    for b in w.bodies:
        bk = dict(b)
        loaded.add_body(bk.pop("shape"), **bk)
    loaded.load(path)
    for s in (split, read, quiet, loaded):
        s.set_body_velocities(V=np.zeros((2, 3)), W=np.zeros((2, 3)))
        step(s, 2)
    g = quiet.populations()
    assert _rel(read.populations(), g) < 1e-9
    assert _rel(loaded.populations(), g) < 1e-9
    assert _rel(g, split.populations()) < 1e-4
