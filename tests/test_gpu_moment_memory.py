"""The moment pass's buffers: without room for them, given back, and held by a batch."""
import numpy as np
import pytest

from paper_1902_10432_gb300 import cbl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


class Pool:
    """PyTorch's allocator up to a number of bytes."""

    def __init__(self):
        self.limit, self.used, self.sizes, self.inner = None, 0, {}, {}

    def allocator(self, device=None, stream=None):
        inner = cbl.torch_allocator_of_torch(stream=stream)

        def alloc(n, user):
            if self.limit is not None and self.used + n > self.limit:
                return None
            p = inner._keep[0](n, user)
            self.sizes[p], self.inner[p] = n, inner
            self.used += n
            return p

        def free(p, user):
            self.used -= self.sizes.pop(p)
            self.inner.pop(p)._keep[1](p, user)

        a = cbl.cbl_allocator(cbl.ALLOC_FN(alloc), cbl.FREE_FN(free), None)
        a._keep = (alloc, free, inner)
        return a


@pytest.fixture
def pool(monkeypatch):
    p = Pool()
    monkeypatch.setattr(cbl, "torch_allocator_of_torch", cbl.torch_allocator, raising=False)
    monkeypatch.setattr(cbl, "torch_allocator", p.allocator)
    return p


def _sim(variant=None):
    s = cbl.Sim(96, 64, 96, prec="fp32")  # 589 824 cells: on the moment pass by the library's choice
    if variant is not None:
        s.set_option("lbm_variant", variant)
    s.add_body("sphere", center=(48.0, 31.0, 40.0), radius=11.0, fixed=True)
    mask = np.zeros((96, 64, 96), np.uint8)
    mask[30:60, 20:50, 20:70] = 1
    s.init_fluid(1.9, 0.12, mask)
    return s


def _same(a, b, tol=1e-5):
    # two passes: FP32 rounding of another association (the bound of the free spheres against the split pass)
    for x, y in zip(a.fields()[:2], b.fields()[:2]):
        assert np.abs(x - y).max() < 10 * tol * np.abs(y).max()
    assert np.abs(a.populations() - b.populations()).max() < tol * np.abs(b.populations()).max()


@pytest.mark.parametrize("asked", [False, True])
def test_room_that_comes_later_is_used(pool, asked):
    ref = _sim(0)
    s = _sim(3 if asked else None)
    pool.limit = pool.used + (1 << 20)
    s.step(2)
    assert s.get_option("lbm_variant") == 0
    pool.limit = None
    for _ in range(20):
        s.step(1)
    assert s.get_option("lbm_variant") == 3
    ref.step(22)
    _same(s, ref)


def test_another_variant_gives_the_buffers_back(pool):
    ref, s = _sim(0), _sim()
    before = pool.used
    s.step(3)
    assert pool.used >= before + 36 * s.N
    s.set_option("lbm_variant", 0)
    assert pool.used == before
    s.step(2)
    s.set_option("lbm_variant", 3)
    s.step(2)
    s.set_option("lbm_variant", 2)
    s.step(2)
    s.set_option("lbm_variant", 3)
    s.step(2)
    s.set_option("lbm_variant", 2)
    s.step(2)
    ref.step(13)
    _same(s, ref)


def test_a_batch_keeps_them(pool):
    ref, s = _sim(0), _sim()
    b = cbl.Batch([s])
    used = pool.used
    b.step(3)
    b.sync()
    s.set_option("lbm_variant", 0)
    assert pool.used == used
    b.step(3)
    b.sync()
    ref.step(6)
    _same(s, ref)
    b.close()
    s.step(2)
    used = pool.used
    s.set_option("lbm_variant", 0)
    assert pool.used == used - 36 * s.N - 2 * 24 * 16 * 24  # a byte per brick of 4 x 4 x 4 cells, twice
    ref.step(2)
    _same(s, ref)
    # a context may go before its batch
    t = _sim()
    b = cbl.Batch([t])
    b.step(1)
    b.sync()
    t.close()
    b.close()
