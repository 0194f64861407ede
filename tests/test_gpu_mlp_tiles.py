"""The network's tiled kernels at the edges of their tiles (32 samples per block, 4 blocks per cluster, 8
blocks and 16-row groups of the window), against the FP64 reference with the same bfloat16 weights.

Bounds, derived from FP32 accumulation over sums of 64 (64 x 2^-24 = 4e-6 of the largest term, three
layers): forward 1e-4 and gradient 1e-3 of the largest value as for the kernels before them; the window's
velocity change, a sum over steps of such forces, 1e-4 of the largest change."""
import math

import numpy as np
import pytest

from oracle import mlp as ref

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def net():
    import __graft_entry__

    __graft_entry__.build()
    from paper_1902_10432_gb300 import cbl

    return cbl.MLP()


@pytest.mark.parametrize("n", [1, 31, 32, 33, 129, 4900])
def test_forward_and_gradient(net, n):
    import torch

    p = ref.init(3) + 0.02 * np.random.default_rng(1).standard_normal(ref.n_params())
    net.set_params(p)
    net.zero_grad()
    r = np.random.default_rng(n)
    x = r.standard_normal((n, 4)).astype(np.float32)
    t = r.standard_normal((n, 6)).astype(np.float32)
    xt, tt = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    y = net.forward(xt).cpu().numpy()
    yr, _ = ref.forward(ref.bf16(p), x.astype(np.float64))
    assert np.abs(y - yr).max() <= 1e-4 * max(1.0, np.abs(yr).max())
    loss = net.grad(xt, tt)
    net.grad(xt, tt, want_loss=False)  # gradients accumulate
    g = net.read_grad()
    lr, gr = ref.loss_grad(ref.bf16(p), x.astype(np.float64), t.astype(np.float64))
    assert abs(loss - lr) <= 1e-4 * lr
    assert np.abs(g - 2 * gr).max() <= 1e-3 * np.abs(2 * gr).max()


def _window64(p, w, norm, steps, dims, cth, sigma):
    """The window in numpy, FP64."""
    xm, xs, lo, hi, ym, ys = (norm[a:b].astype(np.float64) for a, b in ((0, 4), (4, 8), (8, 12), (12, 16), (16, 22), (22, 28)))
    X, V, W = w["X"].copy(), w["V"].copy(), w["W"].copy()
    pairs = w["pairs"].reshape(-1, 2)
    a, b, vl = np.r_[pairs[:, 0], pairs[:, 1]], np.r_[pairs[:, 1], pairs[:, 0]], np.r_[w["VL"], w["VL"]]
    Ra, Rb = w["R"][a], w["R"][b]
    Rs = 2 * Ra * Rb / (Ra + Rb)
    free = w["fixed"] == 0
    for _ in range(steps):
        F, T = w["bias"].copy(), np.zeros_like(X)
        if len(a):
            d = X[b] - X[a]
            d -= dims * np.rint(d / dims)
            r = np.linalg.norm(d, axis=1)
            ez = d / r[:, None]
            on = (np.abs(ez[:, 0]) < 0.9)[:, None]
            ex = np.cross(np.where(on, [[1.0, 0, 0]], [[0, 1.0, 0]]), ez)
            ex /= np.linalg.norm(ex, axis=1)[:, None]
            ey = np.cross(ez, ex)
            f = np.stack([(r - Ra - Rb) * np.sqrt(Rs / vl), np.full_like(r, cth), Ra / Rb, vl / Rs ** 3], 1)
            y = ref.forward(p, (np.clip(f, lo, hi) - xm) / xs)[0] * ys + ym
            sc = (2 * math.pi * Rs * sigma)[:, None]
            world = lambda v: ex * v[:, :1] + ey * v[:, 1:2] + ez * v[:, 2:]  # noqa: E731
            np.add.at(F, a, world(y[:, :3]) * sc)
            np.add.at(T, a, world(y[:, 3:]) * sc * Rs[:, None])
        V[free] += (F / w["M"][:, None])[free]
        X[free] = ((X + V) % dims)[free]
        W[free] += (T * w["Iinv"][:, None])[free]
    return X, V, W


# (bodies, pairs): no pair, one, rows that fill no block, several passes of 64 rows per block, and more than
# the cluster's shared memory holds (the one-block form)
@pytest.mark.parametrize("nb,npairs", [(1, 0), (2, 1), (9, 8), (67, 33), (300, 290), (2048, 1500)])
def test_window(net, nb, npairs):
    import torch

    from paper_1902_10432_gb300 import cbl

    p = ref.init(5)
    net.set_params(p)
    r = np.random.default_rng(nb)
    dims = np.array([300.0, 340.0, 280.0])
    R = r.uniform(8, 14, nb)
    X = r.uniform(0, 1, (nb, 3)) * dims
    pairs = [(k, k + 1) for k in range(npairs)]
    for i, j in pairs:
        e = r.standard_normal(3)
        X[j] = X[i] + e / np.linalg.norm(e) * (R[i] + R[j] + r.uniform(1, 5))
    M = 4 * math.pi / 3 * R ** 3 * 20.0
    w = dict(X=X % dims, V=1e-3 * r.standard_normal((nb, 3)), W=1e-4 * r.standard_normal((nb, 3)), M=M,
             Iinv=1 / (0.4 * M * R * R), R=R, fixed=(r.random(nb) < 0.2).astype(np.int32),
             bias=0.1 * r.standard_normal((nb, 3)), pairs=np.array(pairs, np.int32).reshape(-1, 2),
             VL=r.uniform(200, 800, npairs))
    norm = np.r_[[0.6, 0.7, 1.0, 0.8], [0.4, 0.1, 0.2, 0.3], [-1.0, 0.0, 0.3, 0.0], [4.0, 1.0, 3.0, 3.0],
                 [0.1, 0, -0.4, 0, 0, 0], [0.2, 0.2, 0.3, 0.05, 0.05, 0.02]].astype(np.float32)
    t = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in w.items()}
    steps = 6
    net.advance(t["X"], t["V"], t["W"], t["M"], t["Iinv"], t["R"], t["fixed"], t["bias"], t["pairs"], t["VL"], steps,
                [int(v) for v in dims], 0.7, norm, 3.583e-2)
    Xr, Vr, Wr = _window64(ref.bf16(p), w, norm, steps, dims, 0.7, 3.583e-2)
    held = w["fixed"] == 1
    for got, want, start in ((t["V"], Vr, w["V"]), (t["W"], Wr, w["W"])):
        got = got.cpu().numpy()
        assert np.array_equal(got[held], start[held])
        assert np.abs(got - want).max() <= 1e-4 * np.abs(want - start).max() + 1e-15
    d = t["X"].cpu().numpy() - Xr
    d -= dims * np.rint(d / dims)
    assert np.abs(d).max() <= 1e-4 * steps * np.abs(Vr - w["V"]).max() + 1e-12
