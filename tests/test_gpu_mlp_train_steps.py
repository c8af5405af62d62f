"""Launches of many Adam steps with wider and several chunks per step: batches of
8- and 16-row chunks and of two and three 16-row chunks, the last with rows that
divide unevenly over the CTAs of a cluster, every member against the FP64
replay.  Tolerance as for the shorter chunks: updates whose gradient is above
1e-3 of its group's largest carry a relative error below 1e-3 per step."""
import numpy as np
import pytest

from oracle import mlp_oracle as M
from test_gpu_mlp import data, f32_params, lbm, members_params, shuffled  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E,n,batch", [(5, 400, 128), (5, 650, 200), (5, 1600, 512), (5, 1600, 531), (2, 700, 230)])
def test_several_steps_per_launch(lbm, E, n, batch):  # noqa: F811
    lr, seed, epochs = 1e-3, 4242, 2
    flat, ps = f32_params(members_params(E, 61))
    X, T = data(n, 23)
    net = lbm.MLP(E)
    try:
        net.set_params(flat)
        net.train(X, T, epochs=epochs, batch=batch, lr=lr, shuffle_seed=seed)
        got = net.params().astype(np.float64)
    finally:
        net.close()
    for e in range(E):
        p, t, state = flat[e].astype(np.float64), 0, seed
        m, v, small = np.zeros_like(p), np.zeros_like(p), np.zeros(p.size, dtype=bool)
        for _ in range(epochs):
            perm, state = shuffled(n, state)
            for b0 in range(0, n - batch + 1, batch):
                rows, t = perm[b0:b0 + batch], t + 1
                g = M.flatten(M.backward(M.unflatten(p), X[rows].astype(np.float64), T[rows].astype(np.float64)))
                off = 0
                for _, shp in M.shapes():
                    k = int(np.prod(shp))
                    seg = np.abs(g[off:off + k])
                    small[off:off + k] |= seg < 1e-3 * seg.max()
                    off += k
                p, m, v = M.adam_step(p, g, m, v, t, lr=lr)
        d = np.abs(got[e] - p)
        assert t >= 6 and (~small).mean() > 0.9
        assert d[~small].max() < t * 1e-3 * lr + 1e-7, (e, d[~small].max())
