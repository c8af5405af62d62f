"""Cluster training kernel: every chunk width, cluster size and number of
clusters per member, at the sizes where rows divide unevenly, against the
FP64 network.

Tolerances: a gradient entry is a sum of n products of FP32 values formed
through three 128-term contractions; its rounding error stays below 1e-4 of
the largest entry of its parameter group (the bound the gradient of small
batches is held to).  Adam divides by sqrt(v): updates whose gradient is above
1e-3 of the group's largest carry a relative error below 1e-3 per step.
"""
import numpy as np
import pytest

from oracle import mlp_oracle as M
from test_gpu_mlp import data, f32_params, lbm, members_params, shuffled  # noqa: F401

pytestmark = pytest.mark.gpu


# rows per CTA: below one, exactly 4, 5, 8, 9, 16, 17; several chunks; several
# clusters per member (one or two members, long batches); more members than
# clusters fit at once
@pytest.mark.parametrize("E,n", [(1, 1), (1, 7), (3, 64), (3, 65), (2, 128), (2, 129), (5, 257), (1, 300), (2, 1000),
                                 (1, 4099), (20, 50), (9, 700)])
def test_gradient_at_every_partition(lbm, E, n):  # noqa: F811
    flat, ps = f32_params(members_params(E, 51 + n))
    X, T = data(n, 3 + n)
    net = lbm.MLP(E)
    try:
        net.set_params(flat)
        g = net.gradient(X, T)
        assert np.array_equal(g, net.gradient(X, T))
    finally:
        net.close()
    for e in range(E):
        ref = M.backward(ps[e], X.astype(np.float64), T.astype(np.float64))
        got = M.unflatten(g[e].astype(np.float64))
        for name, _ in M.shapes():
            scale = np.abs(ref[name]).max()
            assert np.abs(got[name] - ref[name]).max() < 1e-4 * scale, (e, name)


# (40, 16): several epochs per launch; (132000, 60000): one epoch per launch
# (the row order of one epoch fills it) and several clusters per member
@pytest.mark.parametrize("n,batch,epochs", [(40, 16, 3), (132000, 60000, 3)])
def test_epochs_follow_the_shuffle(lbm, n, batch, epochs):  # noqa: F811
    lr, seed = 1e-3, 12345
    flat, _ = f32_params(members_params(1, 77))
    X, T = data(n, 19)
    net = lbm.MLP(1)
    try:
        net.set_params(flat)
        net.train(X, T, epochs=epochs, batch=batch, lr=lr, shuffle_seed=seed)
        got = net.params()[0].astype(np.float64)
    finally:
        net.close()
    p, t, state = flat[0].astype(np.float64), 0, seed
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
    d = np.abs(got - p)
    assert (~small).mean() > 0.9
    assert d[~small].max() < t * 1e-3 * lr + 1e-7, d[~small].max()
