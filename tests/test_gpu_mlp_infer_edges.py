"""Inference at the sizes where its paths change: ragged 128-sample tiles,
one tile per CTA and several, the mapped host path and the copying one, host
and device destinations.

GELU's packed form has an absolute error below 3e-7 (degree-6 fit 2e-9, FP32
rounding of a few operations on values up to 6), so outputs stay within the
2e-5 of the largest output that the forward pass is held to; activations far
outside the fit's range (|z| up to 1e3) follow from exp's underflow.
"""
import numpy as np
import pytest

from oracle import mlp_oracle as M
from test_gpu_mlp import data, f32_params, lbm, members_params  # noqa: F401

pytestmark = pytest.mark.gpu


def expected(ps, X):
    Y = np.stack([M.forward(p, X.astype(np.float64))[0] for p in ps])
    mu = Y.mean(axis=0)
    sd = np.sqrt(((Y - mu) ** 2).mean(axis=0))
    return mu, np.max(sd / np.abs(mu), axis=1)


@pytest.mark.parametrize("n", [1, 127, 128, 129, 4096, 4097, 20000])
def test_host_and_device_predictions_agree(lbm, n):  # noqa: F811
    import torch

    E = 3
    ps = members_params(E, 90)
    for p in ps:
        p["b4"] = p["b4"] + 1.0  # outputs around 1, as the surrogate's
    flat, ps = f32_params(ps)
    X, _ = data(n, 91)
    net = lbm.MLP(E)
    try:
        net.set_params(flat)
        mean, spread = net.predict(X)
        xd = torch.from_numpy(X).cuda()
        md, sd = torch.empty(n, 2, device="cuda"), torch.empty(n, device="cuda")
        net.predict_device(xd.data_ptr(), n, md.data_ptr(), sd.data_ptr())
    finally:
        net.close()
    assert np.array_equal(mean, md.cpu().numpy()) and np.array_equal(spread, sd.cpu().numpy())
    mu, sp = expected(ps, X)
    assert np.abs(mean - mu).max() < 2e-5 * np.abs(mu).max()
    assert np.abs(spread - sp).max() < 2e-5 * max(1.0, sp.max()) + 1e-4 * sp.max()


@pytest.mark.parametrize("scale", [1e-3, 30.0, 300.0])
def test_activations_far_from_the_usual_range(lbm, scale):  # noqa: F811
    flat, ps = f32_params(members_params(2, 95))
    X, _ = data(200, 96)
    X = (X * scale).astype(np.float32)
    net = lbm.MLP(2)
    try:
        net.set_params(flat)
        Y = net.forward(X)
        X[7, 2] = np.nan
        bad = net.forward(X)
    finally:
        net.close()
    for e in range(2):
        ref, _ = M.forward(ps[e], np.where(np.isnan(X), 0.0, X).astype(np.float64))
        keep = np.arange(200) != 7
        assert np.abs(Y[e][keep] - ref[keep]).max() < 2e-5 * np.abs(ref).max()
        assert np.isnan(bad[e, 7]).all() and np.array_equal(bad[e][keep], Y[e][keep])
