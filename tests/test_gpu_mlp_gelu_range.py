"""GELU of pre-activations whose double overflows FP32: the activation is the
pre-activation itself (positive side) or zero, on both inference paths, so the
outputs stay at the forward pass's bound of 2e-5 of the largest."""
import numpy as np
import pytest

from oracle import mlp_oracle as M
from test_gpu_mlp import f32_params, lbm, members_params  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("path", ["simt", "tensor"])
def test_huge_finite_activations(lbm, path):  # noqa: F811
    ps = members_params(2, 97)
    for p in ps:
        p["W1"][3] = [1.5 * 2.0 ** 127, 0.0, 0.0, 0.0]  # z = +-2.55e38 in sample 0 / 1
        p["W2"][:, 3] = 2.0 ** -123                      # exact in TF32: contributes 24 to every neuron
    flat, ps = f32_params(ps)
    X = np.array([[1.0, 0.3, -0.2, 0.1], [-1.0, 0.3, -0.2, 0.1], [0.0, 0.5, 0.4, -0.7]], dtype=np.float32)
    net = lbm.MLP(2)
    try:
        net.set_params(flat)
        net.set_infer_path(path)
        Y = net.forward(X)
    finally:
        net.close()
    assert np.isfinite(Y).all()
    for e in range(2):
        ref, _ = M.forward(ps[e], X.astype(np.float64))
        assert np.abs(Y[e] - ref).max() < 2e-5 * np.abs(ref).max()
