"""One training step of a network whose second layer sits at z = -13.3, where gelu' is
2e-38 and its exponential subnormal: the gradient of that layer's biases (first Adam moment)
against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp_oracle as ML
from tests.test_gpu_closure import _closure
from tests.test_gpu_parity import _api, dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("z", [-13.3, -13.25, -13.9])
def test_gradient_through_a_subnormal_exponential(z):
    api, C = _api(), _closure()
    p = {"W1": np.zeros((14, 64)), "b1": np.zeros(64), "W2": np.zeros((64, 64)),
         "b2": np.full(64, np.float32(z), dtype=np.float64), "w3": np.ones(64), "b3": np.array(5.0)}
    S = api.Solver(8, 8, 1, 0.1)
    net = C.Network(S, p)
    feat = np.zeros((8, 16), dtype=np.float32)
    target = np.full(8, 1e6, dtype=np.float32)
    S.mlp_train_step(net.blob, dev(feat), dev(target), dev(np.zeros(1, dtype=np.int32)), 1, 1e-3)
    m = torch.empty(api.NS_MLP_PARAMS, dtype=torch.float32, device="cuda")
    S.mlp_get_moment(net.blob, 1, m)
    got = C.unpack(host(m))["b2"] / 0.1
    _, g = ML.loss_and_grads(p, np.zeros((1, 14)), target[:1].astype(np.float64))
    # the exponent, some -90, is formed in FP32: 6e-8 of it, 5e-6; a subnormal exponential
    # has at least 3 digits down to 1e-42 (z = -13.9: 1.1e-42, 780 units of the last place)
    assert np.all(np.abs(got / g["b2"] - 1) < 2e-3) and np.all(g["b2"] != 0)
