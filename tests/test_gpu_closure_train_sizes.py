"""One training step at the minibatch sizes where its chunking changes: one sample, a
partial chunk of 32, whole chunks, a partial cluster of four, many clusters; the gradient
(first Adam moment), loss and published inference weights against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp_oracle as ML
from tests.test_gpu_closure import _closure
from tests.test_gpu_parity import _api, dev, host, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 32, 33, 128, 129, 5000])
def test_training_step_sizes(n):
    api, C = _api(), _closure()
    rng = np.random.default_rng(n)
    feat = np.zeros((600, 16), dtype=np.float32)
    feat[:, :14] = rng.standard_normal((600, 14)).astype(np.float32)
    target = np.abs(rng.standard_normal(600)).astype(np.float32)
    idx = rng.integers(0, 600, size=n).astype(np.int32)
    p = ML.init_params(8)
    S = api.Solver(8, 8, 1, 0.1)
    net = C.Network(S, p)
    loss = torch.empty(1, dtype=torch.float32, device="cuda")
    S.mlp_train_step(net.blob, dev(feat), dev(target), dev(idx), 1, 1e-3, loss)
    m = torch.empty(api.NS_MLP_PARAMS, dtype=torch.float32, device="cuda")
    S.mlp_get_moment(net.blob, 1, m)
    p64 = {k: np.asarray(v, dtype=np.float64) for k, v in p.items()}
    L, g = ML.loss_and_grads(p64, feat[idx, :14].astype(np.float64), target[idx].astype(np.float64), True,
                             bf16_backward=True)
    # a BF16 value may round the other way after FP32 accumulation: 2^-9 of one operand of
    # some of a gradient's products
    assert abs(loss.item() - L) < 1e-3 * L
    assert rel_l2(host(m).astype(np.float64) / 0.1, C.pack(g).astype(np.float64)) < 2 ** -9
    # the published weights are those of the updated master copy: inference with the trained
    # blob equals inference with a blob set to its parameters
    out = torch.empty(api.NS_MLP_PARAMS, dtype=torch.float32, device="cuda")
    S.mlp_get_params(net.blob, out)
    other = torch.zeros_like(net.blob)
    S.mlp_set_params(other, out)
    sig = torch.ones(600, dtype=torch.float32, device="cuda")
    nu = [torch.empty_like(sig) for _ in range(2)]
    big = api.Solver(600, 1, 1, 0.1)
    for b, o in zip((net.blob, other), nu):
        big.mlp_infer(b, dev(feat), sig, 1.0, o)
    assert torch.equal(*nu)
