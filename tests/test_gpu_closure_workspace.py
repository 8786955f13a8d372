"""ns_workspace_bytes counts the training scratch: that of 4096 samples from the start, the
scratch of a larger minibatch once it has been used, the largest alone after several."""
import pytest

torch = pytest.importorskip("torch")

from tests.test_gpu_closure import _closure
from tests.test_gpu_parity import _api

pytestmark = pytest.mark.gpu


def test_workspace_counts_the_training_scratch():
    api, C = _api(), _closure()
    S = api.Solver(8, 8, 1, 0.1, precision=1)
    # partial gradients of a cluster of 4 x 32 samples (5185 parameters), a loss per sample
    floats = lambda n: -(-n // 128) * (api.NS_MLP_PARAMS + 128) + 16
    # nine stage fields, the reductions' partials (at most 296 x 256 doubles and a few), an error word
    base = S.workspace_bytes()
    assert base >= 9 * 5 * 64 * 4 + 296 * 256 * 8 + 4 * floats(4096)
    net = C.Network(S)
    feat = torch.zeros((300, 16), dtype=torch.float32, device="cuda")
    target = torch.ones(300, dtype=torch.float32, device="cuda")
    step = 0
    for n, extra in ((4096, 0), (4097, floats(4097)), (1000, floats(4097)), (9000, floats(9000)), (5000, floats(9000))):
        step += 1
        S.mlp_train_step(net.blob, feat, target, torch.zeros(n, dtype=torch.int32, device="cuda"), step, 1e-3)
        assert S.workspace_bytes() == base + 4 * extra
