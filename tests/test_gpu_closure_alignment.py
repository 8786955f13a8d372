"""Closure inference on features that begin at any float of a buffer: the bits of an aligned
copy, whole tiles of 32 cells and remainders."""
import pytest

torch = pytest.importorskip("torch")

from tests.test_gpu_closure import _closure
from tests.test_gpu_parity import _api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 32, 600])
@pytest.mark.parametrize("shift", [1, 2, 3])
def test_features_at_any_float(n, shift):
    api, C = _api(), _closure()
    S = api.Solver(n, 1, 1, 0.1)
    net = C.Network(S, seed=4)
    g = torch.Generator(device="cuda").manual_seed(n)
    buf = torch.randn(16 * n + shift, device="cuda", generator=g)
    sig = torch.rand(n + 1, device="cuda", generator=g)[1:]
    nu = [torch.empty(n, device="cuda") for _ in range(2)]
    S.mlp_infer(net.blob, buf[shift:], sig, 1.0, nu[0])
    S.mlp_infer(net.blob, buf[shift:].clone(), sig, 1.0, nu[1])
    assert S.last_error() == 0 and torch.equal(*nu)
