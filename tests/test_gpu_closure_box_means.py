"""The box means behind the closure's features: as exact as FP64 sums where the terms cancel,
finite where a float sum would overflow, a box smaller than a warp."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp_oracle as ML
from paper_1511_06959_gb300 import synth
from tests.test_gpu_parity import _api, dev, host, rel_l2
from tests.test_oracle_primal import params_for

pytestmark = pytest.mark.gpu


def _features(api, w, prec):
    S = api.Solver(*w.shape[:0:-1], 0.1, precision=prec)
    feat = torch.empty((w[0].size, 16), dtype=torch.float32, device="cuda")
    S.mlp_features(dev(w), feat)
    return host(feat)


@pytest.mark.parametrize("prec", [0, 1])
def test_cancelling_terms(prec):
    """u1 by plane: 2^28, 4 + 2^-21, 2^-23, -2^28, 1, 1, 1, 1 (rho 1): the mean is 1 + 2^-24 +
    2^-26, above the middle of two floats, so the mean as a float is 1 + 2^-23.  Sums in float
    pairs lose the 2^-23 beside 4 (half of whose float spacing is 2^-22) while the pair's high
    part holds 2^28, and give the middle, which rounds to 1.  FP64 holds every partial sum of
    a plane set (2^28 to 2^-23) exactly."""
    api = _api()
    u = np.array([2.0 ** 28, 4 + 2.0 ** -21, 2.0 ** -23, -2.0 ** 28, 1, 1, 1, 1])
    # energies whose pressure is positive in FP32 at every plane
    E = 2.5 + 0.5 * u * u + np.where(np.abs(u) > 1e3, 2.0 ** 32, 0.0)
    # 296 blocks of 256 threads: a plane of 296 x 256 cells gives every thread one cell of each
    w = np.zeros((5, 8, 256, 296))
    w[0] = 1.0
    w[1] = u[:, None, None]
    w[4] = E[:, None, None]
    f = _features(api, w, prec).reshape(8, -1, 16)
    p = 0.4 * (E - 0.5 * u * u)
    icb = 1.0 / np.sqrt(1.4 * p.mean())
    ref = -2.0 ** -23 * icb
    # 1 - (1 + 2^-23) is exact; 1 / c_bar has FP32 roundings
    assert np.allclose(f[4:, :, 1], ref, rtol=1e-5, atol=0)


@pytest.mark.parametrize("prec", [0, 1])
def test_sums_beyond_single_precision(prec):
    """rho = p = 1e38 at rest, eight cells a thread: a thread's float sum overflows.  The mean is
    the cells' value, to FP64 rounding, so all features vanish but for FP32 roundings of it."""
    api = _api()
    w = np.zeros((5, 8, 256, 296))
    w[0] = 1e38
    w[4] = 2.5e38
    f = _features(api, w, prec)
    assert np.isfinite(f).all() and np.abs(f).max() < 1e-6


@pytest.mark.parametrize("shape", [(1, 1, 1), (5, 3, 2), (37, 9, 5)])
@pytest.mark.parametrize("prec", [0, 1])
def test_small_boxes(shape, prec):
    api = _api()
    w = synth.perturbed_uniform(*shape, seed=84, amp=0.05)
    P = params_for(w)
    S = api.Solver(*shape, P.dx, gamma=P.gamma, precision=prec)
    feat = torch.empty((w[0].size, 16), dtype=torch.float32, device="cuda")
    S.mlp_features(dev(w), feat)
    ref = ML.features(w, P)
    # FP32 primitives (6e-8 each, a dozen roundings) differenced over 2 dx or from the mean
    assert np.abs(host(feat)[:, :14] - ref).max() < 12 * 6e-8 * 2 / min(P.dx)
