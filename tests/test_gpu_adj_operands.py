"""The adjoint step's outermost operands (FP64 adjoint, source sensitivity), read ahead of their
use: with a sensitivity already accumulated the step adds exactly what it adds to zero, and the
adjoint keeps its bits with and without one, at the edges of the tiles and ranges of each
kernel (32 x 8 and 32 x 4 marching tiles, one- and four-row 2D tiles)."""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1511_06959_gb300 import synth
from tests.test_gpu_parity import _api, dev, host
from tests.test_oracle_primal import params_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flux", [0, 1])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("shape", [(1, 1, 2), (33, 9, 3), (31, 7, 40), (33, 1, 1), (40, 37, 1), (64, 160, 1)])
def test_accumulated_sensitivity(shape, prec, flux):
    api = _api()
    nx, ny, nz = shape
    w = synth.perturbed_uniform(nx, ny, nz, seed=61, amp=0.05)
    P = dataclasses.replace(params_for(w), dx=(0.1, 0.13, 0.08), dt=2e-3)
    S = api.Solver(nx, ny, nz, P.dx, gamma=P.gamma, mu=P.mu, Pr=P.Pr, dt=P.dt, plane_i=P.plane_i, pt_in=P.pt_in,
                   precision=prec, flux=flux)
    lam, s = dev(synth.random_field(w.shape, 62)), dev(0.05 * synth.random_field(w.shape, 63))
    X = synth.random_field(w.shape, 64)
    l0, l1, l2 = (torch.zeros(w.shape, dtype=torch.float64, device="cuda") for _ in range(3))
    s0, s1 = torch.zeros_like(l0), dev(X)
    S.adjoint_step(dev(w), lam, l0, s=s, sbar=s0)
    S.adjoint_step(dev(w), lam, l1, s=s, sbar=s1)
    S.adjoint_step(dev(w), lam, l2, s=s)
    assert np.array_equal(host(l0), host(l1)) and np.array_equal(host(l0), host(l2))
    # one addition, X + sum; FP64 may contract the sum's last product into it (one rounding less)
    if prec == 1:
        assert np.array_equal(host(s1), X + host(s0))
    else:
        assert np.all(np.abs(host(s1) - (X + host(s0))) <= 2.0 ** -52 * (np.abs(X) + np.abs(host(s0))))
    assert S.last_error() == 0
