"""Closed-form ghost pull-backs and the packed boundary cells of the bounded adjoint's
epilogue, at the sizes where the packing changes: boxes of one or two columns or rows
(a cell next to both sides), rows shorter and longer than a warp, and a ratio of specific
heats for which the characteristic ghost takes the general power."""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import ns_oracle as O
from paper_1511_06959_gb300 import synth
from tests.test_gpu_bc import BCS, FAR, WALL_E
from tests.test_gpu_parity import _api, dev, host, rel_l2
from tests.test_oracle_primal import params_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gamma", [1.4, 1.3])
@pytest.mark.parametrize("bc", list(BCS))
@pytest.mark.parametrize("shape", [(1, 4, 2), (2, 2, 1), (5, 1, 3), (3, 33, 2), (65, 3, 2)])
def test_bounded_step_and_its_adjoint_at_the_packing_edges(bc, shape, gamma):
    api = _api()
    nx, ny, nz = shape
    w = synth.perturbed_uniform(nx, ny, nz, seed=61, amp=0.05, gamma=gamma)
    P = dataclasses.replace(params_for(w, mu=0.01, dt=1e-3), gamma=gamma, bc=bc, far=FAR, wall_e=WALL_E)
    lam = synth.random_field(w.shape, 62)
    nu = 0.01 * np.abs(synth.random_field(w.shape[1:], 63))
    S = api.Solver(nx, ny, nz, P.dx, gamma=gamma, mu=P.mu, Pr=P.Pr, dt=P.dt, precision=0, plane_i=P.plane_i,
                   pt_in=P.pt_in)
    S.set_boundaries(BCS[bc], far=FAR, wall_e=WALL_E)
    w1, lam0, sbar = (torch.zeros(w.shape, dtype=torch.float64, device="cuda") for _ in range(3))
    S.primal_step(dev(w), w1)
    S.adjoint_step(dev(w), dev(lam), lam0, nu=dev(nu), sbar=sbar)
    w1_ref, _ = O.rk4_step(w, P)
    lam_ref, sbar_ref = O.rk4_adjoint_step(w, lam, P, nu=nu)
    # four stages of FP64 roundoff, a few hundred operations each, on O(1) values
    assert rel_l2(host(w1), w1_ref) < 1e-12
    assert rel_l2(host(lam0), lam_ref) < 1e-12
    assert rel_l2(host(sbar), sbar_ref) < 1e-12
    assert S.last_error() == 0
