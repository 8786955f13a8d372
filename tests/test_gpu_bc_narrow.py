"""Bounded boxes of rows that share a warp (up to 16 cells, padded or not), at the widths
where the number of rows per warp changes, in batches whose rows do not fill the last warp:
residual, transpose with the added viscosity and a step each way, against the oracle."""
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


@pytest.mark.parametrize("bc", list(BCS))
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("nx", [1, 2, 3, 4, 8, 10, 14, 15, 16, 17])
def test_narrow_rows(bc, prec, nx):
    api = _api()
    ny, nz, B = 7, 3, 3
    ws = [synth.perturbed_uniform(nx, ny, nz, seed=64 + b, amp=0.05) for b in range(B)]
    P = dataclasses.replace(params_for(ws[0], mu=0.01, dt=1e-3), bc=bc, far=FAR, wall_e=WALL_E)
    w, a = np.stack(ws), np.stack([synth.random_field(ws[0].shape, 70 + b) for b in range(B)])
    nu = 0.01 * np.abs(synth.random_field((B, nz, ny, nx), 75)).astype(np.float32)
    S = api.Solver(nx, ny, nz, P.dx, gamma=P.gamma, mu=P.mu, Pr=P.Pr, dt=P.dt, precision=prec, plane_i=P.plane_i,
                   pt_in=P.pt_in, batch=B)
    S.set_boundaries(BCS[bc], far=FAR, wall_e=WALL_E)
    R, T, w1, lam0, sbar = (torch.zeros(w.shape, dtype=torch.float64, device="cuda") for _ in range(5))
    S.rhs(dev(w), R)
    S.rhs_transpose(dev(w), dev(a), T, nu=dev(nu))
    S.primal_step(dev(w), w1)
    S.adjoint_step(dev(w), dev(a), lam0, nu=dev(nu), sbar=sbar)
    # as for the wider boxes: a few hundred roundings of an operator, four stages of a step
    tol = 1e-12 if prec == 0 else 2e-5
    for b in range(B):
        n64 = nu[b].astype(np.float64)
        assert rel_l2(host(R)[b], O.residual(w[b], P, None)) < tol
        assert rel_l2(host(T)[b], O.residual_transpose(w[b], a[b], P) + O.viscosity_apply(a[b], n64, P)) < tol
        assert rel_l2(host(w1)[b], O.rk4_step(w[b], P)[0]) < tol
        lam_ref, sbar_ref = O.rk4_adjoint_step(w[b], a[b], P, nu=n64)
        assert rel_l2(host(lam0)[b], lam_ref) < tol and rel_l2(host(sbar)[b], sbar_ref) < tol
    assert S.last_error() == 0
