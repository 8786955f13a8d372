"""The FP64 stage kernels of 3D boxes (ns_f64.cu) against the oracle at the edges of their
tiles (32 x 4 cells) and of their split into pieces: boxes below one tile, two planes,
columns that outnumber the resident CTAs, pieces that span the end of a column; residual,
transpose with an added viscosity, step and adjoint step with a source, on cells of
unequal sides.  A reciprocal outside FP32's range takes the quotient."""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import ns_oracle as O
from paper_1511_06959_gb300 import synth
from tests.test_gpu_parity import _api, dev, host, rel_l2
from tests.test_oracle_primal import params_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 2), (2, 3, 2), (31, 3, 3), (32, 4, 5), (33, 5, 2), (65, 9, 31), (40, 37, 7)])
def test_stage_products(shape):
    api = _api()
    nx, ny, nz = shape
    w = synth.perturbed_uniform(nx, ny, nz, seed=91, amp=0.06)
    P = dataclasses.replace(params_for(w, mu=2e-2, dt=2e-3), dx=(0.1, 0.13, 0.08))
    a, s = synth.random_field(w.shape, 92), 0.05 * synth.random_field(w.shape, 93)
    nu = 1e-3 * np.abs(synth.random_field(w.shape[1:], 94))
    S = api.Solver(nx, ny, nz, P.dx, gamma=P.gamma, mu=P.mu, Pr=P.Pr, dt=P.dt, plane_i=P.plane_i, pt_in=P.pt_in)
    R, T, w1, lam0, sbar = (torch.zeros(w.shape, dtype=torch.float64, device="cuda") for _ in range(5))
    S.rhs(dev(w), R, dev(s))
    S.rhs_transpose(dev(w), dev(a), T, nu=dev(nu.astype(np.float32)))
    S.primal_step(dev(w), w1, dev(s))
    S.adjoint_step(dev(w), dev(a), lam0, s=dev(s), nu=dev(nu), sbar=sbar)
    # a few hundred roundings of 1.1e-16 on terms of the size of the result (single operators)
    assert rel_l2(host(R), O.residual(w, P, s)) < 1e-12
    ref = O.residual_transpose(w, a, P) + O.viscosity_apply(a, nu.astype(np.float32).astype(np.float64), P)
    assert rel_l2(host(T), ref) < 1e-12
    assert rel_l2(host(w1), O.rk4_step(w, P, s)[0]) < 1e-12
    lam_ref, sbar_ref = O.rk4_adjoint_step(w, a, P, s, nu)
    assert rel_l2(host(lam0), lam_ref) < 1e-12 and rel_l2(host(sbar), sbar_ref) < 1e-12
    assert S.last_error() == 0


def test_density_beyond_single_precision():
    """rho of 1e-35 and 1e+35 (FP32's normal range ends at 1.2e-38 and 3.4e38; the FP32 seed of
    the reciprocal is used well inside it): the residual scales with the state."""
    api = _api()
    w = synth.perturbed_uniform(9, 5, 3, seed=95, amp=0.05)
    S = api.Solver(9, 5, 3, 0.1, mu=0.0, dt=1e-3)
    out = []
    for f in (1.0, 2.0 ** -116, 2.0 ** 116):
        R = torch.zeros(w.shape, dtype=torch.float64, device="cuda")
        S.rhs(dev(f * w), R)
        out.append(host(R) / f)
    # inviscid: R is homogeneous of degree one; the quotient and the Newton form agree to an ulp
    assert rel_l2(out[1], out[0]) < 1e-13 and rel_l2(out[2], out[0]) < 1e-13
