"""The stage kernels' split of the planes among CTAs, driven through all its forms on small
boxes by the number of resident slots (NS_RHS_CTAS, NS_ADJ_CTAS): FP64 pieces of several whole
columns, that end inside a column, begin in the gap between two or span a column's end; FP32
pieces with the columns' second parts, whole waves of one or more ranges per column, even
ranges down to single planes.  Every form gives the bits of the default one, which agrees with
the oracle."""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import ns_oracle as O
from paper_1511_06959_gb300 import synth
from tests.test_gpu_parity import _api, dev, host, rel_l2
from tests.test_oracle_primal import params_for

pytestmark = pytest.mark.gpu

# columns of 32 x 4 (FP64) and 32 x 8 cells (FP32): 9 and 6; 20 and 10 a box; 10 and 6; 4 and 2
SHAPES = [((65, 9, 31), 1), ((40, 37, 7), 2), ((33, 17, 64), 1), ((33, 5, 2), 3)]
# FP32: pieces of (33, 17, 64) at 48, 77 and 96 slots (6 columns <= n / 8, 384 planes >= 4 n), whole
# waves below the columns' number, even ranges between
SLOTS = [1, 2, 3, 5, 7, 11, 24, 48, 77, 96, 300]


def _outputs(api, S, w, a, s, nu):
    out = [torch.zeros(w.shape, dtype=torch.float64, device="cuda") for _ in range(5)]
    S.rhs(w, out[0], s)
    S.rhs_transpose(w, a, out[1], nu=nu)
    S.primal_step(w, out[2], s)
    S.adjoint_step(w, a, out[3], s=s, nu=nu, sbar=out[4])
    assert S.last_error() == 0
    return out


@pytest.mark.parametrize("shape,batch", SHAPES)
@pytest.mark.parametrize("prec", [0, 1])
def test_every_split_gives_the_same_bits(shape, batch, prec, monkeypatch):
    api = _api()
    nx, ny, nz = shape
    ws = [synth.perturbed_uniform(nx, ny, nz, seed=171 + b, amp=0.06) for b in range(batch)]
    P = dataclasses.replace(params_for(ws[0], mu=2e-2, dt=2e-3), dx=(0.1, 0.13, 0.08))
    w, a = np.stack(ws), np.stack([synth.random_field(ws[0].shape, 181 + b) for b in range(batch)])
    s = 0.05 * synth.random_field(w.shape, 191)
    nu = 1e-3 * np.abs(synth.random_field((batch, nz, ny, nx), 192)).astype(np.float32)
    S = api.Solver(nx, ny, nz, P.dx, gamma=P.gamma, mu=P.mu, Pr=P.Pr, dt=P.dt, precision=prec, plane_i=P.plane_i,
                   pt_in=P.pt_in, batch=batch)
    args = [dev(x) for x in (w, a, s, nu)]
    ref = _outputs(api, S, *args)
    # single operators and steps: roundings of FP64 (a few hundred) and of FP32
    tol = 1e-12 if prec == 0 else 2e-5
    for b in range(batch):
        n64 = nu[b].astype(np.float64)
        lam, sb = O.rk4_adjoint_step(w[b], a[b], P, s[b], n64)
        want = [O.residual(w[b], P, s[b]), O.residual_transpose(w[b], a[b], P) + O.viscosity_apply(a[b], n64, P),
                O.rk4_step(w[b], P, s[b])[0], lam, sb]
        for x, y in zip(ref, want):
            assert rel_l2(host(x)[b], y) < tol
    for n in SLOTS:
        monkeypatch.setenv("NS_RHS_CTAS", str(n))
        monkeypatch.setenv("NS_ADJ_CTAS", str(n))
        for i, (x, y) in enumerate(zip(_outputs(api, S, *args), ref)):
            assert torch.equal(x, y), (n, i)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n", [2, 7, 48, 77])
def test_splits_with_the_roe_flux(prec, n, monkeypatch):
    """The Roe kernels' splits against the oracle (their FP32 bits depend on the cuts)."""
    api = _api()
    w = synth.perturbed_uniform(33, 17, 64, seed=173, amp=0.06)
    P = dataclasses.replace(params_for(w, mu=2e-2, dt=2e-3), flux="roe", roe_delta=0.1)
    a = synth.random_field(w.shape, 174)
    S = api.Solver(33, 17, 64, P.dx, gamma=P.gamma, mu=P.mu, Pr=P.Pr, dt=P.dt, precision=prec, plane_i=P.plane_i,
                   pt_in=P.pt_in, flux=1, roe_delta=0.1)
    monkeypatch.setenv("NS_RHS_CTAS", str(n))
    monkeypatch.setenv("NS_ADJ_CTAS", str(n))
    R, T = (torch.zeros(w.shape, dtype=torch.float64, device="cuda") for _ in range(2))
    S.rhs(dev(w), R)
    S.rhs_transpose(dev(w), dev(a), T)
    tol = 1e-12 if prec == 0 else 2e-5
    assert rel_l2(host(R), O.residual(w, P, None)) < tol
    assert rel_l2(host(T), O.residual_transpose(w, a, P)) < tol
    assert S.last_error() == 0
