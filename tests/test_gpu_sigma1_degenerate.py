"""FP64 sigma_1 of flows whose largest singular values coincide or nearly do: solid rotation, in
the plane and about an oblique axis, with noise from the rounding level up, and with an
expansion that brings a third value near, against singular values from numpy."""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import ns_oracle as O
from paper_1511_06959_gb300 import synth
from tests.test_gpu_parity import _api, dev, host, make_solver
from tests.test_oracle_primal import params_for

pytestmark = pytest.mark.gpu


NOISE = (0.0, 1e-15, 1e-12, 1e-7, 1e-4, 1e-3)
CASES = ([((512, 512, 1), 0.0, False)] + [((160, 160, 1), n, False) for n in NOISE] +
         [((48, 40, 24), n, o) for n in NOISE for o in (False, True)])


@pytest.mark.parametrize("shape,noise,oblique", CASES)
def test_solid_rotation(shape, noise, oblique):
    api = _api()
    nx, ny, nz = shape
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    r = np.stack([x - nx / 2, y - ny / 2, z - nz / 2])
    om = 0.64 / ny * np.array([0.3, -0.5, 1.0] if oblique else [0.0, 0.0, 1.0])
    u = np.stack([om[1] * r[2] - om[2] * r[1], om[2] * r[0] - om[0] * r[2], om[0] * r[1] - om[1] * r[0]])
    u += noise * np.random.default_rng(5).standard_normal(u.shape)
    one = np.ones((nz, ny, nx))
    w = synth._conservative(one, u, one / 1.4, 1.4)
    P = params_for(w)
    S = make_solver(api, w, P, 0)
    sig = torch.empty(w.shape[1:], dtype=torch.float64, device="cuda")
    S.growth_sigma1(dev(w), sig)
    ref = O.sigma1_field(w, P)
    # as for the other states: a singular value moves by no more than the matrix, whose entries
    # are differences over 2 dx of primitives of size 2 at most (100 roundings in all), and its
    # own computation adds some 20 eps sigma; 1e-13 sigma more for the coupling of a pair that
    # lies within 1e-14 and for the reference
    eps = 2.0 ** -53
    assert np.all(np.abs(host(sig) - ref) <= 100 * eps * 2.0 / min(P.dx) + 20 * eps * ref + 1e-13 * ref)
    assert S.last_error() == 0


@pytest.mark.parametrize("delta", [0.0, 1e-6, 1e-5, 1e-4, -1e-4, 1e-3, -1e-3, 3e-3, 1e-2])
@pytest.mark.parametrize("noise", [1e-9, 3e-7, 1e-5])
def test_three_singular_values_together(delta, noise):
    """Rotation with expansion at the rate that puts the double singular value of the rotation
    within delta of that of the density and pressure rows, and noise about the pair's gap."""
    api = _api()
    nx, ny, nz, dx = 64, 48, 40, 0.1
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    r = dx * np.stack([x - nx / 2, y - ny / 2, z - nz / 2])
    e = 0.05
    top = np.linalg.norm([[1.5 * e, -1.5 * np.sqrt(0.4) * e], [0.0, 0.9 * e]], 2)
    om = np.sqrt((top * (1 + delta)) ** 2 - 0.25 * e * e) * np.array([0.6, 0.0, 0.8])
    u = e * r + np.stack([om[1] * r[2] - om[2] * r[1], om[2] * r[0] - om[0] * r[2], om[0] * r[1] - om[1] * r[0]])
    u += noise * dx * e * np.random.default_rng(6).standard_normal(u.shape)
    one = np.ones((nz, ny, nx))
    w = synth._conservative(one, u, one / 1.4, 1.4)
    P = dataclasses.replace(params_for(w), dx=(dx,) * 3)
    S = make_solver(api, w, P, 0)
    sig = torch.empty(w.shape[1:], dtype=torch.float64, device="cuda")
    S.growth_sigma1(dev(w), sig)
    ref = O.sigma1_field(w, P)
    # the general iteration resolves a triple root of a polynomial to the third root of its
    # rounding, 4.8e-6 of sigma^2
    assert np.all(np.abs(host(sig) - ref) <= 2.4e-6 * ref)
