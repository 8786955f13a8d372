"""FP64 sigma_1 and adjoint energy against the oracle: states whose growth matrix is regular,
zero, of rank one, with a double largest singular value, with nearly equal ones and of a size
outside FP32's squares; box sizes around the energy kernel's grid."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import ns_oracle as O
from paper_1511_06959_gb300 import synth
from tests.test_gpu_parity import _api, dev, host, make_solver
from tests.test_oracle_primal import params_for

pytestmark = pytest.mark.gpu


def _state(kind, nx, ny, nz):
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    one = np.ones((nz, ny, nx))
    rot = np.stack([0.01 * (y - ny / 2), -0.01 * (x - nx / 2), 0 * one])
    if kind == "random":
        return synth.perturbed_uniform(nx, ny, nz, seed=96, amp=0.1)
    if kind == "uniform":
        return synth._conservative(one, np.stack([0.3 * one] * 3), one / 1.4, 1.4)
    if kind == "shear":
        return synth._conservative(one, np.stack([0.2 * np.sin(y), 0 * one, 0 * one]), one / 1.4, 1.4)
    if kind == "rotation":     # antisymmetric gradient: a double singular value away from the seam
        return synth._conservative(one, rot, one / 1.4, 1.4)
    if kind == "near":         # singular values 1e-1 to 1e-6 apart, growing from cell to cell
        d = np.logspace(-6, -1, nx * ny * nz).reshape(one.shape)
        return synth._conservative(one, rot * (1 + np.cumsum(d, axis=-1) / nx), one / 1.4, 1.4)
    # differences of 1e-16 to 1e-13 of the state: rounding noise and M below the fast path's range
    return synth.perturbed_uniform(nx, ny, nz, seed=97, amp=1e-14)


@pytest.mark.parametrize("shape", [(37, 9, 5), (40, 12, 1), (3, 2, 2)])
@pytest.mark.parametrize("kind", ["random", "uniform", "shear", "rotation", "near", "noise"])
def test_sigma1_field(kind, shape):
    api = _api()
    w = _state(kind, *shape)
    P = params_for(w)
    S = make_solver(api, w, P, 0)
    sig = torch.empty(w.shape[1:], dtype=torch.float64, device="cuda")
    S.growth_sigma1(dev(w), sig)
    ref = O.sigma1_field(w, P)
    # an entry of M is a difference of primitives of size 2 at most (u, c), each rounded a few
    # times, over 2 dx: 8 roundings a side and 25 entries give 100 eps |u| / dx; a singular
    # value moves by no more than the matrix, and its own computation adds some 20 eps sigma
    eps = 2.0 ** -53
    tol = 100 * eps * 2.0 / min(P.dx) + 20 * eps * ref
    assert np.all(np.abs(host(sig) - ref) <= tol)
    # density and pressure scaled beyond FP32: the same sigma_1
    for f in (2.0 ** -110, 2.0 ** 110):
        S.growth_sigma1(dev(f * w), sig)
        assert np.all(np.abs(host(sig) - ref) <= tol)


@pytest.mark.parametrize("shape", [(1, 1, 1), (33, 5, 2), (152, 32, 32), (153, 32, 32)])
def test_energy(shape):
    api = _api()
    w = synth.perturbed_uniform(*shape, seed=98, amp=0.1)
    lam = synth.random_field(w.shape, 99)
    P = params_for(w)
    S = make_solver(api, w, P, 0)
    E = torch.empty(1, dtype=torch.float64, device="cuda")
    S.adjoint_energy(dev(w), dev(lam), E)
    ref = O.adjoint_energy(w, lam, P)
    assert abs(E.item() - ref) < 1e-12 * ref   # as of the other sizes: a sum of squares of a dozen roundings each
