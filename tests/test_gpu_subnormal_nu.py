"""An added viscosity of subnormal size (1e-39) given as floats: on a state at rest with no
viscosity of its own and an adjoint alternating from plane to plane, the transposed residual
inside is the added viscosity's term alone, periodic and bounded."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from tests.test_gpu_parity import _api, dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bc", [0, 1, 2, 3])
@pytest.mark.parametrize("nz", [1, 4])
def test_subnormal_viscosity(bc, nz):
    api = _api()
    nx, ny, dx = 16, 12, 0.5
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    w = np.zeros((5, nz, ny, nx))
    w[0], w[4] = 1.0, 2.5
    # rho component only: its central differences vanish inside, and the others are zero
    a = np.zeros_like(w)
    a[0] = (-1.0) ** x
    nu = np.full((nz, ny, nx), 1e-39, dtype=np.float32)
    S = api.Solver(nx, ny, nz, dx, mu=0.0)
    S.set_viscosity_split(1.0, 1.0, 1.0)
    if bc:
        S.set_boundaries(bc, far=(1.0, 0.1, 0.0, 0.0, 1.0), wall_e=(2.5, 2.5))
    out = torch.zeros(w.shape, dtype=torch.float64, device="cuda")
    S.rhs_transpose(dev(w), dev(a), out, nu=dev(nu))
    # nu (a(x+1) - 2 a(x) + a(x-1)) / dx^2
    ref = float(nu[0, 0, 0]) * -4.0 * a[0] / dx ** 2
    inner = (slice(None), slice(2, -2), slice(2, -2))
    assert np.allclose(host(out)[0][inner], ref[inner], rtol=1e-12, atol=0)
