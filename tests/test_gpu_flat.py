"""The 2D stage kernels (nz = 1) against the marching kernels: a box of two identical planes
has the same differences (every z-difference is zero), so one plane of its result must
equal the 2D box's bit for bit in mixed precision, and to roundoff in FP64.  Sizes at the
edges of the tiles (32 cells by one or four rows), below one tile, and on both sides of
the row count that chooses the tile (304 single-row tiles)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1511_06959_gb300 import synth
from tests.test_gpu_parity import _api, dev, host, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flux", [0, 1])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("shape,batch", [((1, 1), 1), ((3, 2), 1), ((31, 3), 1), ((32, 4), 2), ((33, 5), 1),
                                         ((64, 152), 1), ((65, 153), 1), ((97, 41), 3)])
def test_flat_kernels_equal_the_marching_ones(shape, batch, prec, flux):
    api = _api()
    nx, ny = shape
    w = np.stack([synth.perturbed_uniform(nx, ny, 1, seed=71 + b, amp=0.06) for b in range(batch)])
    lam = synth.random_field(w.shape, 72)
    s = 0.05 * synth.random_field(w.shape, 73)
    nu = (1e-4 * np.abs(synth.random_field((batch, 1, ny, nx), 74))).astype(np.float32)

    def run(nz):
        def rep(x):
            return dev(np.repeat(x, nz, axis=-3))
        S = api.Solver(nx, ny, nz, (0.1, 0.11, 0.09), mu=1e-2, dt=1e-2, precision=prec, plane_i=nx // 2, batch=batch,
                       flux=flux)
        W, L, Q, N = rep(w), rep(lam), rep(s), rep(nu)
        out = [torch.zeros_like(W) for _ in range(4)]
        S.primal_step(W, out[0], Q)
        S.rhs_transpose(W, L, out[1], nu=N)
        S.adjoint_step(W, L, out[2], s=Q, nu=N, sbar=out[3])
        assert S.last_error() == 0
        return [host(o)[..., :1, :, :] for o in out]

    for a, b in zip(run(1), run(2)):
        if prec == 1:
            assert np.array_equal(a, b)
        else:
            # FP64 contractions may differ between the kernels: a few ulps per operation
            assert rel_l2(a, b) < 1e-13
