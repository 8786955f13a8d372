"""Store-all sweeps that keep every step's stage states against the same sweep with the
smallest footprint (the stages recomputed): the same bits, one step and several, both
precisions and schemes; an arena one byte short of either is refused."""
import pytest

torch = pytest.importorskip("torch")

from paper_1511_06959_gb300 import synth
from tests.test_gpu_parity import _api, dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(37, 9, 5), (40, 12, 1)])
@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("nsteps", [1, 5])
def test_kept_stages_give_the_recomputed_bits(shape, scheme, prec, nsteps):
    api = _api()
    nx, ny, nz = shape
    w = dev(synth.perturbed_uniform(nx, ny, nz, seed=81, amp=0.05))
    S = api.Solver(nx, ny, nz, 0.1, mu=1e-2, dt=1e-2, precision=prec, plane_i=nx // 2, scheme=scheme)
    o = S.run_opts(nsteps, api.NS_CKPT_ALL, 0, 1e-4, 0.0, True, True)
    full = S.arena_bytes(o)
    S.set_pipeline(False)
    small = S.arena_bytes(o)
    stage = -(-w.numel() * (8 if prec == 0 else 4) // 256) * 256
    assert full - small == 4 * nsteps * stage

    def run(keep, nbytes):
        S.set_pipeline(keep)
        arena = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        J = torch.empty(1, dtype=torch.float64, device="cuda")
        lam0, sbar = torch.empty_like(w), torch.empty_like(w)
        E = torch.zeros((nsteps + 1, 1), dtype=torch.float64, device="cuda")
        st = torch.zeros((nsteps, 1, 2), dtype=torch.float64, device="cuda")
        S.adjoint_run(w, o, arena, J, lam0, sbar=sbar, energy=E, sigma_stats=st)
        assert S.last_error() == 0
        return [host(t) for t in (J, lam0, sbar, E, st)]

    for a, b in zip(run(True, full), run(False, small)):
        assert (a == b).all()
    for keep, need in ((True, full), (False, small)):
        with pytest.raises(api.NsError) as e:
            run(keep, need - 1)
        assert e.value.code == api.NS_ERR_BUDGET
