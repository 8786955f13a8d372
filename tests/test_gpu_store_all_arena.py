"""A store-all sweep in an arena that holds it without its kept stages (the size from before
stages were kept) runs without them and gives the same bits: called, captured, in halves and
under estimate_lambda; a smaller arena is refused."""
import pytest

torch = pytest.importorskip("torch")

from paper_1511_06959_gb300 import synth
from tests.test_gpu_parity import _api, dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("nsteps", [1, 6])
def test_arena_without_kept_stages(prec, nsteps):
    api = _api()
    nx, ny, nz = 37, 9, 5
    w = dev(synth.perturbed_uniform(nx, ny, nz, seed=83, amp=0.05))
    S = api.Solver(nx, ny, nz, 0.1, mu=1e-2, dt=1e-2, precision=prec, plane_i=nx // 2)
    o = S.run_opts(nsteps, api.NS_CKPT_ALL, 0, 1e-4)
    full = S.arena_bytes(o)
    S.set_pipeline(False)
    small = S.arena_bytes(o)
    S.set_pipeline(True)
    assert full == S.arena_bytes(o) > small
    J = torch.empty(1, dtype=torch.float64, device="cuda")

    def run(nbytes, how):
        arena = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        lam0, sbar = torch.zeros_like(w), torch.zeros_like(w)
        if how == "call":
            S.adjoint_run(w, o, arena, J, lam0, sbar=sbar)
        elif how == "halves":
            S.forward_run(w, o, arena, J)
            S.backward_run(lam0, sbar=sbar)
        else:
            # its own stream: the legacy stream cannot be captured
            st = torch.cuda.Stream()
            st.wait_stream(torch.cuda.current_stream())
            S.set_stream(st)
            G = S.adjoint_run_capture(w, o, arena, J, lam0, sbar=sbar)
            G.launch()
            torch.cuda.synchronize()
            G.close()
            S.set_stream(torch.cuda.current_stream())
        torch.cuda.synchronize()
        assert S.last_error() == 0
        return J.clone(), lam0, sbar

    hows = ("call", "halves", "capture")     # (the halves add the objectives of the steps in another order)
    ref = {how: run(full, how) for how in hows}
    # the exact smaller size, and sizes up to one step's entry (four stage fields) below the full
    for nbytes in (small, (small + full - (full - small) // nsteps) // 2 // 256 * 256, full - (full - small) // nsteps):
        for how in hows:
            for a, b in zip(run(nbytes, how), ref[how]):
                assert torch.equal(a, b), (nbytes - small, how)
    with pytest.raises(api.NsError) as e:
        run(small - 1, "call")
    assert e.value.code == api.NS_ERR_BUDGET
    if nsteps > 1:
        work = torch.empty(S.estimate_work_bytes(o), dtype=torch.uint8, device="cuda")
        got = [S.estimate_lambda(w, o, [0.0, 1e-4, 1e-3], torch.empty(n, dtype=torch.uint8, device="cuda"), work)
               for n in (full, small)]
        assert got[0] == got[1]
        with pytest.raises(api.NsError) as e:
            S.estimate_lambda(w, o, [0.0, 1e-4], torch.empty(small - 1, dtype=torch.uint8, device="cuda"), work)
        assert e.value.code == api.NS_ERR_BUDGET
