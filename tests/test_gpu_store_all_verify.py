"""A verified store-all sweep: whatever byte of its arena changes between the forward and the
backward half, the gradient has the undisturbed sweep's bits or the error word says
NS_ERR_CORRUPT.  Nothing a checksum does not cover may reach the gradient, but for the last
state, which the forward half hands over in a working buffer and no plan stores."""
import pytest

torch = pytest.importorskip("torch")

from paper_1511_06959_gb300 import synth
from tests.test_gpu_parity import _api, dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("scheme", [0, 1])
def test_no_unverified_word_reaches_the_gradient(prec, scheme):
    api = _api()
    nx, ny, nz, N = 33, 10, 3, 5
    w = dev(synth.perturbed_uniform(nx, ny, nz, seed=82, amp=0.05))
    S = api.Solver(nx, ny, nz, 0.1, mu=1e-2, dt=1e-2, precision=prec, plane_i=nx // 2, scheme=scheme)
    o = S.run_opts(N, api.NS_CKPT_ALL, 0, 1e-4, verify=True)
    need = S.arena_bytes(o)
    S.set_pipeline(False)
    assert need == S.arena_bytes(o)      # nothing kept beside the snapshots
    S.set_pipeline(True)
    J = torch.empty(1, dtype=torch.float64, device="cuda")
    ref, lam = torch.empty_like(w), torch.empty_like(w)
    arena = torch.zeros(need, dtype=torch.uint8, device="cuda")
    S.adjoint_run(w, o, arena, J, ref)
    assert S.last_error() == 0
    state = -(-w.numel() * 8 // 256) * 256
    wN = w
    for _ in range(N):
        nxt = torch.empty_like(w)
        S.primal_step(wN, nxt)
        wN = nxt
    reported = 0
    flips = 64
    for i in range(flips):
        S.forward_run(w, o, arena, J)
        # the top byte of a 64-bit word: sign or exponent of a double, of a float's upper half
        at = (need // 8 * (2 * i + 1) // (2 * flips)) * 8 + 7
        first = at // state * state
        held = arena[first:first + w.numel() * 8]
        if held.numel() == w.numel() * 8 and torch.equal(held.view(torch.float64), wN.flatten()):
            continue
        arena[at] ^= 0x41
        S.backward_run(lam)
        err = S.last_error()
        reported += err == api.NS_ERR_CORRUPT
        assert err == api.NS_ERR_CORRUPT or (err == 0 and torch.equal(lam, ref)), (i, at, err)
    assert reported > 0
