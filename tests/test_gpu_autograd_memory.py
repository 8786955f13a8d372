"""A source problem whose store-all arena with kept stages does not fit the device takes the
arena without them: the same loss and gradients, to the bit; without room for that either, or
for another schedule, the allocator's error stands."""
import pytest

torch = pytest.importorskip("torch")

from paper_1511_06959_gb300 import synth
from tests.test_gpu_parity import _api, dev

pytestmark = pytest.mark.gpu


def test_kept_stages_beyond_the_device_memory(monkeypatch):
    api = _api()
    from paper_1511_06959_gb300 import autograd
    nx, ny, nz, N = 33, 10, 3, 6
    w0 = synth.perturbed_uniform(nx, ny, nz, seed=85, amp=0.05)[None]
    phi = dev(synth.forcing_bumps(nx, ny, nz, n=3))
    S = api.Solver(nx, ny, nz, 0.1, mu=1e-2, dt=1e-2, precision=1, plane_i=nx // 2)

    def run():
        problem = autograd.SourceProblem(S, phi, N)
        w = dev(w0).requires_grad_()
        theta = torch.linspace(0.1, 0.3, phi.shape[0], dtype=torch.float64, device="cuda").requires_grad_()
        J = problem(w, theta)
        J.sum().backward()
        return problem.arena.numel(), J.detach(), w.grad, theta.grad

    ref = run()
    opts = S.run_opts(N, api.NS_CKPT_ALL)
    full = S.arena_bytes(opts)
    assert ref[0] == full
    S.set_pipeline(False)
    small = S.arena_bytes(opts)
    S.set_pipeline(True)
    limit = full - 1
    empty = torch.empty

    def short(*a, **k):
        if k.get("dtype") is torch.uint8 and a and isinstance(a[0], int) and a[0] > limit:
            raise torch.cuda.OutOfMemoryError("no room")
        return empty(*a, **k)

    monkeypatch.setattr(torch, "empty", short)
    got = run()
    assert got[0] == small and S.arena_bytes(opts) == full
    for x, y in zip(got[1:], ref[1:]):
        assert torch.equal(x, y)
    limit = small - 1
    with pytest.raises(torch.cuda.OutOfMemoryError):
        autograd.SourceProblem(S, phi, N)
    limit = 0
    with pytest.raises(torch.cuda.OutOfMemoryError):
        autograd.SourceProblem(S, phi, N, api.NS_CKPT_STRIDE, 2)
    limit = small
    S.set_pipeline(False)
    assert autograd.SourceProblem(S, phi, N).arena.numel() == small
    assert S.arena_bytes(opts) == small       # the switch is as the caller left it
