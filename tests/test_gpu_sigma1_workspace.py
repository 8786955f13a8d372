"""The workspace of sigma_1's statistics in large batches, and sigma_1 with its statistics on
batches where that bounds the split of the columns, against single boxes."""
import pytest

torch = pytest.importorskip("torch")

from paper_1511_06959_gb300 import synth
from tests.test_gpu_parity import _api, dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,batch,most_mb", [((64, 64, 1), 256, 30), ((64, 64, 1), 1024, 22), ((32, 32, 32), 64, 9),
                                                 ((128, 64, 64), 1, 3)])
def test_workspace(shape, batch, most_mb):
    api = _api()
    S = api.Solver(*shape, 0.1, precision=1, batch=batch)
    field = 5 * shape[0] * shape[1] * shape[2] * batch * 4
    # beside the nine stage fields: the reductions' partials.  256 boxes of 64x64: 27 columns a
    # box (a ghost layer counted), a pair of doubles for every column and box, 28.3 MB; more
    # boxes than 256 have no sigma_1 statistics: 2368 doubles a box of the other reductions
    assert S.workspace_bytes() - 9 * field < most_mb * 1e6


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("shape,batch", [((40, 9, 4), 256), ((33, 17, 9), 200), ((5, 3, 2), 256), ((70, 8, 64), 205)])
def test_statistics_of_batches(shape, batch, prec):
    api = _api()
    one = [dev(synth.perturbed_uniform(*shape, seed=700 + i, amp=0.05)) for i in range(4)]
    w = torch.stack([one[i % 4] for i in range(batch)]).contiguous()
    S, S1 = (api.Solver(*shape, 0.1, precision=prec, batch=b) for b in (batch, 1))
    sig = torch.empty((batch,) + tuple(w.shape[2:]), dtype=torch.float32, device="cuda")
    st = torch.empty((batch, 2), dtype=torch.float64, device="cuda")
    S.growth_sigma1(w, sig, st)
    for i in range(4):
        ref, rst = torch.empty_like(sig[:1]), torch.empty((1, 2), dtype=torch.float64, device="cuda")
        S1.growth_sigma1(one[i], ref, rst)
        assert torch.equal(sig[i::4], ref.expand_as(sig[i::4]))
        # the same maximum; sums of at most 35840 terms in another order: FP64 partials (4e-12 at
        # the very worst), float pairs of 2^-44 within a CTA
        assert torch.equal(st[i::4, 0], rst[:, 0].expand_as(st[i::4, 0]))
        assert (st[i::4, 1] / rst[0, 1] - 1).abs().max() < 1e-11
