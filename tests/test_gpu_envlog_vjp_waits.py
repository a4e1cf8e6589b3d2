"""The bounded waits of the envelope's one-launch VJP, run out on purpose from the host
(US_OPT_FAULT_BARRIER: every block but the first waits, 1 ms, for one arrival that no block makes).  The
first block's waits succeed, so with the image's maximum in its line the only thing wrong there is the
others' share of the sum over all pixels: no number may come out of that either."""
import pytest
import torch

from paper_2604_15017_gb300 import phantoms as P
from paper_2604_15017_gb300 import usrt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nl,nd,per_block", [(64, 256, 1), (2, 16, 1), (609, 64, 3)])
@pytest.mark.parametrize("top", [0, 1])
def test_an_expired_wait_leaves_no_number_that_depends_on_it(nl, nd, per_block, top):
    ctx = usrt.Context(0)
    img = P.image(nl, nd, 0.0, 1.0, 0.0, 1.0)
    g = torch.Generator().manual_seed(nl)
    irf = torch.randn(nl, nd, generator=g)
    irf[top] *= 100.0  # the image's maximum: in the first block's line, or in another's
    irf, gb = irf.cuda(), torch.randn(nl, nd, generator=g).cuda()
    ref = ctx.envlog_vjp(img, irf, gb)
    assert torch.isfinite(ref).all() and ctx.device_status() == usrt.US_OK
    ctx.set_option(usrt.OPT_FAULT_BARRIER, 1)
    try:
        got = ctx.envlog_vjp(img, irf, gb)
    finally:
        ctx.set_option(usrt.OPT_FAULT_BARRIER, 0)
    assert ctx.device_status(clear=True) == usrt.US_ERR_TIMEOUT
    blocks = -(-nl // per_block)  # a block's lines are its number and every `blocks`-th one after it
    first = torch.arange(nl, device="cuda") % blocks == 0
    assert torch.isnan(got[~first]).all()
    assert torch.isnan(got[top]).all()
    # the first block's other lines need the maximum alone, and that it had
    rest = first.clone()
    rest[top] = False
    assert torch.equal(got[rest], ref[rest])
    again = ctx.envlog_vjp(img, irf, gb)
    assert ctx.device_status() == usrt.US_OK
    assert torch.equal(again, ref)
    ctx.close()
