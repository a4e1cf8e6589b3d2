"""The longest arrival list that the splat takes, 2^32 - 17 entries (indexes stepped past its end do not
fit 32 bits): all but seven of them lie before the record, and those seven make the channel data."""
import numpy as np
import pytest
import torch

from paper_2604_15017_gb300 import phantoms as P
from paper_2604_15017_gb300 import usrt

pytestmark = pytest.mark.gpu


def test_longest_arrival_list():
    n = (1 << 32) - 17
    need = 2 * 4 * n + 2 * 8 * (n + n // 8)  # two of the four arrays (shared below), the buckets twice
    if torch.cuda.mem_get_info()[0] < need + (8 << 30):
        pytest.skip("needs %d GB" % (need >> 30))
    acq = P.acquisition(4, 0.3e-3, 1024, [0.0], 1, 1, 1540.0)
    zero = torch.zeros(n, dtype=torch.int32, device="cuda")  # transmit and element
    tau = torch.full((n,), -1.0, device="cuda")              # times, and amplitudes
    at = torch.tensor([0, 1, (1 << 31) - 1, 1 << 31, n - 5000000, n - 8192, n - 1], device="cuda")
    tau[at] = torch.tensor(np.linspace(2e-6, 20e-6, len(at)), dtype=torch.float32, device="cuda")
    ctx = usrt.Context(0)
    rf = ctx.splat(acq, 5e6, zero, zero, tau, tau)
    few = tau[at]
    want = ctx.splat(acq, 5e6, zero[:len(at)], zero[:len(at)], few, few)
    assert float(want.abs().max()) > 0.0
    assert torch.equal(rf, want)
    ctx.close()
    del zero, tau
    torch.cuda.empty_cache()
