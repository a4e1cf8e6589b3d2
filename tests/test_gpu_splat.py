"""Splat and its adjoint at the edges of the row kernel's segments and of the vector reads, against
the FP64 oracle: records below, at and past a segment, rows without arrivals, arrivals outside
the time range and across segment borders, buffers that are not 16-byte aligned.  Splat within 1e-5
relative L2 (as test_gpu_parity.py); the adjoint's recurrences grow to a few 1e-6 of the sum of
their terms' magnitudes, so each value within 1e-5 of that sum."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2604_15017_gb300 import phantoms as P
from test_gpu_edges import ctx, dev, rel_l2  # noqa: F401  (ctx: the fixture)

pytestmark = pytest.mark.gpu

MM = 1e-3


def arrivals(ns, n, seed, ne=5, ntx=2):
    rng = np.random.default_rng(seed)
    tau = rng.uniform(-3e-6, ns / 40e6 + 3e-6, n)
    border = 2048 / 40e6 + rng.uniform(-1e-6, 1e-6, n)  # around the first segment border
    tau = np.where((rng.random(n) < 0.3) & (ns > 2048), border, tau).astype(np.float32).astype(np.float64)
    e = rng.integers(0, ne - 1, n).astype(np.int32)  # the last element's rows stay empty
    return rng.integers(0, ntx, n).astype(np.int32), e, tau, rng.normal(size=n).astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("ns,n", [(4, 50), (2044, 700), (2048, 1), (2052, 3000), (4096, 20000)])
def test_splat_segments(ctx, ns, n):
    acq = P.acquisition(5, 0.3 * MM, ns, [0.0, 4.0], 1, 1, 1540.0)
    tx, e, tau, a = arrivals(ns, n, ns)
    ref = O.splat(acq, 5e6, tx, e, tau, a)
    got = ctx.splat(acq, 5e6, dev(tx, torch.int32), dev(e, torch.int32), dev(tau), dev(a)).cpu().numpy()
    assert rel_l2(got, ref) <= 1e-5, rel_l2(got, ref)
    assert not got[:, 4].any()


def test_splat_of_nothing(ctx):
    acq = P.acquisition(5, 0.3 * MM, 2052, [0.0], 1, 1, 1540.0)
    z = torch.zeros(0, device="cuda")
    rf = ctx.splat(acq, 5e6, z.int(), z.int(), z, z, rf=torch.full((1, 5, 2052), 7.0, device="cuda"))
    assert not rf.any()


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("ns", [4, 1020, 4096])
def test_splat_adjoint_on_aligned_and_unaligned_rows(ctx, ns, shift):
    acq = P.acquisition(5, 0.3 * MM, ns, [0.0, 4.0], 1, 1, 1540.0)
    tx, e, tau, a = arrivals(ns, 2000, ns + 1)
    g = np.random.default_rng(ns).normal(size=(2, 5, ns)).astype(np.float32).astype(np.float64)
    buf = torch.zeros(g.size + shift, device="cuda")
    grf = buf[shift:].view(2, 5, ns)
    grf.copy_(dev(g))
    assert (grf.data_ptr() % 16 == 0) == (shift == 0)
    args = (dev(tx, torch.int32), dev(e, torch.int32), dev(tau), dev(a))
    got = [v.double().cpu().numpy() for v in ctx.splat_adjoint(acq, 5e6, *args, grf)]
    ref = O.splat_adjoint(acq, 5e6, tx, e, tau, a, g)
    # magnitudes: |g| against the pulse's envelope, its slope (2 pi f0 + 2 |x| / sigma) and its
    # derivative in f0 (2 pi |x| + 2 x^2 / (sigma f0)), |x| <= 4 sqrt(sigma)
    sigma = 4 * np.log(2) / (np.pi * 0.6 * 5e6) ** 2
    n = np.arange(ns)
    for k, (x, r) in enumerate(zip(got, ref)):
        t = n[None, :] / 40e6 - tau[:, None]
        env = np.abs(g[tx, e]) * np.exp(-t * t / sigma) * (np.abs(t) <= 4 * np.sqrt(sigma))
        w = [1.0, 2 * np.pi * 5e6 + 2 * np.abs(t) / sigma, 2 * np.pi * np.abs(t) + 2 * t * t / (sigma * 5e6)][k]
        scale = (env * w).sum(axis=1) * (1.0 if k == 0 else np.abs(a))
        # the time in the library is the float32 tau x fs: 2^-24 relative of up to 4096 samples
        slope = (env * (2 * np.pi * 5e6 + 2 * np.abs(t) / sigma) * w).sum(axis=1) * (1.0 if k == 0 else np.abs(a))
        assert np.all(np.abs(x - r) <= 1e-5 * scale + 1e-12 * slope + 1e-30)
