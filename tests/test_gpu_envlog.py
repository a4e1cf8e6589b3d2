"""The envelope's VJP and the loss at the edges of their one-launch kernels: one to four lines per
block, one line more than those take, the shortest and longest depths; images around the largest
one-launch loss.

Tolerances.  The lines are carriers of a quarter of the depth under a band-limited modulation
between 0.5 and 3.5, so that the envelope is the modulation and no pixel is ill-conditioned.  A
pixel then holds a few FP32 roundings of g c / E and of one transform back, and the envelope's own
error, log2(n) eps of the line: under 1e-5 of the line's l2 norm.  The line with the maximum also
holds the sum S of all live gradients: chains of up to 100 additions, 1e-5 of sum |g|.  The loss
adds positive terms in chains of up to 100: 1e-5 of itself; its gradient is a few roundings."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2604_15017_gb300 import phantoms as P
from paper_2604_15017_gb300 import usrt
from test_gpu_edges import ctx, dev  # noqa: F401  (ctx: the fixture)

pytestmark = pytest.mark.gpu


def image(nl, nd):
    return P.image(nl, nd, -0.01, 0.01, 0.0, 0.04)


@pytest.mark.parametrize("nl,nd", [
    (1, 16), (5, 64),
    (608, 32), (609, 32),  # one line per block, two
    (2433, 16),            # more than four per block
    (128, 512), (152, 4096), (153, 4096), (305, 4096),
])
def test_envlog_vjp_one_launch_and_four(ctx, nl, nd):
    rng = np.random.default_rng(nl * 10000 + nd)
    spec = np.zeros((nl, nd // 2 + 1), np.complex128)
    m = nd // 8
    spec[:, 1:m + 1] = rng.normal(size=(nl, m)) + 1j * rng.normal(size=(nl, m))
    mod = np.fft.irfft(spec, nd, axis=1)
    mod = 2.0 + 1.5 * mod / np.abs(mod).max(axis=1, keepdims=True)
    # line amplitudes over 80 dB: with the range of 60 dB some lines are clipped
    amp = 10.0 ** (-4.0 * rng.random((nl, 1)))
    ph = 0.5 * np.pi * np.arange(nd)[None, :] + 2.0 * np.pi * rng.random((nl, 1))
    irf = (amp * mod * np.cos(ph)).astype(np.float32)
    gb = rng.normal(size=(nl, nd)).astype(np.float32)
    img = image(nl, nd)
    ref = O.envlog_vjp(img, irf.astype(np.float64), gb.astype(np.float64))
    env = O.envelope(img, irf.astype(np.float64))
    tol = np.repeat(1e-5 * np.linalg.norm(ref, axis=1, keepdims=True), nd, axis=1)
    line = int(env.argmax()) // nd
    tol[line] += 1e-5 * 8.685889638065036 * np.abs(gb).sum(dtype=np.float64) / env.max()
    got = ctx.envlog_vjp(img, dev(irf), dev(gb)).cpu().numpy()
    usrt.set_envlog_fused(False)
    try:
        four = ctx.envlog_vjp(img, dev(irf), dev(gb)).cpu().numpy()
    finally:
        usrt.set_envlog_fused(True)
    assert np.all(np.abs(got - ref) <= tol), np.max(np.abs(got - ref) / np.maximum(tol, 1e-300))
    assert np.all(np.abs(four - ref) <= tol), np.max(np.abs(four - ref) / np.maximum(tol, 1e-300))


@pytest.mark.parametrize("nl,nd", [(1, 16), (3, 32), (101, 256), (512, 1024), (513, 1024)])
@pytest.mark.parametrize("grad", [True, False])
def test_loss_around_the_largest_single_launch(ctx, nl, nd, grad):
    rng = np.random.default_rng(nl + nd)
    b = (-60.0 * rng.random((nl, nd))).astype(np.float32)
    bref = np.where(rng.random((nl, nd)) < 0.1, b, (-60.0 * rng.random((nl, nd))).astype(np.float32))
    img = dict(image(nl, nd), lambda1=float(np.float32(0.7)), lambda2=float(np.float32(0.3)))
    val, g = O.loss(img, b.astype(np.float64), bref.astype(np.float64))
    loss, gb = ctx.loss(img, dev(b), dev(bref), grad=grad)
    assert abs(float(loss) - val) <= 1e-5 * abs(val)
    if not grad:
        assert gb is None
        return
    r = np.abs(b.astype(np.float64) - bref)
    bound = 1e-6 * (0.7 + 0.6 * r) / (nl * nd)
    assert np.all(np.abs(gb.cpu().numpy() - g) <= bound)
    assert np.all(gb.cpu().numpy()[r == 0.0] == 0.0)
