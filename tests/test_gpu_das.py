"""DAS at the edges of its tiling against the FP64 oracle: images smaller than a tile and ragged
ones, element counts around the chunk of 32 and the four element groups, 1 to 64 transmits,
records that end inside the image (the checked taps), both apodisations.  Per pixel within 2e-3 of
the DAS of |RF| (the bound of test_gpu_parity.py)."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2604_15017_gb300 import phantoms as P
from test_gpu_edges import ctx, dev  # noqa: F401  (ctx: the fixture)

pytestmark = pytest.mark.gpu

MM = 1e-3


@pytest.mark.parametrize("ne,ntx,ns,nl,nd,depth,f", [
    (1, 1, 64, 1, 16, 2.0, 0.0),
    (3, 1, 1024, 7, 32, 15.0, 0.0),
    (31, 2, 1024, 9, 16, 15.0, 1.5),
    (32, 5, 2048, 8, 64, 60.0, 0.0),
    (33, 3, 1020, 13, 256, 30.0, 2.0),
    (95, 1, 2044, 101, 32, 39.0, 0.0),
    (129, 17, 512, 5, 64, 12.0, 0.0),
    (12, 64, 512, 17, 16, 9.0, 1.5),
    (256, 2, 4096, 3, 128, 70.0, 1.0),
])
def test_das_matches_oracle_on_ragged_tiles(ctx, ne, ntx, ns, nl, nd, depth, f):
    angles = [7.0] if ntx == 1 else list(np.linspace(-25.0, 25.0, ntx))
    acq = P.acquisition(ne, 0.3 * MM, ns, angles, 1, 1, 1540.0)
    # wider than the array on one side, so that transmit delays fall below zero there
    img = P.image(nl, nd, -0.2 * ne * MM - 3 * MM, 0.15 * ne * MM, 0.0, depth * MM, f_number=f)
    rng = np.random.default_rng(ne * 1000 + ntx)
    rf = rng.normal(size=(ntx, ne, ns)).astype(np.float32).astype(np.float64)
    q, im = dict(acq), dict(img)
    for k in ("pitch", "c_bf", "fs"):
        q[k] = float(np.float32(q[k]))
    for k in ("x0", "x1", "z0", "z1"):
        im[k] = float(np.float32(im[k]))
    q["angles"] = [float(np.float32(v)) for v in acq["angles"]]
    ref = O.das(q, im, rf)
    bound = 2e-3 * O.das(q, im, np.abs(rf)) + 1e-6 * np.abs(ref).max()
    got = ctx.das(acq, img, dev(rf)).cpu().numpy()
    assert np.all(np.abs(got - ref) <= bound), np.max(np.abs(got - ref) - bound)


@pytest.mark.parametrize("ne,ntx,ns,nl,nd,depth", [
    (7, 3, 256, 5, 16, 4.0),       # fewer lines and depths than a tile
    (100, 1, 4096, 33, 64, 60.0),  # coarse depths: windows of the largest size, some longer
    (31, 15, 2048, 40, 256, 39.0),  # one element per batch but 15 columns
    (101, 11, 3000, 97, 512, 57.0),
    (24, 36, 1024, 20, 32, 15.0),  # the most transmits the tiled kernel takes, and one more
    (24, 37, 1024, 20, 32, 15.0),
])
def test_transposed_das_tiled_equals_untiled(ctx, ne, ntx, ns, nl, nd, depth):
    """The same fixed-point shares summed either way: the same bits, whatever window length, batch
    of elements and split over blocks the sizes lead to."""
    from paper_2604_15017_gb300 import usrt

    angles = [7.0] if ntx == 1 else list(np.linspace(-20.0, 20.0, ntx))
    acq = P.acquisition(ne, 0.3 * MM, ns, angles, 1, 1, 1540.0)
    img = P.image(nl, nd, -0.16 * ne * MM, 0.15 * ne * MM, 0.0, depth * MM, f_number=1.5 if ntx == 15 else 0.0)
    g = torch.Generator(device="cpu").manual_seed(ne)
    gi = torch.randn(nl, nd, generator=g).cuda()
    tiled = ctx.das_adjoint(acq, img, gi)
    usrt.set_das_adj_tiled(False)
    try:
        plain = ctx.das_adjoint(acq, img, gi)
    finally:
        usrt.set_das_adj_tiled(True)
    assert torch.equal(tiled, plain)
    assert float(tiled.abs().max()) > 0.0


def test_das_far_beside_the_array(ctx):
    """Pixels 4.2e6 samples beside the array under a steering of 88 degrees: the transmit delay falls
    below -2^22 samples, past which a pixel's taps are not checked all at once, and the sums run
    across the record's end."""
    from test_gpu_acq import exact_angles

    degs = [88.0, 87.99]
    acq = dict(P.acquisition(33, float(np.float32(0.3 * MM)), 2720, degs, 1, 1, 1540.0), angles=exact_angles(degs))
    img = P.image(9, 32, float(np.float32(-161.66)), float(np.float32(-161.58)), 0.0, float(np.float32(0.03)))
    rf = np.random.default_rng(5).normal(size=(2, 33, 2720)).astype(np.float32)
    for k in ("pitch", "c_bf", "fs"):
        acq[k] = float(np.float32(acq[k]))
    ref = O.das(acq, img, rf.astype(np.float64))
    bound = 2e-3 * O.das(acq, img, np.abs(rf).astype(np.float64)) + 1e-6 * np.abs(ref).max()
    got = ctx.das(acq, img, dev(rf)).cpu().numpy()
    assert np.all(np.abs(got - ref) <= bound), np.max(np.abs(got - ref) - bound)
