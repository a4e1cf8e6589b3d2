"""The acquisition-gradient DAS at the edges of its tiles (8 lines x 32 depths, elements in pairs)
against the FP64 oracle: images smaller than a tile and ragged ones, one element, odd and even
counts, 1 to 64 transmits, records that end inside the image, both apodisations.  Per component
within 1e-3 (the bound of test_gpu_acq.py) of the sum over lines of that line's share in absolute
value: a component may cancel between lines."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2604_15017_gb300 import phantoms as P
from test_gpu_acq import MM, exact_angles, f32
from test_gpu_edges import ctx, dev  # noqa: F401  (ctx: the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ne,ntx,ns,nl,nd,f", [
    (1, 1, 1024, 1, 16, 0.0),
    (2, 1, 1024, 9, 32, 0.0),
    (31, 3, 1024, 7, 64, 1.5),
    (32, 2, 1020, 17, 16, 0.0),
    (33, 5, 500, 8, 128, 0.0),  # the record ends inside the image
    (255, 2, 512, 3, 64, 2.0),
    (6, 64, 1024, 5, 32, 0.0),
])
def test_das_acq_on_ragged_tiles(ctx, ne, ntx, ns, nl, nd, f):
    degs = [6.0] if ntx == 1 else list(np.linspace(-14.0, 15.0, ntx))
    acq = dict(P.acquisition(ne, float(np.float32(0.3 * MM)), ns, degs, 1, 1, 1540.0), angles=exact_angles(degs))
    img = P.image(nl, nd, *(float(np.float32(v)) for v in (-4.1 * MM, 3.7 * MM, 2 * MM, 15 * MM)), f_number=f)
    rng = np.random.default_rng(ne * 100 + ntx)
    n = 3000 * ntx
    rf = f32(O.splat(acq, 5e6, rng.integers(0, ntx, n), rng.integers(0, ne, n), rng.uniform(0, ns / 40e6, n),
                     rng.normal(size=n)))
    gi = f32(rng.normal(size=(nl, nd)))
    lines = np.stack([O.das_acq_vjp(acq, img, rf, gi * (np.arange(nl) == l)[:, None]) for l in range(nl)])
    got = ctx.das_acq_vjp(acq, img, dev(rf), dev(gi)).double().cpu().numpy()
    ref, size = lines.sum(axis=0), np.abs(lines).sum(axis=0)
    assert np.all(np.abs(got - ref) <= 1e-3 * size), np.c_[got, ref, size]
