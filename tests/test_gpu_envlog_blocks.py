"""The envelope's VJP where its one launch goes from one line per block to two, three, four and to four
kernels: by the number of lines (two blocks' partial sums per SM, 304) and, in long lines, by the
blocks whose lines fit the SMs' shared memory together (304 of one line of 4096 depths, 152 of two or
three, 760 of one of 2048).  Against the oracle, as in test_gpu_envlog.py."""
import pytest
import torch

from test_gpu_edges import ctx  # noqa: F401  (the fixture)
from test_gpu_envlog import image, test_envlog_vjp_one_launch_and_four as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nl,nd", [(304, 16), (305, 16), (608, 64), (912, 64), (1216, 64), (1217, 64), (304, 4096),
                                   (400, 4096), (608, 2048)])
def test_lines_per_block(ctx, nl, nd):
    check(ctx, nl, nd)


@pytest.mark.parametrize("nl,nd,kernels", [(304, 16, 1), (1216, 64, 1), (1217, 64, 4), (304, 4096, 1), (608, 4096, 1),
                                           (609, 4096, 4)])
def test_launches(ctx, nl, nd, kernels):
    irf = torch.randn(nl, nd, device="cuda")
    ctx.profile(True)
    ctx.envlog_vjp(image(nl, nd), irf, irf.clone())
    torch.cuda.synchronize()
    n = ctx.profile_read()["envlog_vjp"][1]
    ctx.profile(False)
    assert n == kernels


@pytest.mark.parametrize("nl,nd", [(1300, 16), (1217, 32), (1300, 64), (1217, 128), (1217, 256)])
def test_short_lines_in_four_kernels(ctx, nl, nd):
    # as many threads as a line has pixels, from 64 to 256
    check(ctx, nl, nd)


@pytest.mark.parametrize("nl,kernels", [(256, 1), (257, 2)])
def test_loss_launches(ctx, nl, kernels):
    # one launch up to 2^18 pixels; the values at both sides against 64 bits
    b, ref = (-60.0 * torch.rand(nl, 1024, generator=torch.Generator().manual_seed(k)).cuda() for k in (1, 2))
    img = dict(image(nl, 1024), lambda1=0.5, lambda2=0.25)
    ctx.profile(True)
    loss, gb = ctx.loss(img, b, ref)
    torch.cuda.synchronize()
    n = ctx.profile_read()["loss"][1]
    ctx.profile(False)
    assert n == kernels
    r = b.double() - ref.double()
    want = float((0.5 * r.abs() + 0.25 * r * r).mean())
    assert abs(float(loss) - want) <= 1e-5 * want  # positive terms in chains of up to 100
    g = (0.5 * r.sign() + 0.5 * r) / r.numel()
    assert float((gb - g).abs().max()) <= 1e-6 * float(g.abs().max())


def test_two_launches_that_each_fill_the_gpu(ctx):
    """304 lines of 4096 depths take every block that fits; two such VJPs on two streams, beside each other,
    wait for blocks of their own launch only and give the bits of one after the other."""
    from paper_2604_15017_gb300 import usrt

    other = usrt.Context(0)
    img = image(304, 4096)
    sides = []
    for c, k in ((ctx, 1), (other, 2)):
        gen = torch.Generator("cuda").manual_seed(k)
        irf, gb = (torch.randn(304, 4096, generator=gen, device="cuda") for _ in range(2))
        sides.append((c, irf, gb, torch.cuda.Stream(), c.envlog_vjp(img, irf, gb)))
    torch.cuda.synchronize()
    out = [[], []]
    for _ in range(20):
        for j, (c, irf, gb, st, _) in enumerate(sides):
            with torch.cuda.stream(st):
                out[j].append(c.envlog_vjp(img, irf, gb))
    torch.cuda.synchronize()
    for j, (c, *_, want) in enumerate(sides):
        assert c.device_status() == usrt.US_OK
        assert all(torch.equal(v, want) for v in out[j])
    other.close()
