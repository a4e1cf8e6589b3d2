"""Blocks of a cluster that reach into each other's shared memory: the target must be known to have
started, so a cluster barrier has to come first."""
import os
import re

import numpy as np
import pytest

from paper_2604_15017_gb300 import build, phantoms as P


def kernels():
    """(file, name, body) of every kernel of the library."""
    for f in sorted(os.listdir(build.CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        src = re.sub(r"//[^\n]*", "", open(os.path.join(build.CSRC, f)).read())
        for m in re.finditer(r"__global__\s+void\b[^{;]*?\b(k_\w+)\s*\([^{;]*\)\s*\{", src):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(src[i], 0)
                i += 1
            yield f, m.group(1), src[m.end():i]


def test_remote_shared_memory_is_touched_after_a_cluster_barrier():
    found = list(kernels())
    assert len(found) > 30
    remote = [(f, k, b) for f, k, b in found if "map_shared_rank" in b or "shared::cluster" in b and "mapa" in b]
    assert remote  # the loss
    for f, k, body in remote:
        first = re.search(r"map_shared_rank|mapa", body).start()
        assert re.search(r"\bbarrier_wait\s*\(|\bcl\.sync\s*\(|barrier\.cluster\.wait", body[:first]), (f, k)


@pytest.mark.gpu
@pytest.mark.parametrize("nl,nd", [(1, 16), (3, 64), (7, 1024), (8, 1024), (9, 1024), (256, 1024)])
def test_loss_of_images_that_leave_blocks_of_the_cluster_idle(nl, nd):
    """Back-to-back losses of images of fewer pixels than the cluster has threads (8192), one row
    either side of it, and the largest: the sums are added in one order, so every call gives the same
    bits, within 1e-5 of the 64-bit value (positive terms in chains of up to 100)."""
    import torch

    from paper_2604_15017_gb300 import usrt

    rng = np.random.default_rng(nl)
    b, ref = (torch.tensor(-60.0 * rng.random((nl, nd)), dtype=torch.float32, device="cuda") for _ in range(2))
    img = dict(P.image(nl, nd, -0.01, 0.01, 0.0, 0.04), lambda1=0.5, lambda2=0.25)
    ctx = usrt.Context(0)
    got = torch.stack([ctx.loss(img, b, ref)[0].reshape(()) for _ in range(200)])
    r = (b.double() - ref.double()).abs()
    want = float((0.5 * r + 0.25 * r * r).mean())
    ctx.close()
    assert torch.equal(got, got[:1].expand_as(got))
    assert abs(float(got[0]) - want) <= 1e-5 * want
