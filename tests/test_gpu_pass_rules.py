"""Which passes sort: the stages that a call launches, at both sides of each line that the library draws by
the number of paths, of triangles and of scatterers."""
import numpy as np
import pytest
import torch

from paper_2604_15017_gb300 import phantoms as P
from test_gpu_edges import ctx  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu

MM = 1e-3
LARGE = 33000  # rays per element of 64: more than 2^21 paths


def boxes(n, n_rays):
    """The two-layer phantom (12 triangles) with n boxes of 12 triangles in its first layer."""
    w = P.two_layer(n_rays=n_rays, k_max=2)
    tris, media = [np.asarray(w["tris"]).reshape(-1, 9)], [np.asarray(w["media"])]
    for i in range(n):
        c = np.array([-6.0 + 4.0 * i, 0.0, 8.0]) * MM
        tris.append(np.asarray(P.box_mesh(c - 1.0 * MM, c + 1.0 * MM)).reshape(-1, 9))
        media.append(np.tile(np.array([[0, 1]], media[0].dtype), (12, 1)))
    w["tris"], w["media"] = np.concatenate(tris), np.concatenate(media)
    return w


def launches(ctx, w):
    sid = ctx.upload_workload(w)
    ctx.profile(True)
    ctx.forward(sid, w["theta"], w["acq"], seed=3)
    torch.cuda.synchronize()
    n = {k: v[1] for k, v in ctx.profile_read().items()}
    ctx.profile(False)
    ctx.release_scene(sid)
    return n


@pytest.mark.parametrize("make,rays", [
    (lambda: boxes(0, 32768), False),  # 2^21 paths
    (lambda: boxes(3, 32768), False),
    (lambda: boxes(0, LARGE), False),  # 12 triangles
    (lambda: boxes(1, LARGE), False),  # 24
    (lambda: boxes(2, LARGE), True),   # 36
    (lambda: P.slab_scatterers(n_rays=32768, n_scat=500, k_max=2), False),
    (lambda: P.slab_scatterers(n_rays=LARGE, n_scat=500, k_max=2), True),
])
def test_rays_are_sorted_in_large_passes_of_scenes_with_many_nodes(ctx, make, rays):
    assert (launches(ctx, make())["ray_sort"] > 0) == rays
