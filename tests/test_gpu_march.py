"""Closest hits at the edges of the kernels' work distribution, against the FP64 oracle: queues
smaller than a warp, around one item per resident warp and past one full wave; grid cells that
hold more spheres than a record (chains of records), clusters on cell faces, grids one cell
thick.  Tolerances as in test_gpu_edges.py."""
import numpy as np
import pytest

from paper_2604_15017_gb300 import phantoms as P
from test_gpu_edges import ctx, no_triangles, parity  # noqa: F401  (ctx: the fixture)

pytestmark = pytest.mark.gpu

MM = 1e-3


@pytest.mark.parametrize("n_rays", [1, 3, 75, 305, 2600])
def test_queue_sizes_from_a_few_rays_to_more_than_a_wave(ctx, n_rays):
    # 64 elements: 64 .. 166400 rays; 152 SMs x 32 resident warps take 4 .. 32 lanes each
    parity(ctx, P.slab_scatterers(n_rays=n_rays, n_scat=4000))


@pytest.mark.parametrize("cluster,spread", [(3, 0.02), (4, 0.02), (5, 0.3), (64, 0.02), (200, 0.05)])
def test_crowded_cells(ctx, cluster, spread):
    w = no_triangles(P.slab_scatterers(n_rays=400, n_scat=600))
    rng = np.random.default_rng(cluster)
    centres = np.stack([rng.uniform(-8, 8, 40), rng.uniform(-1, 1, 40), rng.uniform(6, 20, 40)], axis=1) * MM
    n = 40 if cluster < 64 else 2
    pts = (centres[:n, None] + spread * MM * rng.normal(size=(n, cluster, 3))).reshape(-1, 3)
    w["scat_pos"] = np.concatenate([w["scat_pos"], pts])
    w["scat_amp"] = rng.normal(size=len(w["scat_pos"]))
    parity(ctx, w)


@pytest.mark.parametrize("axis", [0, 1, 2])
def test_grids_one_cell_thick(ctx, axis):
    w = no_triangles(P.slab_scatterers(n_rays=400, n_scat=3000))
    w["scat_pos"][:, axis] = [0.0, 0.0, 12 * MM][axis]  # a sheet of scatterers
    parity(ctx, w)
