"""What the batch autotuner may choose: a traversal grid only where a request of the batch launches the
traversal by itself."""
import pytest
import torch

from paper_2604_15017_gb300 import phantoms as P
from paper_2604_15017_gb300 import usrt

pytestmark = pytest.mark.gpu


def item(ctx, w):
    return dict(scene=ctx.upload_workload(w), theta=w["theta"], acq=w["acq"], img=w["img"], seed=1)


def test_traversal_grid_is_tuned_only_where_it_is_used():
    ctx = usrt.Context(0)
    joint = usrt.Batch(ctx, [item(ctx, P.slab_scatterers(n_rays=100, n_scat=500)) for _ in range(2)])
    grids = {joint.autotune()[1] for _ in range(6)}
    assert len(grids) == 1  # nothing in this batch depends on it
    grid = grids.pop()
    for w in (P.two_layer(n_rays=100), P.slab_scatterers(n_rays=33000, n_scat=500)):
        lanes, tuned = usrt.Batch(ctx, [item(ctx, w)]).autotune()
        assert lanes in (1, 2, 4, 8) and tuned in (grid // 2, grid, 2 * grid)
        assert joint.autotune()[1] == tuned  # and stays what was tuned
    ctx.close()


@pytest.mark.parametrize("n_rays", [1, 40, 3000])
def test_every_traversal_grid_makes_the_same_records(n_rays):
    """Small queues are spread over one wave of resident warps, whatever the grid: the tuned context's
    records are the fresh one's."""
    w = P.hollow_cylinder(n_rays=n_rays, n_scat=0)
    recs = []
    for tune in (False, True):
        ctx = usrt.Context(0)
        it = item(ctx, w)
        if tune:
            usrt.Batch(ctx, [it]).autotune()
        ctx.forward(it["scene"], w["theta"], w["acq"], seed=1, keep_record=True)
        n = w["acq"]["n_elem"] * w["acq"]["n_rays"]
        recs.append(ctx.record(0, n, w["acq"]["k_max"]).clone())
        assert ctx.stats()["status"] == 0
        ctx.close()
    assert torch.equal(*recs)
