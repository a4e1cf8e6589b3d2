"""What the batch autotuner chooses, and what its choices leave alone."""
import pytest
import torch

from paper_2604_15017_gb300 import phantoms as P
from paper_2604_15017_gb300 import usrt

pytestmark = pytest.mark.gpu


def item(ctx, w):
    return dict(scene=ctx.upload_workload(w), theta=w["theta"], acq=w["acq"], img=w["img"], seed=1)


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
