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


def launches(ctx, w, **kw):
    sid = ctx.upload_workload(w)
    ctx.profile(True)
    ctx.forward(sid, w["theta"], w["acq"], seed=3, **kw)
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


@pytest.mark.parametrize("make,jobs,recorded", [
    (lambda: P.with_roughness(boxes(0, 32768), [0.0, 0.3]), False, False),
    (lambda: P.with_roughness(boxes(0, LARGE), [0.0, 0.3]), False, True),  # its rays are not sorted
    (lambda: P.with_roughness(boxes(2, LARGE), [0.0, 0.3]), True, True),
    (lambda: boxes(0, LARGE), False, False),                               # none to sort
    (lambda: P.slab_scatterers(n_rays=32768, n_scat=500, k_max=2), False, False),
    (lambda: P.slab_scatterers(n_rays=LARGE, n_scat=500, k_max=2), True, True),
])
def test_secondary_ray_jobs_are_sorted_in_large_passes(ctx, make, jobs, recorded):
    w = make()
    assert (launches(ctx, w)["job_sort"] > 0) == jobs
    assert (launches(ctx, w, keep_record=True)["job_sort"] > 0) == recorded


@pytest.mark.parametrize("rough_nee", [0, 1])
def test_recorded_rough_jobs_in_a_large_unsorted_pass(ctx, rough_nee):
    """Two rough layers at more than 2^21 paths (unsorted rays, sorted jobs when recorded): channel data and
    gradient equal the sum over four sub-apertures, whose small passes sort nothing, for one
    dL/dRF, up to the FP32 order of sums (as in test_gpu_edges.py)."""
    w = P.with_roughness(boxes(0, LARGE), [0.0, 0.3])
    acq = dict(w["acq"], rough_nee=rough_nee)
    sid = ctx.upload_workload(w)
    rf, _ = ctx.forward(sid, w["theta"], acq, seed=3, keep_record=True)
    grf = torch.randn(rf.shape, generator=torch.Generator("cuda").manual_seed(1), device="cuda")
    g = ctx.transport_vjp(sid, w["theta"], acq, 3, grf)
    rf_sum, g_sum = torch.zeros_like(rf), torch.zeros_like(g)
    for b in range(4):
        part = dict(acq, tx_elem=16 * b, n_tx_elem=16)
        rf_sum += ctx.forward(sid, w["theta"], part, seed=3, keep_record=True)[0]
        g_sum += ctx.transport_vjp(sid, w["theta"], part, 3, grf)
    assert float(rf.norm()) > 0 and float(g.abs().max()) > 0
    assert float((rf_sum - rf).norm()) <= 1e-5 * float(rf.norm())
    assert torch.allclose(g_sum, g, rtol=1e-4, atol=1e-5 * float(g.abs().max())), (g, g_sum)
    ctx.release_scene(sid)


def test_a_march_of_more_rays_makes_the_same_records(ctx):
    """More than 2^22 rays are claimed 64 at a time: word for word the records of sub-apertures of at most
    2^21 paths, which claim fewer and are not sorted."""
    w = P.slab_scatterers(n_rays=66000, n_scat=2000, k_max=2)
    acq = w["acq"]
    assert acq["n_elem"] * acq["n_rays"] > 1 << 22
    sid = ctx.upload_workload(w)
    ctx.forward(sid, w["theta"], acq, seed=5, keep_record=True)
    full = ctx.record(0, acq["n_elem"] * acq["n_rays"], acq["k_max"]).clone()
    m = 16 * acq["n_rays"]
    for b in range(4):
        ctx.forward(sid, w["theta"], dict(acq, tx_elem=16 * b, n_tx_elem=16), seed=5, keep_record=True)
        assert torch.equal(ctx.record(0, m, acq["k_max"]), full[b * m:(b + 1) * m])
    ctx.release_scene(sid)
