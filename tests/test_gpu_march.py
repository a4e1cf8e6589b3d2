"""Closest hits at the edges of the kernels' work distribution, against the FP64 oracle: queues
smaller than a warp, around one item per resident warp and past one full wave; grid cells that
hold more spheres than a record (chains of records), clusters on cell faces, grids one cell
thick.  Checked is what the queries decide: the event sequences (>= 99.99 % of the paths) and the
channel data (1e-4 relative L2), as in test_gpu_edges.py; the image of a dense cloud has dark pixels
that amplify the RF's rounding past that file's 0.05 dB."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2604_15017_gb300 import phantoms as P
from test_gpu_edges import ctx, no_triangles, rel_l2  # noqa: F401  (ctx: the fixture)

pytestmark = pytest.mark.gpu

MM = 1e-3


def parity(ctx, w):
    sid = ctx.upload_workload(w)
    rf, _ = ctx.forward(sid, w["theta"], w["acq"], seed=w["seed"], keep_record=True)
    torch.cuda.synchronize()
    st = ctx.stats()
    assert st["status"] == 0 and st["dropped"] == 0
    acq = w["acq"]
    rec = ctx.record(0, len(acq["angles"]) * acq["n_elem"] * acq["n_rays"], acq["k_max"]).cpu().numpy()
    ref = O.forward(w)
    ora = ref["run"].records()
    r = rec.astype(np.int64) & 0xFFFFFFFF
    same = (((r >> 20) & 3) == ora["cls"]) & (((r & 0xFFFFF) == ora["id"]) | (ora["cls"] == 0))
    assert same.all(axis=1).mean() >= 0.9999
    rf_g = rf.double().cpu().numpy()
    assert rel_l2(rf_g, ref["rf"]) <= 1e-4 if np.abs(ref["rf"]).max() > 0 else np.all(rf_g == 0)
    ctx.release_scene(sid)


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


@pytest.mark.parametrize("make", [
    lambda: P.slab_scatterers(n_rays=33000, n_scat=4000),
    lambda: P.with_roughness(P.hollow_cylinder(n_rays=33000), [0.0, 0.2, 0.0]),
    lambda: P.inclusions(n_regions=3, n_scat=2000, n_rays=33000, angles_deg=[0.0], n_elem=64, n_samples=2048, n_lat=20,
                         n_lon=40),
    lambda: no_triangles(P.slab_scatterers(n_rays=33000, n_scat=4000)),
    lambda: P.hollow_cylinder(n_rays=33000, n_scat=1),
], ids=["slab", "rough", "inclusions", "scatterers", "surfaces"])
def test_small_and_large_passes_decide_alike(ctx, make):
    """A pass of more than 2^21 paths sorts its rays and searches surfaces before scatterers; one of
    fewer searches both at once, unsorted.  Sub-apertures partition the full aperture's
    realisation, so four small passes make the large one's records, word for word."""
    w = make()
    acq = w["acq"]
    n = acq["n_elem"] * acq["n_rays"]
    assert n > 1 << 21
    sid = ctx.upload_workload(w)
    ctx.forward(sid, w["theta"], acq, seed=5, keep_record=True)
    full = ctx.record(0, n, acq["k_max"])
    st = ctx.stats()
    segments = arrivals = 0
    for b in range(4):
        part = dict(acq, tx_elem=16 * b, n_tx_elem=16)
        ctx.forward(sid, w["theta"], part, seed=5, keep_record=True)
        m = 16 * acq["n_rays"]
        assert torch.equal(ctx.record(0, m, acq["k_max"]), full[b * m:(b + 1) * m])
        s = ctx.stats()
        assert s["status"] == 0
        segments += s["segments"]
        arrivals += s["arrivals"]
    assert (segments, arrivals) == (st["segments"], st["arrivals"])
    ctx.release_scene(sid)
