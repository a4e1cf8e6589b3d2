"""Gradients of passes above 2^21 paths: rays and secondary-ray jobs in sorted order, surfaces searched
before scatterers, stored secondary-ray results (record) or chunks traced again (recompute).  The
oracle's cases in the other files are smaller and unsorted; sub-apertures with one seed partition a
pass, so the large pass's channel data and gradients are the sums over small passes, for one dL/dRF.

Tolerance.  Both sides add the same FP32 terms in other orders.  dL/dRF is noise, so a gradient is about
the root of its terms' square sum, and so is, times eps and the root of the longest chain (some
thousand terms per thread), its error: 1e-5 of the gradient; ten times that for a component that
cancels further, and for components far below the largest sensitivity 1e-5 of that (each times its
parameter, as the parameters' units differ)."""
import numpy as np
import pytest
import torch

from paper_2604_15017_gb300 import phantoms as P
from paper_2604_15017_gb300 import usrt
from test_gpu_edges import ctx  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu

SCENES = {
    "slab": lambda n: P.slab_scatterers(n_rays=n, n_scat=4000),
    "rough": lambda n: P.with_roughness(P.hollow_cylinder(n_rays=n), [0.0, 0.2, 0.1]),
    "inclusions": lambda n: P.inclusions(n_regions=3, n_scat=2000, n_rays=n, k_max=4, angles_deg=[4.0], n_elem=64,
                                         n_samples=2048, n_lat=20, n_lon=40),
}


def parts(acq, n=4):
    m = acq["n_elem"] // n
    return [dict(acq, tx_elem=m * b, n_tx_elem=m) for b in range(n)]


def noise(rf):
    return torch.randn(rf.shape, generator=torch.Generator("cuda").manual_seed(2), device="cuda")


def close(a, b, scale):
    a, b = a.double().cpu().numpy() * scale, b.double().cpu().numpy() * scale
    assert np.abs(b).max() > 0
    assert np.all(np.abs(a - b) <= 1e-4 * np.abs(b) + 1e-5 * np.abs(b).max()), np.c_[a, b]


def rel(a, b):
    return float((a.double() - b.double()).norm() / b.double().norm())


@pytest.mark.parametrize("mode", ["record", "recompute"])
@pytest.mark.parametrize("name,n_rays", [("slab", 33000), ("slab", 67000), ("rough", 33000), ("inclusions", 33000)])
def test_large_pass_is_the_sum_of_its_sub_apertures(ctx, name, n_rays, mode):
    # 67,000 rays per element: past 2^22 paths, where recompute traces a sorted chunk and a small one
    w = SCENES[name](n_rays)
    acq, th = w["acq"], w["theta"]
    assert acq["n_elem"] * acq["n_rays"] > 1 << 21
    m = usrt.MODE_RECORD if mode == "record" else usrt.MODE_RECOMPUTE
    sid = ctx.upload_workload(w)
    rf, _ = ctx.forward(sid, th, acq, seed=5, keep_record=mode == "record")
    grf = noise(rf)
    g = ctx.transport_vjp(sid, th, acq, 5, grf, mode=m)
    assert ctx.device_status() == usrt.US_OK
    rf_sum, g_sum = torch.zeros_like(rf), torch.zeros_like(g)
    for a in parts(acq):
        rf_sum += ctx.forward(sid, th, a, seed=5, keep_record=True)[0]
        g_sum += ctx.transport_vjp(sid, th, a, 5, grf)
    assert rel(rf, rf_sum) <= 1e-5
    close(g, g_sum, np.where(th == 0.0, 1.0, np.abs(th)))
    ctx.release_scene(sid)


@pytest.mark.parametrize("name", ["rough", "inclusions"])
def test_acquisition_and_shape_gradients_of_large_passes(ctx, name):
    w = SCENES[name](33000)
    acq, th, nt = w["acq"], w["theta"], len(w["tris"])
    sid = ctx.upload_workload(w)
    rf, _ = ctx.forward(sid, th, acq, seed=5, keep_record=True)
    grf = noise(rf)
    _, ga = ctx.transport_vjp_acq(sid, th, acq, 5, grf)
    _, gt = ctx.transport_vjp_shape(sid, th, acq, 5, grf, nt)
    ga_sum, gt_sum = torch.zeros_like(ga), torch.zeros_like(gt)
    for a in parts(acq):
        ctx.forward(sid, th, a, seed=5, keep_record=True)
        ga_sum += ctx.transport_vjp_acq(sid, th, a, 5, grf)[1]
        gt_sum += ctx.transport_vjp_shape(sid, th, a, 5, grf, nt)[1]
    scale = np.array([acq["c_bf"], acq["pitch"]] + [1.0] * len(acq["angles"]))
    ga, ga_sum = (v.double().cpu().numpy() * scale for v in (ga, ga_sum))
    assert np.all(np.abs(ga - ga_sum) <= 1e-4 * np.abs(ga_sum) + 1e-5 * np.abs(ga_sum).max()), np.c_[ga, ga_sum]
    assert rel(gt, gt_sum) <= 1e-4
    ctx.release_scene(sid)


@pytest.mark.parametrize("name", ["slab", "rough"])
def test_second_stream_of_a_sorted_pass(ctx, name):
    """The job sort and the secondary rays on the lane's second stream against one stream, and against a
    batch's lane."""
    w = SCENES[name](33000)
    sid = ctx.upload_workload(w)
    out = {}
    for opt in (0, 100):
        ctx.set_option(usrt.OPT_NEE_STREAM, opt)
        try:
            rf, b = ctx.forward(sid, w["theta"], w["acq"], w["img"], seed=5, keep_record=True)
            g = ctx.transport_vjp(sid, w["theta"], w["acq"], 5, noise(rf))
        finally:
            ctx.set_option(usrt.OPT_NEE_STREAM, 100)
        out[opt] = rf.clone(), b.clone(), g.clone(), ctx.stats()
    (rf0, b0, g0, s0), (rf1, b1, g1, s1) = out[0], out[100]
    for k in ("segments", "nee_queries", "arrivals", "status"):
        assert s0[k] == s1[k]
    assert rel(rf1, rf0) <= 1e-5
    close(g1, g0, np.where(w["theta"] == 0.0, 1.0, np.abs(w["theta"])))
    bref = b0 + 1.0
    loss, gb = ctx.loss(w["img"], b1, bref)
    rf2, _ = ctx.forward(sid, w["theta"], w["acq"], w["img"], seed=5, keep_record=True)
    gth, _ = ctx.adjoint(sid, w["theta"], w["acq"], w["img"], 5, rf2, gb)
    it = dict(scene=sid, theta=w["theta"], acq=w["acq"], img=w["img"], seed=5, bref=bref)
    o = usrt.Batch(ctx, [it, it]).run()
    torch.cuda.synchronize()
    for v in o:
        assert rel(v["rf"], rf0) <= 1e-5
        assert abs(float(v["loss"]) - float(loss)) <= 1e-3 * abs(float(loss))
        # through the image: the pixels near the clip may fall on either side of it
        assert rel(v["grad"], gth) <= 1e-3
    ctx.release_scene(sid)
