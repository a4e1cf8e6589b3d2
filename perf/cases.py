"""The framework's work as its users ask for it: whole simulations (forward, and forward + loss +
adjoint) through a `usrt.Context`, a batch of requests, and the single stages (splat, delay-and-sum,
envelope and log compression, each with its adjoint), at the sizes of the benchmark, the tests and
the batch generator.

One pass is what a program does once per frame, per optimiser iteration or per call; scenes are
uploaded beforehand, as a program that renders them more than once does.  Outputs are whole.
"""
import math

import numpy as np
import torch

from paper_2604_15017_gb300 import phantoms as P
from paper_2604_15017_gb300 import usrt

MM = 1e-3
FS, BW, F0 = 40e6, 0.6, 5e6  # sampling rate, fractional bandwidth, centre frequency of the phantoms
PITCH = 0.3 * MM

_context = None


def _ctx():
    """A program's one context (scenes and workspaces stay resident in it)."""
    global _context
    if _context is None:
        _context = usrt.Context(0)
    return _context


class _Scene:
    """A resident scene, released with the state that holds it."""

    def __init__(self, w):
        self.id = _ctx().upload_workload(w)

    def __del__(self):
        try:
            _ctx().release_scene(self.id)
        except Exception:
            pass


# --------------------------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------------------------
def _transport(name, scene, n_elem, n_tx, n_rays, k_max, n_samples, n_lines, n_depth, grad, mode="record",
               n_regions=0, n_lat=0, n_scat=0, rough=0.0, f_number=0.0):
    return dict(name=name, kind="transport", scene=scene, n_elem=n_elem, n_tx=n_tx, n_rays=n_rays, k_max=k_max,
                n_samples=n_samples, n_lines=n_lines, n_depth=n_depth, grad=grad, mode=mode, n_regions=n_regions,
                n_lat=n_lat, n_scat=n_scat, rough=rough, f_number=f_number)


def _image(name, kind, n_elem, n_tx, n_samples, n_lines, n_depth, f_number=0.0):
    return dict(name=name, kind=kind, n_elem=n_elem, n_tx=n_tx, n_samples=n_samples, n_lines=n_lines,
                n_depth=n_depth, f_number=f_number)


def listed():
    return [
        # the benchmark's frame: one optimisation step (forward, loss, adjoint) on the inclusion
        # phantom, 16 compounded plane waves, 16 million paths
        _transport("frame_step", "inclusions", 128, 16, 7813, 8, 4096, 256, 1024, "theta", n_regions=12, n_lat=65,
                   n_scat=100000),
        # rendering a medium-sized scene of the batch generator's ranges with the widest array,
        # forward only (data generation)
        _transport("render_wide", "inclusions", 192, 7, 521, 8, 2048, 128, 512, "none", n_regions=5, n_lat=40,
                   n_scat=30000),
        # the two-layer phantom at its stated size, forward only: a first simulation
        _transport("two_layer", "two_layer", 64, 1, 10000, 4, 2048, 128, 1024, "none"),
        # one iteration of the inverse problem at its stated size: 1e5 rays, one plane wave
        _transport("inverse_step", "inclusions", 128, 1, 782, 4, 4096, 256, 1024, "theta", n_regions=12, n_lat=65,
                   n_scat=100000),
        # the same kind of iteration in the mode that keeps no record (memory-bound users), small scene
        _transport("slab_recompute", "slab", 64, 1, 2000, 4, 2048, 128, 1024, "theta", mode="recompute", n_scat=1000),
        # one iteration of the shape-aware inverse problem: rough-walled hollow cylinder, gradient of
        # its vertices and of its radius
        _transport("cylinder_shape", "cylinder", 64, 1, 750, 4, 2048, 128, 512, "shape", n_scat=3000, rough=0.2),
        # calibration of the probe: gradients of sound speed, pitch and steering angles with a
        # dynamic receive aperture, odd numbers of elements, transmits and lines
        _transport("probe_gradient", "inclusions", 95, 5, 997, 6, 2044, 101, 1024, "acq", n_regions=3, n_lat=20,
                   n_scat=3000, f_number=1.5),
        # a batch of uneven requests (half of them with loss and adjoint) on the library's lanes
        dict(name="batch_uneven", kind="batch", n=8, scale=0.25, sizes=4),
        # beamforming recorded channel data at the frame's size: DAS, envelope, log compression
        _image("bmode_frame", "bmode", 128, 16, 4096, 256, 1024),
        # DAS and its transpose as a linear operator pair (iterative reconstruction), odd sizes
        _image("das_pair", "das_pair", 101, 11, 3000, 97, 512),
        # the smallest calls: envelope/log of one image, its loss and its VJP
        _image("envlog_small", "envlog", 0, 0, 0, 128, 512),
        # channel data from an explicit list of arrivals and the splat's adjoint, as many arrivals as
        # the frame makes
        dict(name="splat_pair", kind="splat", n_elem=128, n_tx=16, n_samples=4096, n_arrivals=7900000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["transport", "transport", "transport", "batch", "bmode", "das_pair", "envlog", "splat"])
    n_samples = 4 * rng.randint(256, 1024)
    n_lines, n_depth = rng.randint(31, 256), rng.choice([256, 512, 1024])
    if kind == "batch":
        return dict(kind="batch", n=rng.randint(3, 8), scale=round(0.02 * 12.0 ** rng.random(), 4),
                    sizes=rng.randint(5, 10000))
    if kind == "splat":
        return dict(kind="splat", n_elem=rng.randint(16, 192), n_tx=rng.randint(1, 16), n_samples=n_samples,
                    n_arrivals=_log(rng, 1000, 7900000))
    if kind in ("bmode", "das_pair", "envlog"):
        c = _image("", kind, rng.randint(16, 128), rng.randint(1, 16), n_samples, n_lines, n_depth,
                   rng.choice([0.0, 0.0, 1.5]))
        if kind == "envlog":
            c.update(n_elem=0, n_tx=0, n_samples=0, f_number=0.0, n_depth=rng.choice([64, 256, 1024, 2048]))
        del c["name"]
        return c
    scene = rng.choice(["inclusions", "inclusions", "two_layer", "slab", "cylinder"])
    n_elem = rng.randint(16, 192) if scene != "cylinder" else 64
    n_tx = 1 if scene in ("two_layer", "slab") else rng.randint(1, 9)
    rays_tx = _log(rng, 5000, 400000)
    grad = rng.choice(["none", "theta", "theta", "acq", "shape"])
    c = _transport("", scene, n_elem, n_tx, max(1, rays_tx // n_elem), rng.randint(2, 8), n_samples, n_lines, n_depth,
                   grad, mode=rng.choice(["record", "record", "record", "recompute"]),
                   n_regions=rng.randint(1, 12) if scene == "inclusions" else 0,
                   n_lat=rng.randint(6, 65) if scene == "inclusions" else 0,
                   n_scat=0 if scene == "two_layer" else _log(rng, 1000, 100000 if scene == "inclusions" else 3000),
                   rough=rng.choice([0.0, 0.0, 0.3]) if scene in ("inclusions", "cylinder") else 0.0,
                   f_number=rng.choice([0.0, 0.0, 2.0]))
    del c["name"]
    return c


# --------------------------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------------------------
def _angles(n_tx):
    return [0.0] if n_tx == 1 else list(np.linspace(-15.0, 15.0, n_tx))


def _workload(c, seed):
    """The phantom of a transport case: geometry and scatterers of this seed."""
    s = int(seed)
    if c["scene"] == "inclusions":
        w = P.inclusions(n_regions=c["n_regions"], n_scat=c["n_scat"], n_rays=c["n_rays"], k_max=c["k_max"],
                         n_samples=c["n_samples"], angles_deg=_angles(c["n_tx"]), n_lines=c["n_lines"],
                         n_depth=c["n_depth"], n_elem=c["n_elem"], n_lat=c["n_lat"], n_lon=2 * c["n_lat"],
                         seed_geom=2 * s + 1, seed_scat=2 * s + 2)
        depth = min(60 * MM, 1540.0 * (c["n_samples"] - 1) / (2 * FS))
    elif c["scene"] == "cylinder":
        w = P.hollow_cylinder(n_rays=c["n_rays"], n_scat=c["n_scat"], k_max=c["k_max"], n_elem=c["n_elem"],
                              n_samples=c["n_samples"], angles_deg=_angles(c["n_tx"]), seed_scat=2 * s + 2)
        depth = min(30 * MM, 1540.0 * (c["n_samples"] - 1) / (2 * FS))
    else:
        w = P.two_layer(n_rays=c["n_rays"], k_max=c["k_max"], n_samples=c["n_samples"], n_depth=c["n_depth"],
                        n_lines=c["n_lines"], n_elem=c["n_elem"])
        rng = np.random.default_rng(2 * s + 2)
        # the slab's own density and attenuation differ from one scene to the next
        w["theta"] = w["theta"] * (1.0 + 0.02 * rng.uniform(-1.0, 1.0, len(w["theta"])) * [1, 1, 0, 1, 1, 1, 0, 0])
        if c["scene"] == "slab":
            n = c["n_scat"]
            w["scat_pos"] = np.stack([rng.uniform(-18 * MM, 18 * MM, n), rng.uniform(-2 * MM, 2 * MM, n),
                                      rng.uniform(21 * MM, 37 * MM, n)], axis=1)
            w["scat_amp"] = rng.normal(size=n)
        depth = w["img"]["z1"]
    half = 0.5 * (c["n_elem"] - 1) * PITCH
    w["img"] = P.image(c["n_lines"], c["n_depth"], -half, half, 0.0, depth, lambda1=0.1, f_number=c["f_number"])
    if c["rough"] > 0:
        w = P.with_roughness(w, [0.0] + [c["rough"]] * (w["M"] - 1))
    w["seed"] = 1000003 * s + 17
    w["target"] = P.perturbed_theta(w["theta"], s + 7, frac=0.02)
    return w


def _image_setup(c):
    acq = P.acquisition(c["n_elem"], PITCH, c["n_samples"], _angles(c["n_tx"]), 1, 4, 1540.0)
    half = 0.5 * (c["n_elem"] - 1) * PITCH
    depth = min(60 * MM, 1540.0 * (c["n_samples"] - 1) / (2 * FS))
    return acq, P.image(c["n_lines"], c["n_depth"], -half, half, 0.0, depth, f_number=c["f_number"])


def _band_noise(shape, seed, centre, width):
    """Band-limited noise along the last axis (centre and width as shares of the sampling rate)
    whose strength falls by 30 dB over the record: what channel data and beamformed lines look like."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    n = shape[-1]
    x = torch.randn(shape, generator=g, device="cuda")
    f = torch.arange(n // 2 + 1, device="cuda", dtype=torch.float32) / n
    x = torch.fft.irfft(torch.fft.rfft(x) * torch.exp(-(((f - centre) / width) ** 2)), n=n)
    x = x / x.square().mean().sqrt()
    t = torch.arange(n, device="cuda", dtype=torch.float32) / n
    return (x * torch.pow(10.0, -1.5 * t)).contiguous()


def _rf(c, seed):
    return _band_noise((c["n_tx"], c["n_elem"], c["n_samples"]), seed, F0 / FS, 0.5 * BW * F0 / FS)


def _beamformed(c, seed):
    # 5 MHz over a 1540 m/s image of 40 mm: cycles per pixel
    return _band_noise((c["n_lines"], c["n_depth"]), seed, min(0.25, 260.0 / c["n_depth"]),
                       min(0.08, 80.0 / c["n_depth"]))


def _arrivals(c, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    n, dev = c["n_arrivals"], "cuda"
    tx = torch.randint(0, c["n_tx"], (n,), generator=g, device=dev, dtype=torch.int32)
    e = torch.randint(0, c["n_elem"], (n,), generator=g, device=dev, dtype=torch.int32)
    # some of them lie before the end of the record, some after it
    tau = torch.rand(n, generator=g, device=dev) * (1.05 * c["n_samples"] / FS)
    a = torch.randn(n, generator=g, device=dev) * torch.exp(-3.0 * tau * (FS / c["n_samples"]))
    return tx, e, tau, a


def prepare(case, seed):
    c, ctx, seed = case, _ctx(), int(seed)
    kind = c["kind"]
    if kind == "transport":
        w = _workload(c, seed)
        scene = _Scene(w)
        st = dict(kind=kind, ctx=ctx, scene=scene, theta=w["theta"], acq=w["acq"], img=w["img"], seed=w["seed"],
                  grad=c["grad"], mode=usrt.MODE_RECORD if c["mode"] == "record" else usrt.MODE_RECOMPUTE,
                  n_tris=len(w["tris"]), tangents=None, bref=None)
        if c["grad"] != "none":  # the image to match, rendered with the parameters to recover
            _, bref = ctx.forward(scene.id, w["target"], w["acq"], w["img"], seed=w["seed"])
            st["bref"] = bref.clone()
        if c["grad"] == "shape":  # the vertex tangents of the shape parameters
            t = w.get("dtris_dR")
            if t is None:  # depth of the whole mesh, and its scale
                t = np.stack([np.tile([0.0, 0.0, 1.0], (len(w["tris"]), 3)), np.asarray(w["tris"])])
            t = np.asarray(t).reshape(-1, len(w["tris"]), 9)
            st["tangents"] = torch.tensor(t, dtype=torch.float32, device="cuda")
        return st
    if kind == "batch":
        items, scenes = [], []
        rng = np.random.default_rng(2 * seed + 1)
        for w in P.batch_workloads(n=c["n"], seed=c["sizes"], scale=c["scale"]):
            n = len(w["scat_amp"])
            w["scat_pos"] = rng.uniform([-20 * MM, -20 * MM, 0.0], [20 * MM, 20 * MM, 60 * MM], size=(n, 3))
            w["scat_amp"] = rng.normal(size=n)
            sc = _Scene(w)
            scenes.append(sc)
            it = dict(scene=sc.id, theta=w["theta"], acq=w["acq"], img=w["img"], seed=w["seed"] + 1000003 * seed)
            if w["adjoint"]:
                _, bref = ctx.forward(sc.id, w["theta_target"], w["acq"], w["img"], seed=it["seed"])
                it["bref"] = bref.clone()
            items.append(it)
        return dict(kind=kind, scenes=scenes, batch=usrt.Batch(ctx, items))
    if kind == "splat":
        acq = P.acquisition(c["n_elem"], PITCH, c["n_samples"], _angles(c["n_tx"]), 1, 4, 1540.0)
        return dict(kind=kind, ctx=ctx, acq=acq, arrivals=_arrivals(c, seed), grf=_rf(c, seed + 1))
    if kind == "envlog":
        irf = _beamformed(c, seed)
        img = P.image(c["n_lines"], c["n_depth"], -9 * MM, 9 * MM, 0.0, 40 * MM, lambda1=0.1)
        return dict(kind=kind, ctx=ctx, img=img, irf=irf, bref=ctx.envlog(img, _beamformed(c, seed + 1)))
    acq, img = _image_setup(c)
    st = dict(kind=kind, ctx=ctx, acq=acq, img=img, rf=_rf(c, seed))
    if kind == "das_pair":
        st["gi"] = _beamformed(c, seed + 1)
    return st


# --------------------------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------------------------
def run(st):
    kind = st["kind"]
    if kind == "batch":
        out = []
        for o in st["batch"].run():
            out.append([o["rf"], o["bmode"]] if o["loss"] is None else [o["rf"], o["bmode"], o["loss"], o["grad"]])
        return out
    ctx = st["ctx"]
    if kind == "transport":
        sc, th, acq, img, seed, grad, mode = (st["scene"].id, st["theta"], st["acq"], st["img"], st["seed"], st["grad"],
                                              st["mode"])
        rf, b = ctx.forward(sc, th, acq, img, seed, keep_record=grad != "none" and mode == usrt.MODE_RECORD)
        if grad == "none":
            return dict(rf=rf, bmode=b)
        loss, gb = ctx.loss(img, b, st["bref"])
        out = dict(rf=rf, bmode=b, loss=loss)
        if grad == "theta":
            out["gtheta"], _ = ctx.adjoint(sc, th, acq, img, seed, rf, gb, mode=mode)
        elif grad == "acq":
            out["gtheta"], out["gacq"] = ctx.adjoint_acq(sc, th, acq, img, seed, rf, gb, mode=mode)
        else:
            out["gtheta"], out["gtris"] = ctx.adjoint_shape(sc, th, acq, img, seed, rf, gb, st["n_tris"], mode=mode)
            out["gshape"] = ctx.shape_param_grad(out["gtris"], st["tangents"])
        return out
    if kind == "bmode":
        return ctx.bmode(st["acq"], st["img"], st["rf"])
    if kind == "das_pair":
        return [ctx.das(st["acq"], st["img"], st["rf"]), ctx.das_adjoint(st["acq"], st["img"], st["gi"])]
    if kind == "envlog":
        b = ctx.envlog(st["img"], st["irf"])
        loss, gb = ctx.loss(st["img"], b, st["bref"])
        return [b, loss, gb, ctx.envlog_vjp(st["img"], st["irf"], gb)]
    rf = ctx.splat(st["acq"], F0, *st["arrivals"])
    return [rf, *ctx.splat_adjoint(st["acq"], F0, *st["arrivals"], st["grf"])]


# --------------------------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------------------------
# segments and secondary rays per path, as counted on the phantoms (they depend on the scene's
# density: rounded means), and tree searches of 2 log2(N) box pairs and 4 primitives per query
_PER_PATH = dict(inclusions=(2.4, 1.1), two_layer=(1.3, 0.0), slab=(1.4, 0.1), cylinder=(1.8, 0.5))


def _transport_work(scene, n_paths, n_tris, n_scat, n_rf, n_px, ntx, n_elem, n_samples, grad):
    seg, sec = (n_paths * v for v in _PER_PATH[scene])
    query = 24.0 * 2.0 * math.log2(max(2, n_tris + n_scat)) + 120.0
    taps = float(n_px) * n_elem * ntx
    flops = (seg + sec) * query + seg * 150.0 + (0.5 * sec + 0.05 * n_paths) * 57 * 4 + 4.0 * taps
    nbytes = 44.0 * n_tris + 16.0 * n_scat + 4.0 * (n_rf + n_px)
    if grad != "none":
        flops += seg * 300.0 + (0.5 * sec + 0.05 * n_paths) * 57 * 6 + 4.0 * taps
        nbytes += 4.0 * n_px + (36.0 * n_tris if grad == "shape" else 0.0)
    return dict(bytes=nbytes, flops=flops)


def work(case):
    c, kind = case, case["kind"]
    if kind == "batch":
        tot = dict(bytes=0.0, flops=0.0)
        for w in P.batch_workloads(n=c["n"], seed=c["sizes"], scale=c["scale"]):
            q, im = w["acq"], w["img"]
            ntx = len(q["angles"])
            v = _transport_work("inclusions", ntx * q["n_elem"] * q["n_rays"], len(w["tris"]), len(w["scat_amp"]),
                                ntx * q["n_elem"] * q["n_samples"], im["n_lines"] * im["n_depth"], ntx, q["n_elem"],
                                q["n_samples"], "theta" if w["adjoint"] else "none")
            tot = {k: tot[k] + v[k] for k in tot}
        return tot
    n_rf = float(c["n_tx"]) * c["n_elem"] * c["n_samples"]
    if kind == "splat":
        n = float(c["n_arrivals"])
        return dict(bytes=n * (16 + 12) + 8.0 * n_rf, flops=n * 57 * 10)
    n_px = float(c["n_lines"]) * c["n_depth"]
    fft = 5.0 * math.log2(c["n_depth"])
    if kind == "envlog":
        return dict(bytes=4.0 * n_px * 5, flops=n_px * (6 * fft + 30))
    taps = n_px * c["n_elem"] * c["n_tx"]
    if kind == "bmode":
        return dict(bytes=4.0 * (n_rf + n_px), flops=4.0 * taps + n_px * 2 * fft)
    if kind == "das_pair":
        return dict(bytes=8.0 * (n_rf + n_px), flops=8.0 * taps)
    n_tris = {"inclusions": 4.0 * c["n_lat"] * (c["n_lat"] - 1) * c["n_regions"], "cylinder": 2304.0}.get(c["scene"], 12.0)
    return _transport_work(c["scene"], float(c["n_tx"]) * c["n_elem"] * c["n_rays"], n_tris, c["n_scat"], n_rf, n_px,
                           c["n_tx"], c["n_elem"], c["n_samples"], c["grad"])


# --------------------------------------------------------------------------------------------
# 64-bit values
# --------------------------------------------------------------------------------------------
def _f32(v):
    """A number as the library takes it (float32), in 64 bits."""
    return float(np.float32(v))


def _t64(x):
    return x.to(torch.float64)


def _das_taps(q, im, e, th):
    """(first sample, fraction) of every pixel for one element and steering angle, and its weight."""
    pitch, c, fs = _f32(q["pitch"]), _f32(q["c_bf"]), _f32(q["fs"])
    lin = lambda a, b, n: _f32(a) + (_f32(b) - _f32(a)) * torch.arange(n, device="cuda", dtype=torch.float64) / max(1, n - 1)  # noqa: E731
    x, z = lin(im["x0"], im["x1"], im["n_lines"])[:, None], lin(im["z0"], im["z1"], im["n_depth"])[None, :]
    ne, th = q["n_elem"], _f32(th)
    xe = (e - 0.5 * (ne - 1)) * pitch
    u = (x * math.sin(th) + z * math.cos(th) + 0.5 * (ne - 1) * pitch * abs(math.sin(th))
         + torch.sqrt((x - xe) ** 2 + z * z)) * (fs / c)
    i = torch.floor(u)
    f = _f32(im["f_number"])
    if f > 0:
        xi = (xe - x) / torch.clamp(z / (2 * f), min=pitch)
        w = torch.where(xi.abs() < 1, torch.cos(0.5 * math.pi * xi) ** 2, 0.0)
    else:
        w = torch.tensor(0.5 * (1 - math.cos(2 * math.pi * (e + 1) / (ne + 1))), device="cuda", dtype=torch.float64)
    return i.to(torch.int64), u - i, w


def _das64(q, im, rf):
    rf = torch.nn.functional.pad(_t64(rf), (1, 2))  # one zero before the record, two after it
    out = torch.zeros((im["n_lines"], im["n_depth"]), device="cuda", dtype=torch.float64)
    for t, th in enumerate(q["angles"]):
        for e in range(q["n_elem"]):
            i, f, w = _das_taps(q, im, e, th)
            row, j = rf[t, e], torch.clamp(i + 1, 0, q["n_samples"] + 1)
            a = torch.where(i >= -1, row[j], 0.0)
            b = torch.where((i >= -1) & (i < q["n_samples"]), row[torch.clamp(j + 1, max=q["n_samples"] + 2)], 0.0)
            out += w * ((1 - f) * a + f * b)
    return out


def _das_adjoint64(q, im, gi):
    ns = q["n_samples"]
    out = torch.zeros((len(q["angles"]), q["n_elem"], ns), device="cuda", dtype=torch.float64)
    g = _t64(gi)
    for t, th in enumerate(q["angles"]):
        for e in range(q["n_elem"]):
            i, f, w = _das_taps(q, im, e, th)
            for k, share in ((i, (1 - f) * w * g), (i + 1, f * w * g)):
                ok = (k >= 0) & (k < ns)
                out[t, e].index_add_(0, torch.where(ok, k, 0).reshape(-1), torch.where(ok, share, 0.0).reshape(-1))
    return out


def _hilbert64(x):
    n = x.shape[-1]
    h = torch.zeros(n, device="cuda", dtype=torch.float64)
    h[0] = h[n // 2] = 1.0
    h[1:n // 2] = 2.0
    return torch.fft.ifft(torch.fft.fft(x) * h).imag


def _log64(im, irf):
    y = _hilbert64(irf)
    env = torch.sqrt(irf * irf + y * y)
    db = 20 * torch.log10(env / env.max())
    return y, env, torch.clamp(db, min=-_f32(im["dr_db"])), db > -_f32(im["dr_db"])


def _splat64(q, rows, tau, a):
    """Channel data of the arrivals (row, time, amplitude)."""
    n_rows, ns, fs = len(q["angles"]) * q["n_elem"], q["n_samples"], _f32(q["fs"])
    sigma = 4 * math.log(2) / (math.pi * _f32(q["bw"]) * F0) ** 2
    half = 4 * math.sqrt(sigma)
    out = torch.zeros(n_rows * ns, device="cuda", dtype=torch.float64)
    n0 = torch.ceil((tau - half) * fs).to(torch.int64)
    for k in range(int(2 * half * fs) + 2):
        n = n0 + k
        t = n / fs - tau
        ok = (n >= 0) & (n < ns) & (t <= half)
        s = a * torch.sin(2 * math.pi * F0 * t) * torch.exp(-t * t / sigma)
        out.index_add_(0, torch.where(ok, rows * ns + n, 0), torch.where(ok, s, 0.0))
    return out.reshape(len(q["angles"]), q["n_elem"], ns)


def _splat_adjoint64(q, rows, tau, a, grf):
    ns, fs = q["n_samples"], _f32(q["fs"])
    sigma = 4 * math.log(2) / (math.pi * _f32(q["bw"]) * F0) ** 2
    half, w = 4 * math.sqrt(sigma), 2 * math.pi * F0
    g = _t64(grf).reshape(-1)
    ga, gt, gf = (torch.zeros_like(tau) for _ in range(3))
    n0 = torch.ceil((tau - half) * fs).to(torch.int64)
    for k in range(int(2 * half * fs) + 2):
        n = n0 + k
        t = n / fs - tau
        ok = (n >= 0) & (n < ns) & (t <= half)
        v = torch.where(ok, g[torch.where(ok, rows * ns + n, 0)], 0.0) * torch.exp(-t * t / sigma)
        si, co = torch.sin(w * t), torch.cos(w * t)
        ga += v * si
        gt -= v * a * (w * co - 2 * t / sigma * si)
        gf += v * a * (2 * math.pi * t * co - 2 * t * t / (sigma * F0) * si)
    return ga, gt, gf


def _philox(ray, block, k0, k1):
    """Four 24-bit uniforms per ray of event `block` (transmit 0, stream 0)."""
    m = np.uint64(0xFFFFFFFF)
    c = [ray.astype(np.uint64), np.zeros(len(ray), np.uint64), np.zeros(len(ray), np.uint64),
         np.full(len(ray), block, np.uint64)]
    for r in range(10):
        a, b = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        ka, kb = np.uint64((k0 + r * 0x9E3779B9) & 0xFFFFFFFF), np.uint64((k1 + r * 0xBB67AE85) & 0xFFFFFFFF)
        c = [(b >> np.uint64(32)) ^ c[1] ^ ka, b & m, (a >> np.uint64(32)) ^ c[3] ^ kb, a & m]
    return [(v >> np.uint64(8)).astype(np.float64) / 16777216.0 for v in c]


def _two_layer64(w):
    """(element, time, amplitude) of every arrival of the two-layer phantom (smooth interfaces, no
    scatterers, one transmit), all triangles tested for every ray."""
    q, th = w["acq"], np.float32(w["theta"]).astype(np.float64)
    pitch, hel, ne, nr = _f32(q["pitch"]), _f32(q["h_el"]), q["n_elem"], q["n_rays"]
    c, rho, al = th[0:6:3], th[1:6:3], th[2:6:3]
    kappa = math.log(10) / 20 * 1e-4 * th[7]
    am, ac = _f32(q["alpha_m"]), _f32(q["alpha_c"])
    tris = np.float32(w["tris"]).astype(np.float64)
    v0, e1, e2 = tris[:, 0:3], tris[:, 3:6] - tris[:, 0:3], tris[:, 6:9] - tris[:, 0:3]
    nrm = np.cross(e1, e2)
    nrm /= np.linalg.norm(nrm, axis=1)[:, None]
    k0, k1 = w["seed"] & 0xFFFFFFFF, w["seed"] >> 32
    ray = np.arange(ne * nr)
    u = _philox(ray, 0, k0, k1)
    o = np.stack([(ray // nr - 0.5 * (ne - 1) + u[0] - 0.5) * pitch, (u[1] - 0.5) * hel, 0 * u[0]], 1)
    r, ph = np.sqrt(u[2]), 2 * math.pi * u[3]
    d = np.stack([r * np.cos(ph), r * np.sin(ph), np.sqrt(1 - u[2])], 1)
    a, tau, med = np.full(len(ray), math.pi / nr), np.zeros(len(ray)), np.zeros(len(ray), np.int64)
    out = []
    for k in range(q["k_max"] + 1):
        best, hit = np.full(len(ray), np.inf), np.full(len(ray), -1)
        with np.errstate(divide="ignore", invalid="ignore"):
            t = -o[:, 2] / d[:, 2]
            x, y = o[:, 0] + t * d[:, 0], o[:, 1] + t * d[:, 1]
            arr = (d[:, 2] < 0) & (t > 1e-7) & (np.abs(x) <= 0.5 * ne * pitch) & (np.abs(y) <= 0.5 * hel)
            best[arr], hit[arr] = t[arr], len(tris)
            for j in range(len(tris)):
                p = np.cross(d, e2[j])
                inv = 1.0 / (p @ e1[j])
                tv = o - v0[j]
                b1 = np.einsum("ij,ij->i", tv, p) * inv
                qv = np.cross(tv, e1[j])
                b2 = np.einsum("ij,ij->i", d, qv) * inv
                tj = (qv @ e2[j]) * inv
                ok = (b1 >= 0) & (b2 >= 0) & (b1 + b2 <= 1) & (tj > 1e-7) & (tj < best)
                best[ok], hit[ok] = tj[ok], j
        live = hit >= 0
        ray, o, d, a, tau, med, best, hit, x = (v[live] for v in (ray, o, d, a, tau, med, best, hit, x))
        a = a * np.exp(-kappa * al[med] * best)
        tau = tau + best / c[med]
        arr = hit == len(tris)
        ang = np.arccos(np.clip(-d[:, 2], -1, 1))
        f = np.clip((ac - ang) / (ac - am), 0.0, 1.0)
        sel = arr & (f > 0)
        e = np.clip(np.floor((x + 0.5 * ne * pitch) / pitch), 0, ne - 1).astype(np.int64)
        out.append((e[sel], tau[sel], (a * f)[sel]))
        if k == q["k_max"]:
            break
        keep = ~arr
        ray, o, d, a, tau, best, hit = (v[keep] for v in (ray, o, d, a, tau, best, hit))
        u0 = _philox(ray, k + 1, k0, k1)[0]
        n = nrm[hit]
        dn = np.einsum("ij,ij->i", d, n)
        m1 = np.where(dn < 0, 0, 1)
        n = np.where((dn < 0)[:, None], n, -n)
        m2, ci = 1 - m1, np.abs(dn)
        ratio = c[m2] / c[m1]
        st2 = ratio ** 2 * np.clip(1 - ci ** 2, 0, None)
        tir = st2 >= 1
        ct = np.sqrt(np.clip(1 - st2, 0, None))
        za, zb = rho[m2] * c[m2] * ci, rho[m1] * c[m1] * ct
        R = np.where(tir, 1.0, (za - zb) / (za + zb))
        refl = tir | (u0 < R * R)
        with np.errstate(divide="ignore", invalid="ignore"):
            a = a * np.where(tir, 1.0, np.where(refl, 1.0 / R, (1 + R) / (1 - R * R)))
        o = o + d * best[:, None]
        d = np.where(refl[:, None], d + 2 * ci[:, None] * n, ratio[:, None] * d + (ratio * ci - ct)[:, None] * n)
        med = np.where(refl, m1, m2)
    return [np.concatenate(v) for v in zip(*out)]


def exact(case, seed):
    """64-bit values of the single stages and of the two-layer simulation.  The other transport cases
    have none: every ray against up to 3e5 primitives, and the derivative of the whole path, take far
    longer than a few seconds."""
    c, kind, seed = case, case["kind"], int(seed)
    if kind == "splat":
        acq = P.acquisition(c["n_elem"], PITCH, c["n_samples"], _angles(c["n_tx"]), 1, 4, 1540.0)
        tx, e, tau, a = _arrivals(c, seed)
        rows, tau, a = tx.to(torch.int64) * c["n_elem"] + e.to(torch.int64), _t64(tau), _t64(a)
        return [_splat64(acq, rows, tau, a), *_splat_adjoint64(acq, rows, tau, a, _rf(c, seed + 1))]
    if kind == "bmode":
        acq, img = _image_setup(c)
        return _log64(img, _das64(acq, img, _rf(c, seed)))[2]
    if kind == "das_pair":
        acq, img = _image_setup(c)
        return [_das64(acq, img, _rf(c, seed)), _das_adjoint64(acq, img, _beamformed(c, seed + 1))]
    if kind == "envlog":
        im = dict(dr_db=60.0)
        irf, l1, l2, n = _t64(_beamformed(c, seed)), _f32(0.1), 1.0, c["n_lines"] * c["n_depth"]
        y, env, b, live = _log64(im, irf)
        r = b - _log64(im, _t64(_beamformed(c, seed + 1)))[2]
        gb = (l1 * torch.sign(r) + 2 * l2 * r) / n
        k = 20 / math.log(10)
        ge = torch.where(live, gb * k / env, 0.0)
        top = int(env.argmax())
        ge.view(-1)[top] -= k * (gb * live).sum() / env.max()
        gi = irf / env * ge - _hilbert64(y / env * ge)
        return [b, (l1 * r.abs().sum() + l2 * r.square().sum()) / n, gb, gi]
    if kind == "transport" and c["scene"] == "two_layer" and c["grad"] == "none":
        w = _workload(c, seed)
        e, tau, a = _two_layer64(w)
        dev = lambda v: torch.from_numpy(v).to("cuda")  # noqa: E731
        rf = _splat64(w["acq"], dev(e), dev(tau), dev(a))
        return dict(rf=rf, bmode=_log64(w["img"], _das64(w["acq"], w["img"], rf))[2])
    return None
