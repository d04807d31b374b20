"""The work that users of this framework have it do, as measurable cases.

A case is one call, or the few calls of one step, of motion-compensated
cone-beam reconstruction: backprojection of filtered projections, its
vector-Jacobian products, a motion-estimation step or job, a batch of served
jobs, and the filtering that comes before.  Geometry: a circular short scan
(source-isocenter 750 mm, source-detector 1200 mm, 200 degrees) or the full
circle, ellipsoid head phantoms with closed-form line integrals, cosine,
short-scan and Shepp-Logan filtering, smooth rigid motion per view.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2401_09283_gb300 import autograd as AG
from paper_2401_09283_gb300 import bp
from paper_2401_09283_gb300 import job as J

DEV = "cuda"
DTYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}


# ------------------------------------------------------------------- the cases

def _scan(name, kind, shape, spacing, views, det, pitch, **kw):
    """A case on one scan: volume (nz, ny, nx) voxels of `spacing` mm, `views`
    views, detector (nv, nu) pixels of `pitch` mm."""
    c = dict(kind=kind, nz=shape[0], ny=shape[1], nx=shape[2], spacing=spacing, views=views,
             nv=det[0], nu=det[1], pitch=pitch, arc=200.0, sid=750.0, sdd=1200.0, dtype="f32",
             scale=False, weight="fdk", deriv="central", want="motion", trans=5.0, rot=3.0,
             knots=12, noise=0.01, nodes=0, iters=1, loss="sharpness", opt="adam")
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: a gradient check's instance, where launches and
        # host work are all there is; exact derivative, both gradients
        _scan("autograd-16", "autograd", (16, 16, 16), 4.0, 12, (24, 32), 6.4, deriv="exact",
              want="both", trans=3.0, rot=2.0, knots=6, noise=0.0),
        # one registration step at a small size, call by call as a script does
        # it: forward, sharpness loss, motion gradient, Adam update
        _scan("step-64", "step", (64, 64, 64), 1.0, 60, (96, 128), 1.6, trans=3.0, rot=2.0,
              knots=6, noise=0.0),
        # a head-size reconstruction
        _scan("forward-256", "forward", (256, 256, 256), 1.0, 248, (480, 616), 0.616),
        # its motion gradient, the largest part of motion estimation
        _scan("vjp-motion-256", "vjp", (256, 256, 256), 1.0, 248, (480, 616), 0.616),
        # motion and data gradients in one call, as learned pipelines need them
        _scan("vjp-both-256", "vjp", (256, 256, 256), 1.0, 248, (480, 616), 0.616, want="both"),
        # forward and backward through torch.autograd with the spline motion
        # model, gradients to the projections and to the spline's nodes
        _scan("autograd-192", "autograd", (192, 192, 192), 1.33, 180, (240, 320), 1.30,
              want="both", trans=3.0, rot=2.0, knots=6, noise=0.0, nodes=12),
        # the largest reconstruction, projections stored in half precision
        _scan("forward-512-f16", "forward", (512, 512, 512), 0.5, 496, (960, 1240), 0.308,
              dtype="f16", trans=3.0, rot=2.0, knots=6, noise=0.0),
        # a served job's largest volume, bfloat16 storage with a scale per view
        _scan("vjp-motion-384-bf16", "vjp", (384, 384, 384), 2.0 / 3.0, 248, (366, 488), 0.8533,
              dtype="bf16", scale=True),
        # motion estimation of one scan on the full circle: job, iterations of
        # the decaying gradient step on spline nodes, read-back
        _scan("job-128", "job", (128, 128, 128), 2.0, 360, (500, 700), 0.64, arc=360.0, sid=785.0,
              trans=5.0, rot=5.0, knots=10, nodes=30, opt="gd", iters=10),
        # serving: jobs of several sizes in half precision advanced as a batch
        dict(name="batch-serving-f16", kind="batch", jobs="128x120,192x120,128x248,256x120",
             dtype="f16", iters=5, loss="tv", opt="adam", noise=0.01),
        # FDK preprocessing of a head-size scan, once per scan
        _scan("filter-616", "filter", (256, 256, 256), 1.0, 248, (480, 616), 0.616, ext=0),
        # a clinical-looking odd size: no dimension fits a tile or a 16-byte
        # row, plain backprojection weight, forward and both gradients
        _scan("ragged-bf16", "ragged", (143, 187, 161), 1.3, 111, (301, 401), 1.03, dtype="bf16",
              scale=True, weight="none", want="both"),
    ]


def draw(rng):
    """One more case of the ranges above; no more work than the largest listed."""
    def logu(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["forward", "forward", "vjp", "vjp", "vjp", "autograd", "step", "job",
                       "batch", "filter", "ragged"])
    if kind == "batch":
        n = rng.randint(2, 6)
        jobs = ",".join("%dx%d" % (rng.choice([128, 192, 256]), rng.choice([120, 248]))
                        for _ in range(n))
        return dict(kind="batch", jobs=jobs, dtype=rng.choice(["f32", "f16", "bf16"]),
                    iters=rng.randint(2, 5), loss=rng.choice(["tv", "sharpness"]),
                    opt="adam", noise=0.01)
    if kind == "filter":
        nu = logu(96, 1400)
        nv = max(1, int(nu * rng.uniform(0.5, 0.9)))
        views = min(logu(12, 500), max(4, int(3e8 / (nu * nv))))
        return _scan(None, "filter", (64, 64, 64), 1.0, views, (nv, nu), 379.5 / nu,
                     ext=rng.choice([0, 0, nu // 10]), arc=rng.choice([200.0, 220.0, 360.0]))
    cap = {"forward": 6.5e10, "vjp": 1.3e10, "autograd": 4e9, "step": 1e9, "job": 6e8,
           "ragged": 3e9}[kind]
    for _ in range(1000):
        n = logu(16, 512 if kind == "forward" else 384)
        shape = tuple(max(8, int(n * rng.uniform(0.6, 1.0))) for _ in range(3))
        views = logu(12, 496)
        if shape[0] * shape[1] * shape[2] * views <= cap:
            break
    spacing = 256.0 / n * rng.uniform(0.8, 1.0)
    nu = int(min(1240, max(24, n * rng.uniform(1.2, 2.6))))
    nv = max(16, int(nu * rng.uniform(0.7, 0.8)))
    if kind != "ragged" and rng.random() < 0.7:  # most detectors are a multiple of 8 wide
        nu = (nu + 7) // 8 * 8
    kw = dict(dtype=rng.choice(["f32", "f32", "f16", "bf16"]),
              weight=rng.choice(["fdk", "fdk", "none"]), deriv=rng.choice(["central"] * 3 + ["exact"]),
              want=rng.choice(["motion", "motion", "both", "data"]), trans=rng.uniform(1.0, 5.0),
              rot=rng.uniform(0.5, 4.0), knots=rng.randint(4, 12),
              loss=rng.choice(["tv", "sharpness"]))
    kw["scale"] = kw["dtype"] != "f32" and rng.random() < 0.5
    if kind == "ragged":
        kw["want"] = "both"
    if kind == "autograd":
        kw.update(dtype="f32", scale=False, want="both", nodes=rng.choice([0, 8, 30]))
    if kind in ("job", "step"):
        kw.update(deriv="central", want="motion", dtype=rng.choice(["f32", "f16"]), scale=False)
    if kind == "job":
        kw.update(nodes=rng.choice([0, 12, 30]), iters=rng.randint(4, 10),
                  opt=rng.choice(["adam", "gd"]))
    return _scan(None, kind, shape, spacing, views, (nv, nu), 414.0 / nu, **kw)


# ---------------------------------------------------------------------- inputs

def _origin(c):
    return tuple(-(c[k] - 1) / 2.0 * c["spacing"] for k in ("nx", "ny", "nz"))


def _angles(c):
    arc, V = math.radians(c["arc"]), c["views"]
    if c["arc"] >= 360.0:
        return np.arange(V) * (arc / V)
    return -arc / 2 + np.arange(V) * (arc / (V - 1))


def _delta_beta(c):
    return math.radians(c["arc"]) / (c["views"] if c["arc"] >= 360.0 else c["views"] - 1)


def _matrices(c):
    f = c["sdd"] / c["pitch"]
    K = np.array([[f, 0, (c["nu"] - 1) / 2], [0, f, (c["nv"] - 1) / 2], [0, 0, 1.0]])
    P = np.zeros((c["views"], 3, 4))
    for j, b in enumerate(_angles(c)):
        co, si = math.cos(b), math.sin(b)
        R = np.array([[-si, co, 0], [0, 0, 1.0], [-co, -si, 0]])
        P[j] = K @ np.hstack([R, (-R @ (c["sid"] * np.array([co, si, 0])))[:, None]])
    return P


def _rigid(th):
    """T (V,4,4) and dT/dtheta (V,6,4,4), float64 tensors; R = Rz Ry Rx."""
    V = th.shape[0]
    s, co = torch.sin(th[:, 3:]), torch.cos(th[:, 3:])
    o, l = torch.zeros(V, dtype=th.dtype, device=th.device), torch.ones(V, dtype=th.dtype,
                                                                      device=th.device)

    def mat(*rows):
        return torch.stack([torch.stack(r, -1) for r in rows], -2)

    def rots(a, d):
        S, C, one = (s[:, a], co[:, a], l) if not d else (co[:, a], -s[:, a], o)
        if a == 0:
            return mat((one, o, o), (o, C, -S), (o, S, C))
        if a == 1:
            return mat((C, o, S), (o, one, o), (-S, o, C))
        return mat((C, -S, o), (S, C, o), (o, o, one))

    def R(d):
        return rots(2, d == 2) @ rots(1, d == 1) @ rots(0, d == 0)

    T = torch.zeros(V, 4, 4, dtype=th.dtype, device=th.device)
    T[:, :3, :3], T[:, :3, 3], T[:, 3, 3] = R(-1), th[:, :3], 1.0
    D = torch.zeros(V, 6, 4, 4, dtype=th.dtype, device=th.device)
    for a in range(3):
        D[:, a, a, 3] = 1.0
        D[:, 3 + a, :3, :3] = R(a)
    return T, D


def _motion(c, rng):
    """Smooth zero-mean motion: cosine interpolation between random knots."""
    V, n = c["views"], c["knots"]
    x = np.linspace(0, n - 1, V)
    i = np.minimum(x.astype(int), n - 2)
    f = 0.5 - 0.5 * np.cos(np.pi * (x - i))
    out = np.zeros((V, 6))
    for m, A in enumerate([c["trans"]] * 3 + [math.radians(c["rot"])] * 3):
        y = rng.uniform(-A, A, n)
        t = y[i] * (1 - f) + y[i + 1] * f
        t -= t.mean()
        out[:, m] = t * (A / max(np.abs(t).max(), 1e-12))
    return out


def _raw(c, P, rng):
    """Line integrals (V, nv, nu) float32 of a random ellipsoid head."""
    V, nv, nu = c["views"], c["nv"], c["nu"]
    R = min(0.45 * max(c["nx"], c["ny"], c["nz"]) * c["spacing"], 105.0)
    skull = np.array([0.7, 0.9, 0.8]) * R
    cen, axe, rho = [np.zeros(3)] * 2, [skull, 0.9 * skull], [1.0, -0.8]
    for _ in range(12):
        a = rng.uniform(0.03, 0.25, 3) * R
        d = rng.standard_normal(3)
        cen.append(d / np.linalg.norm(d) * rng.uniform(0, 0.6) * skull)
        axe.append(a)
        rho.append(rng.uniform(-0.1, 0.3))
    shift = np.array([[1, 0, (nu - 1) / 2], [0, 1, (nv - 1) / 2], [0, 0, 1.0]])
    Mi = np.linalg.inv(P[:, :, :3])
    S = -np.einsum("vij,vj->vi", Mi, P[:, :, 3])
    Mi = Mi @ shift  # rays of pixels counted from the detector centre

    def poly(Q):  # (V,3,3) quadratic form of (u, v, 1) -> 6 coefficients
        k = np.stack([Q[:, 2, 2], 2 * Q[:, 0, 2], 2 * Q[:, 1, 2], Q[:, 0, 0], 2 * Q[:, 0, 1],
                      Q[:, 1, 1]], 1)
        return torch.as_tensor(k, dtype=torch.float32, device=DEV)[:, :, None, None]

    u = (torch.arange(nu, device=DEV) - (nu - 1) / 2).float()[None, None, :]
    v = (torch.arange(nv, device=DEV) - (nv - 1) / 2).float()[None, :, None]

    def ev(k):
        return (k[:, 0] + k[:, 2] * v + k[:, 5] * v * v) + ((k[:, 1] + k[:, 4] * v) + k[:, 3] * u) * u

    terms = []
    for x, a, r in zip(cen, axe, rho):
        Q = np.linalg.qr(rng.standard_normal((3, 3)))[0] if len(terms) > 1 else np.eye(3)
        A = Q.T / a[:, None]
        G = A @ Mi
        oe = (S - x) @ A.T
        qa = np.einsum("vki,vkj->vij", G, G)
        qb = np.einsum("vk,vki->vi", oe, G)
        disc = qb[:, :, None] * qb[:, None, :] - qa * ((oe * oe).sum(1) - 1.0)[:, None, None]
        terms.append((poly(qa), poly(disc), 2.0 * r))
    dd = poly(np.einsum("vki,vkj->vij", Mi, Mi))
    out = torch.empty(V, nv, nu, device=DEV)
    step = max(1, int(4e7 / (nu * nv)))
    for j in range(0, V, step):
        e = slice(j, min(V, j + step))
        acc = 0.0
        for qa, disc, r in terms:
            acc = acc + r * ev(disc[e]).clamp_(min=0).sqrt_() / ev(qa[e])
        out[e] = acc * ev(dd[e]).sqrt_()
    if c["noise"] > 0:
        g = torch.Generator(device=DEV).manual_seed(int(rng.integers(1 << 31)))
        out.add_(torch.randn(out.shape, generator=g, device=DEV), alpha=c["noise"] * 0.3 * R)
    return out


def _parker(c):
    """Short-scan weights (V, nu) float64; 1/2 on the full circle."""
    if c["arc"] >= 360.0:
        return np.full((c["views"], c["nu"]), 0.5)
    arc = math.radians(c["arc"])
    d = (arc - math.pi) / 2
    b = (np.arange(c["views"]) * _delta_beta(c))[:, None]
    g = np.arctan((np.arange(c["nu"]) - (c["nu"] - 1) / 2) * c["pitch"] / c["sdd"])[None]
    with np.errstate(divide="ignore", invalid="ignore"):
        up = np.sin(math.pi / 4 * b / (d + g)) ** 2
        dn = np.sin(math.pi / 4 * (math.pi + 2 * d - b) / (d - g)) ** 2
    return np.clip(np.where(b < 2 * d + 2 * g, up, np.where(b > math.pi + 2 * g, dn, 1.0)), 0, 1)


def _filtered(c, raw, dtype=torch.float32):
    """Cosine and short-scan weights, Shepp-Logan ramp along u (by FFT)."""
    V, nv, nu = raw.shape
    ext, tau = c.get("ext", 0), c["pitch"] * c["sid"] / c["sdd"]
    x = (torch.arange(nu, device=DEV, dtype=torch.float64) - (nu - 1) / 2) * c["pitch"]
    y = (torch.arange(nv, device=DEV, dtype=torch.float64) - (nv - 1) / 2) * c["pitch"]
    cosw = c["sdd"] / torch.sqrt(c["sdd"] ** 2 + x[None] ** 2 + y[:, None] ** 2)
    park = torch.as_tensor(_parker(c), device=DEV)
    n = nu + 2 * ext
    L = 1 << (2 * n - 1).bit_length()
    m = torch.arange(L, device=DEV, dtype=torch.float64)
    m = torch.minimum(m, L - m)
    h = torch.where(m < n, -2.0 / (math.pi ** 2 * tau ** 2 * (4 * m * m - 1)), 0.0)
    H = torch.fft.rfft(h).real.to(dtype)
    fall = (1 - torch.arange(1, ext + 1, device=DEV, dtype=torch.float64) / max(ext, 1)).to(dtype)
    out = torch.empty(V, nv, nu, device=DEV, dtype=dtype)
    for j in range(0, V, 16):
        p = raw[j:j + 16].to(dtype) * (cosw[None] * park[j:j + 16, None, :]).to(dtype)
        if ext:
            p = torch.cat([p[..., :1] * fall.flip(0), p, p[..., -1:] * fall], -1)
        q = torch.fft.irfft(torch.fft.rfft(p, n=L) * H, n=L)
        out[j:j + 16] = q[..., ext:ext + nu] * tau
    return out


def _inputs(c, seed):
    """Everything of one scan: stored projections, matrices, motion, weights."""
    rng = np.random.default_rng(seed)
    P, th = _matrices(c), _motion(c, rng)
    Pm = P @ _rigid(torch.as_tensor(th))[0].numpy()
    raw = _raw(c, Pm, rng)
    s = dict(P=torch.as_tensor(P, device=DEV), theta=torch.as_tensor(th, device=DEV),
             vw=torch.full((c["views"],), _delta_beta(c) if c["weight"] == "fdk" else 1.0,
                           dtype=torch.float64, device=DEV), view_scale=None)
    if c["kind"] == "filter":
        s["raw"] = raw
        return s
    proj = _filtered(c, raw)
    del raw
    if c["scale"]:
        s["view_scale"] = proj.abs().amax((1, 2)).clamp_(min=1e-6).contiguous()
        proj = proj / s["view_scale"][:, None, None]
    s["proj"] = proj.to(DTYPES[c["dtype"]])
    if c["kind"] in ("vjp", "ragged", "autograd"):
        g = torch.Generator(device=DEV).manual_seed(int(rng.integers(1 << 31)))
        s["delta"] = torch.randn((c["nz"], c["ny"], c["nx"]), generator=g, device=DEV)
    if c["nodes"]:  # spline node values near the motion, as an estimate under way
        k = np.linspace(0, c["views"] - 1, c["nodes"]).round().astype(int)
        amp = np.array([0.2 * c["trans"]] * 3 + [0.2 * math.radians(c["rot"])] * 3)
        s["nodes"] = torch.as_tensor(th[k] + amp * rng.uniform(-1, 1, (c["nodes"], 6)), device=DEV)
    return s


def _job_cases(c):
    """The scans of a batch: 256 mm field of view, pixels of 0.6 to 1.6 mm."""
    out = []
    for part in c["jobs"].split(","):
        n, views = (int(x) for x in part.split("x"))
        pitch = min(max(0.8 * 256.0 / n * 1.6, 0.6), 1.6)
        nu = (int(math.ceil(414.0 / pitch)) + 7) // 8 * 8
        out.append(_scan(None, "job", (n, n, n), 256.0 / n, views, (int(math.ceil(0.75 * nu)), nu),
                         pitch, dtype=c["dtype"], loss=c["loss"], opt=c["opt"], iters=c["iters"],
                         noise=c["noise"]))
    return out


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "batch":
        return dict(c=c, jobs=[(k, _inputs(k, seed * 64 + i)) for i, k in enumerate(_job_cases(c))])
    s = dict(c=c, geo=dict(spacing=(c["spacing"],) * 3, origin=_origin(c), sid=c["sid"]),
             shape=(c["nz"], c["ny"], c["nx"]), **_inputs(c, seed))
    if c["kind"] == "autograd":
        s["proj"].requires_grad_(True)
        leaf = s["nodes"] if c["nodes"] else s["theta"]
        s["leaf"] = leaf.clone().requires_grad_(True)
    return s


# ------------------------------------------------------------------- the passes

def _forward(s):
    c = s["c"]
    return bp.bp_forward(s["proj"], s["P"], s["theta"], vol_shape=s["shape"], view_weight=s["vw"],
                         weight=c["weight"], view_scale=s["view_scale"], **s["geo"])


def _vjp(s, dvol, want):
    c = s["c"]
    gm, _, gd = bp.bp_vjp(dvol, s["proj"], s["P"], s["theta"], view_weight=s["vw"],
                          weight=c["weight"], deriv=c["deriv"], view_scale=s["view_scale"],
                          want_motion=want != "data", want_proj=want != "motion", **s["geo"])
    return {k: v for k, v in (("dmotion", gm), ("dproj", gd)) if v is not None}


def _make_job(c, s):
    lr, lr_rot = (0.2, 0.004) if c["opt"] == "adam" else (20.0, 2e-3)
    return J.MotionJob(s["proj"], s["P"], vol_shape=(c["nz"], c["ny"], c["nx"]),
                       spacing=(c["spacing"],) * 3, origin=_origin(c), sid=c["sid"],
                       view_weight=s["vw"], weight=c["weight"], deriv=c["deriv"],
                       view_scale=s["view_scale"], optimizer=c["opt"], lr=lr, lr_rot=lr_rot,
                       loss=c["loss"], motion_nodes=c["nodes"], max_iters=c["iters"])


def run(state):
    c = state["c"]
    kind = c["kind"]
    if kind == "forward":
        return _forward(state)
    if kind == "vjp":
        return _vjp(state, state["delta"], c["want"])
    if kind == "ragged":
        return {"vol": _forward(state), **_vjp(state, state["delta"], "both")}
    if kind == "filter":
        return bp.bp_fdk_filter(state["raw"], pitch=c["pitch"], sid=c["sid"], sdd=c["sdd"],
                                arc=math.radians(c["arc"]), ext=c["ext"])
    if kind == "step":
        vol = _forward(state)
        loss, dvol = bp.bp_tv(vol) if c["loss"] == "tv" else bp.bp_sharpness(vol)
        g = _vjp(state, dvol, "motion")["dmotion"]
        theta = state["theta"].clone()
        m1, m2 = torch.zeros_like(theta), torch.zeros_like(theta)
        bp.bp_adam_step(theta, g, m1, m2, 0.01, 1)
        return {"vol": vol, "loss": loss, "dvol": dvol, "dmotion": g, "theta": theta}
    if kind == "autograd":
        motion = AG.akima_motion(state["leaf"], c["views"]) if c["nodes"] else state["leaf"]
        vol = AG.backproject(state["proj"], motion, state["P"], vol_shape=state["shape"],
                             view_weight=state["vw"], weight=c["weight"], deriv=c["deriv"],
                             **state["geo"])
        gp, gl = torch.autograd.grad(vol, (state["proj"], state["leaf"]), state["delta"])
        return {"vol": vol.detach(), "dproj": gp, "dleaf": gl}
    if kind == "job":
        job = _make_job(c, state)
        job.step(c["iters"])
        theta, hist, _ = job.motion()
        job.close()
        return {"theta": theta, "loss": hist}
    jobs = [_make_job(k, s) for k, s in state["jobs"]]
    batch = J.Batch(max_jobs=len(jobs))
    batch.set_jobs(jobs)
    batch.step(c["iters"])
    out = [j.motion()[:2] for j in jobs]
    batch.close()
    for j in jobs:
        j.close()
    return out


# --------------------------------------------------------------- necessary work

def _flops_bytes(c, iters=1, motion=False, data=False, fwd=False, loss=False):
    vox, px = c["nx"] * c["ny"] * c["nz"], c["views"] * c["nu"] * c["nv"]
    e = 4 if c["dtype"] == "f32" else 2
    ops = (28 if fwd else 0) + (50 if motion else 0) + (16 if data else 0)
    by = (px * e + 4 * vox if fwd else 0) + (px * e + 4 * vox if motion else 0)
    by += 4 * px + (0 if motion else 4 * vox) if data else 0
    by += 8 * vox if loss else 0
    return iters * by, iters * (ops * vox * c["views"] + (30 * vox if loss else 0))


def work(case):
    c = case
    kind = c["kind"]
    if kind == "batch":
        parts = [_flops_bytes(k, c["iters"], motion=True, fwd=True, loss=True)
                 for k in _job_cases(c)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    if kind == "filter":
        px, n = c["views"] * c["nu"] * c["nv"], c["nu"] + 2 * c["ext"]
        # a real convolution by FFT: two transforms of 2.5 L log2 L, L about 2 n
        return {"bytes": 8 * px, "flops": px / c["nu"] * (10 * n * math.log2(2 * n) + 6 * n)}
    both = kind in ("autograd", "ragged")
    b, f = _flops_bytes(c, c["iters"] if kind == "job" else 1,
                        fwd=kind in ("forward", "ragged", "step", "autograd", "job"),
                        motion=both or kind in ("step", "job") or (kind == "vjp" and c["want"] != "data"),
                        data=both or (kind == "vjp" and c["want"] != "motion"),
                        loss=kind in ("step", "job"))
    return {"bytes": b, "flops": f}


# -------------------------------------------------------- the same in 64 bits

class _View:
    """Detector positions of all voxels in one view, float64."""

    def __init__(self, c, Phat):
        ax = [_origin(c)[a] + c["spacing"] * torch.arange(c[k], device=DEV, dtype=torch.float64)
              for a, k in enumerate(("nx", "ny", "nz"))]
        self.ax = ax

        def row(p):
            return (p[0] * ax[0])[None, None, :] + (p[1] * ax[1])[None, :, None] + \
                (p[2] * ax[2] + p[3])[:, None, None]

        w = row(Phat[2])
        self.ok = w > 0
        self.r = torch.where(self.ok, 1.0 / w, 0.0)
        del w
        self.x, self.y = row(Phat[0]) * self.r, row(Phat[1]) * self.r
        nu, nv = c["nu"], c["nv"]
        x = self.x.clamp(-1.5, nu + 0.5)
        y = self.y.clamp(-1.5, nv + 0.5)
        fx, fy = torch.floor(x), torch.floor(y)
        self.tu, self.tv = x - fx, y - fy
        self.W = nu + 4  # images are padded by two pixels of zeros
        self.i = ((fy + 2) * self.W + (fx + 2)).to(torch.int64)

    def bilinear(self, pad, du=False, dv=False):
        f, t, W = pad.reshape(-1), [], self.W
        t = [f[self.i + o] for o in (0, 1, W, W + 1)]
        if du:
            return (t[1] - t[0]) * (1 - self.tv) + (t[3] - t[2]) * self.tv
        if dv:
            return (t[2] - t[0]) * (1 - self.tu) + (t[3] - t[1]) * self.tu
        top = t[0] + self.tu * (t[1] - t[0])
        return top + self.tv * (t[2] + self.tu * (t[3] - t[2]) - top)


def _pad(img):
    return torch.nn.functional.pad(img, (2, 2, 2, 2))


def _gradient(img, dim):
    if img.shape[dim] < 2:
        return torch.zeros_like(img)
    return torch.gradient(img, dim=dim)[0]


def _exact_scan(c, s, theta, want_vol, delta, want):
    """Volume and gradients by Eqs. 1-5 in float64: {vol, dmotion, dproj}."""
    T, D = _rigid(theta)
    Phat = s["P"] @ T
    V = c["views"]
    vol = torch.zeros((c["nz"], c["ny"], c["nx"]), dtype=torch.float64, device=DEV)
    gP = torch.zeros(V, 3, 4, dtype=torch.float64, device=DEV)
    out = {}
    if "data" in want:
        out["dproj"] = torch.zeros(V, c["nv"], c["nu"], dtype=torch.float64, device=DEV)
    for j in range(V):
        q = _View(c, Phat[j].tolist())
        img = s["proj"][j].detach().double()
        if s["view_scale"] is not None:
            img = img * s["view_scale"][j].double()
        om = float(s["vw"][j]) * ((c["sid"] * q.r) ** 2 if c["weight"] == "fdk"
                                  else q.ok.double())
        pad = _pad(img)
        if want_vol:
            vol += om * q.bilinear(pad)
        if "motion" in want:
            if c["deriv"] == "exact":
                gu, gv = q.bilinear(pad, du=True), q.bilinear(pad, dv=True)
            else:
                gu, gv = (q.bilinear(_pad(_gradient(img, d))) for d in (1, 0))
            sr = delta * om * q.r
            a = [sr * gu, sr * gv]
            a.append(-(a[0] * q.x + a[1] * q.y))
            if c["weight"] == "fdk":
                a[2] -= 2 * sr * q.bilinear(pad)
            for r in range(3):
                gP[j, r, 0] = a[r].sum((0, 1)) @ q.ax[0]
                gP[j, r, 1] = a[r].sum((0, 2)) @ q.ax[1]
                gP[j, r, 2] = a[r].sum((1, 2)) @ q.ax[2]
                gP[j, r, 3] = a[r].sum()
        if "data" in want:
            g = torch.zeros(pad.numel(), dtype=torch.float64, device=DEV)
            sd = delta * om
            for o, w in ((0, (1 - q.tu) * (1 - q.tv)), (1, q.tu * (1 - q.tv)),
                         (q.W, (1 - q.tu) * q.tv), (q.W + 1, q.tu * q.tv)):
                g.index_add_(0, (q.i + o).reshape(-1), (sd * w).reshape(-1))
            out["dproj"][j] = g.reshape(pad.shape)[2:-2, 2:-2]
    if want_vol:
        out["vol"] = vol
    if "motion" in want:
        out["dmotion"] = torch.einsum("vij,vik,vmkj->vm", gP, s["P"], D)
    return out


def _exact_loss(vol, kind):
    v = vol.clone().requires_grad_(True)
    d = [v[:, :, 1:] - v[:, :, :-1], v[:, 1:] - v[:, :-1], v[1:] - v[:-1]]
    if kind == "tv":
        g = [d[0][:-1, :-1], d[1][:-1, :, :-1], d[2][:, :-1, :-1]]
        loss = torch.sqrt(sum(x * x for x in g) + 1e-6).sum() / v.numel()
    else:
        loss = -sum((x * x).sum() for x in d) / v.numel()
    return loss.detach(), torch.autograd.grad(loss, v)[0]


def _akima(nodes, V):
    """Akima spline through nodes (n,6) at even knots, values at 0..V-1."""
    n = nodes.shape[0]
    h = (V - 1) / (n - 1)
    m = (nodes[1:] - nodes[:-1]) / h
    a = 2 * m[:1] - (m[1:2] if n > 2 else m[:1])
    z = 2 * m[-1:] - (m[-2:-1] if n > 2 else m[-1:])
    m = torch.cat([2 * a - m[:1], a, m, z, 2 * z - m[-1:]])
    w1, w2 = (m[3:] - m[2:-1]).abs(), (m[1:-2] - m[:-3]).abs()
    den = w1 + w2
    t = torch.where(den > 0, (w1 * m[1:-2] + w2 * m[2:-1]) / torch.where(den > 0, den, 1.0),
                    0.5 * (m[1:-2] + m[2:-1]))
    j = torch.arange(V, device=nodes.device, dtype=torch.float64)
    i = torch.div(torch.arange(V, device=nodes.device) * (n - 1), V - 1,
                  rounding_mode="floor").clamp(max=n - 2)
    e = (j - i * h)[:, None]
    s = m[i + 2]
    return nodes[i] + e * t[i] + e * e * ((3 * s - 2 * t[i] - t[i + 1]) / h) + \
        e ** 3 * ((t[i] + t[i + 1] - 2 * s) / h ** 2)


def exact(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind in ("job", "batch"):  # many dependent iterations: not in 20 seconds
        return None
    s = _inputs(c, seed)
    if kind == "filter":
        return _filtered(c, s["raw"], torch.float64)
    size = c["nx"] * c["ny"] * c["nz"] * c["views"]
    if size > (3e10 if kind == "forward" else 1.5e10):
        return None
    if kind == "forward":
        return _exact_scan(c, s, s["theta"], True, None, ())["vol"]
    if kind in ("vjp", "ragged"):
        want = {"both": ("motion", "data"), "motion": ("motion",), "data": ("data",)}[c["want"]]
        r = _exact_scan(c, s, s["theta"], kind == "ragged", s["delta"].double(), want)
        return {k: r[k] for k in (("vol",) if kind == "ragged" else ()) + ("dmotion", "dproj")
                if k in r}
    if kind == "step":
        vol = _exact_scan(c, s, s["theta"], True, None, ())["vol"]
        loss, dvol = _exact_loss(vol, c["loss"])
        g = _exact_scan(c, s, s["theta"], False, dvol, ("motion",))["dmotion"]
        th = s["theta"] - 0.01 * g / (g.abs() + 1e-8)  # the first Adam step
        return {"vol": vol, "loss": loss, "dvol": dvol, "dmotion": g,
                "theta": th - th.mean(0, keepdim=True)}
    delta = s["delta"].double()
    if c["nodes"]:
        nodes = s["nodes"].clone().requires_grad_(True)
        theta = _akima(nodes, c["views"])
        r = _exact_scan(c, s, theta.detach(), True, delta, ("motion", "data"))
        leaf = torch.autograd.grad(theta, nodes, r["dmotion"])[0]
    else:
        r = _exact_scan(c, s, s["theta"], True, delta, ("motion", "data"))
        leaf = r["dmotion"]
    return {"vol": r["vol"], "dproj": r["dproj"], "dleaf": leaf}
