"""Which kernel variant a call takes, on scans whose views are all wide (more than 4 px
per voxel), none, or some: calls on odd rows, which copy them and choose per view on the
device, against the same calls captured, which do neither and read global memory, bit
for bit; both against the oracle; and the number of kernels that they launch."""
import numpy as np
import pytest
import torch

import oracle
from cases import motion_errors, random_case, rel_l2
from paper_2401_09283_gb300 import bp
from paper_2401_09283_gb300 import native as N
from paper_2401_09283_gb300.job import Batch, MotionJob

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda", 0)


def scan(kind, nu, views=64, n=42):
    """Random data; pitch 0.3 is 5 px per voxel (wide), 1.2 is 1.3 px."""
    out = {p: random_case(9, (n, n - 1, n - 2), views, nu, 150, p, 1.0) for p in (0.3, 1.2)}
    cfg, P, th, proj, delta, origin = out[0.3 if kind == "wide" else 1.2]
    if kind == "mixed":  # the first view of every chunk is wide, others are not
        P = P.copy()
        P[::2] = out[0.3][1][::2]
    u, v = np.meshgrid(np.arange(nu), np.arange(150))
    smooth = np.stack([np.sin(0.05 * u + j) * np.cos(0.04 * v) for j in range(views)])
    return cfg, P, th, smooth.astype(np.float32), delta, origin


def captured(f):
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        out = f()
    g.replay()
    torch.cuda.synchronize()
    return out


# The specification's bounds (volume and data gradient 1e-5, motion gradient 1e-3); the
# exact derivative jumps at pixel borders, so smooth data.
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("deriv", ["central", "exact"])
@pytest.mark.parametrize("kind", ["wide", "mixed", "narrow"])
def test_chosen_variants_agree_with_the_global_one(kind, deriv, dtype):
    cfg, P, th, proj, delta, origin = scan(kind, 181)
    stored = torch.as_tensor(proj).to(dtype)
    used, shape, vw = stored.double().numpy(), delta.shape, np.full(len(P), 0.02)
    assert delta.size * len(P) >= 1 << 22 and 181 > 4 * 42
    p, Pd, thd, vwd, dv = (torch.as_tensor(x, device=DEV) for x in (stored, P, th, vw, delta))
    geo = dict(spacing=(1.0,) * 3, origin=origin, view_weight=vwd, sid=cfg.sid)

    def forward():
        return bp.bp_forward(p, Pd, thd, vol_shape=shape, **geo)

    def vjp(data):
        return bp.bp_vjp(dv, p, Pd, thd, deriv=deriv, want_proj=data, **geo)[0::2]
    n0 = N.launch_count(0)
    vol = forward()
    n1 = N.launch_count(0)
    gm = vjp(False)[0]
    gm2, gd = vjp(True)
    n2 = N.launch_count(0)
    volc = captured(forward)
    n3 = N.launch_count(0)
    gmc = captured(lambda: vjp(False))[0]
    assert torch.equal(vol, volc) and torch.equal(gm, gmc) and torch.equal(gm, gm2)
    assert n1 - n0 == 4  # composition, copy, both variants
    assert n3 - n2 == 2  # composition, forward
    Ph = oracle.compose(P, th)
    o = ((1.0,) * 3, origin, vw, oracle.WEIGHT_FDK)
    ref = oracle.bp_forward(Ph, used, shape, *o, cfg.sid)
    oP, oD = oracle.bp_vjp(Ph, used, delta.astype(np.float64), *o, oracle.DERIV_CENTRAL
                           if deriv == "central" else oracle.DERIV_BILINEAR_EXACT, cfg.sid)
    assert rel_l2(vol.cpu().numpy(), ref) <= 1e-5
    e = motion_errors(gm.cpu().numpy(), oracle.chain_motion(P, th, oP))
    assert e[0] <= 1e-3 and e[1] <= 1e-3
    assert rel_l2(gd.cpu().numpy(), oD) <= 1e-5


def step(P, proj, shape, origin, sid, dtype, batch=False):
    """Motion and loss after one step of a job, or of a job in a batch of two."""
    def job():
        return MotionJob(torch.as_tensor(proj).to(dtype).to(DEV), torch.as_tensor(P, device=DEV),
                         vol_shape=shape, spacing=(1.0,) * 3, origin=origin, sid=sid,
                         optimizer="gd", lr=1e3, lr_rot=1.0, gauge=False, max_iters=1)
    jobs = [job(), job()] if batch else [job()]
    if batch:
        b = Batch(max_jobs=2)
        b.set_jobs(jobs)
        b.step(1)
    else:
        jobs[0].step(1)
    got = [j.motion()[:2] for j in jobs]
    if batch:
        b.close()
    for j in jobs:
        j.close()
    return got[-1]


# Inside the detector, so that a column of zeros beside it changes nothing but the rows'
# alignment: such a job is not staged.
@pytest.mark.parametrize("dtype", [torch.float32, torch.float16])
@pytest.mark.parametrize("shape,views", [((16, 16, 16), 2), ((13, 20, 18), 9), ((24, 17, 16), 17)])
def test_half_tiles_keep_the_bits_of_the_global_kernels(shape, views, dtype):
    nu, nv = 176, 176
    cfg, P, _, proj, _, origin = random_case(views, shape, views, nu, nv, 1 / 3, 1.0)
    wide = np.concatenate([proj, np.zeros((views, nv, 1), np.float32)], 2)
    th, hist = step(P, proj, shape, origin, cfg.sid, dtype)
    th1, hist1 = step(P, wide, shape, origin, cfg.sid, dtype)
    assert np.array_equal(th, th1) and np.array_equal(hist, hist1)
    assert np.abs(th).max() > 0.0
    thb, histb = step(P, proj, shape, origin, cfg.sid, dtype, batch=True)
    assert np.array_equal(th, thb) and np.array_equal(hist, histb)
