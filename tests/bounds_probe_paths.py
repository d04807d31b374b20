"""Run by tests/test_gpu_bounds_paths.py in a child process whose BP_GB300_LIB points at
the bounds-checking debug build: the paths that need larger problems, jobs or batches --
footprints staged by half tiles, the batch's persistent forward, rows copied to an
aligned pitch, the 16-slice forward of more than 304 tiles.
Prints the errors against the oracle and the device flag word as one JSON line."""
import ctypes
import json
import os
import sys

import numpy as np
import torch

HERE = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, HERE)
sys.path.insert(0, os.path.dirname(HERE))

import oracle  # noqa: E402
from cases import random_case, rel_l2  # noqa: E402
from paper_2401_09283_gb300 import bp  # noqa: E402
from paper_2401_09283_gb300 import native as N  # noqa: E402
from paper_2401_09283_gb300.job import Batch, MotionJob  # noqa: E402

DEV = torch.device("cuda:0")


def scan(seed, shape, views, nu, nv, pitch, dtype):
    cfg, P, _, proj, delta, origin = random_case(seed, shape, views, nu, nv, pitch, 1.0)
    stored = torch.as_tensor(proj).to(dtype)
    return cfg, P, stored, stored.double().numpy(), delta, origin


def calls(name, shape, views, nu, nv, pitch, dtype, deriv):
    cfg, P, stored, used, delta, origin = scan(4, shape, views, nu, nv, pitch, dtype)
    geo = dict(spacing=(1.0,) * 3, origin=origin, sid=cfg.sid)
    args = [stored.to(DEV), torch.as_tensor(P, device=DEV), None]
    vol = bp.bp_forward(*args, vol_shape=shape, **geo)
    d = torch.as_tensor(delta, device=DEV)
    gP = bp.bp_vjp(d, *args, deriv=deriv, want_motion=False, want_Phat=True, **geo)[1]
    _, gP2, gD = bp.bp_vjp(d, *args, deriv=deriv, want_motion=False, want_Phat=True, want_proj=True,
                           **geo)
    o = ((1.0,) * 3, origin, None, oracle.WEIGHT_FDK)
    ref = oracle.bp_forward(P, used, shape, *o, cfg.sid)
    oP, oD = oracle.bp_vjp(P, used, delta.astype(np.float64), *o, oracle.DERIV_CENTRAL
                           if deriv == "central" else oracle.DERIV_BILINEAR_EXACT, cfg.sid)
    return [name, max(rel_l2(vol.cpu().numpy(), ref), rel_l2(gD.cpu().numpy(), oD)),
            rel_l2(gP.cpu().numpy(), oP) if deriv == "central" else 0.0, bool(torch.equal(gP, gP2))]


def jobs(name, shapes, views, nu, nv, pitch, dtype, batch):
    """One gradient step of each job against the oracle's."""
    made, want = [], []
    for k, shape in enumerate(shapes):
        cfg, P, stored, used, _, origin = scan(20 + k, shape, views, nu, nv, pitch, dtype)
        vol = oracle.bp_forward(P, used, shape, (1.0,) * 3, origin, None, oracle.WEIGHT_FDK, cfg.sid)
        _, dvol = oracle.sharpness(vol)
        gP, _ = oracle.bp_vjp(P, used, dvol, (1.0,) * 3, origin, None, oracle.WEIGHT_FDK,
                              oracle.DERIV_CENTRAL, cfg.sid, want_proj=False)
        g = oracle.chain_motion(P, np.zeros((views, 6)), gP)
        s = 0.1 / np.abs(g).max()
        want.append(-s * g)
        made.append(MotionJob(stored.to(DEV), torch.as_tensor(P, device=DEV), vol_shape=shape,
                              spacing=(1.0,) * 3, origin=origin, sid=cfg.sid, optimizer="gd", lr=s,
                              lr_rot=s, gauge=False, max_iters=1))
    if batch:
        b = Batch(max_jobs=len(made))
        b.set_jobs(made)
        b.step(1)
    else:
        for j in made:
            j.step(1)
    e = [max(rel_l2(j.motion()[0][:, q], w[:, q]) for q in (slice(0, 3), slice(3, 6)))
         for j, w in zip(made, want)]
    if batch:
        b.close()
    for j in made:
        j.close()
    return [name, 0.0, max(e), True]


def main():
    cases = []
    for dt in (torch.float32, torch.float16):
        n = str(dt)[6:]
        cases.append(jobs("half-" + n, [(33, 20, 18), (24, 17, 40)], 9, 160, 96, 0.34, dt, False))
        cases.append(jobs("half-batch-" + n, [(33, 20, 18), (9, 48, 31)], 9, 160, 96, 0.34, dt, True))
        cases.append(jobs("batch-" + n, [(19, 21, 37), (40, 33, 17)], 35, 48, 40, 1.3, dt, True))
        cases.append(calls("odd-" + n, (40, 41, 42), 64, 61, 47, 1.2, dt, "central"))
        cases.append(calls("odd-edge-" + n, (40, 81, 42), 40, 45, 31, 1.2, dt, "central"))
    cases.append(calls("odd-exact", (40, 41, 42), 64, 61, 47, 1.2, torch.float32, "exact"))
    cases.append(calls("tiles", (112, 112, 100), 5, 136, 130, 1.5, torch.float32, "central"))
    cases.append(calls("tiles-bf16", (100, 112, 112), 5, 136, 90, 1.5, torch.bfloat16, "central"))
    torch.cuda.synchronize()
    flags, first = ctypes.c_uint(), ctypes.c_longlong()
    ctx = N.context(0)
    N.check("bp_bounds_check", N.lib().bp_bounds_check(ctx, 0, ctypes.byref(flags),
                                                       ctypes.byref(first)), ctx)
    print(json.dumps({"library": N.library_path(), "cases": cases, "flags": int(flags.value),
                      "first": int(first.value)}))


if __name__ == "__main__":
    main()
