"""Run by tests/test_gpu_lost_copy.py in a child process whose BP_GB300_LIB points at
the bounds-checking debug build, in which the footprints of one view can be announced
and never copied: the wait for them runs out and the kernels return, with
NaN where the view's footprint was needed and in what follows it.  Prints one JSON
line."""
import ctypes
import json
import os
import sys
import time

import numpy as np
import torch

HERE = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, HERE)
sys.path.insert(0, os.path.dirname(HERE))

from cases import random_case  # noqa: E402
from paper_2401_09283_gb300 import bp  # noqa: E402
from paper_2401_09283_gb300 import native as N  # noqa: E402
from paper_2401_09283_gb300.job import Batch, MotionJob  # noqa: E402

DEV = torch.device("cuda:0")
LOST = 3


def lose(view):
    flags, first = ctypes.c_uint(), ctypes.c_longlong(view)
    ctx = N.context(0)
    N.check("bp_bounds_check", N.lib().bp_bounds_check(ctx, 3, ctypes.byref(flags),
                                                       ctypes.byref(first)), ctx)


def calls(dtype):
    """Volume, motion gradient alone and with the data gradient; a job's and a batch's
    motion.  Everything projects inside the detector, so every tile is staged."""
    out = {}
    for name, shape, views, nu, nv, pitch in (("tile", (40, 40, 40), 180, 96, 80, 1.2),
                                              ("half", (16, 16, 16), 9, 128, 96, 1 / 3)):
        cfg, P, th, proj, delta, origin = random_case(3, shape, views, nu, nv, pitch, 1.0)
        p, Pd, d = (torch.as_tensor(x, device=DEV) for x in (proj, P, delta))
        p = p.to(dtype)
        geo = dict(spacing=(1.0,) * 3, origin=origin, sid=cfg.sid)
        if name == "tile":
            out["vol"] = bp.bp_forward(p, Pd, None, vol_shape=shape, **geo)
            out["motion"] = bp.bp_vjp(d, p, Pd, None, **geo)[0]
            out["both"] = bp.bp_vjp(d, p, Pd, None, want_proj=True, **geo)[0]
            out["exact"] = bp.bp_vjp(d, p, Pd, None, deriv="exact", **geo)[0]

        def job():
            return MotionJob(p, Pd, vol_shape=shape, optimizer="gd", lr=1.0, lr_rot=1e-3,
                             gauge=False, max_iters=1, **geo)
        j = job()
        j.step(1)
        out["job-" + name] = j.motion()[0]
        j.close()
        jobs = [job(), job()]
        b = Batch(max_jobs=2)
        b.set_jobs(jobs)
        b.step(1)
        out["batch-" + name] = np.concatenate([q.motion()[0] for q in jobs], 1)
        b.close()
        for q in jobs:
            q.close()
    return {k: np.asarray(torch.as_tensor(v).cpu()) for k, v in out.items()}


def main():
    res = {"library": N.library_path()}
    for dtype in (torch.float32, torch.bfloat16):
        clean = calls(dtype)
        lose(LOST)
        t = time.time()
        lost = calls(dtype)
        res["seconds"] = min(res.get("seconds", 1e9), time.time() - t)
        lose(-1)
        again = calls(dtype)
        n = str(dtype)
        res[n] = {k: {"finite": bool(np.isfinite(clean[k]).all()),
                      "same after": bool(np.array_equal(clean[k], again[k])),
                      "nan": np.isnan(lost[k]).mean(),
                      "early kept": bool(np.array_equal(lost[k][:LOST - 1], clean[k][:LOST - 1])),
                      "lost nan": bool(np.isnan(lost[k][LOST]).all())} for k in clean}
    print(json.dumps(res))


if __name__ == "__main__":
    main()
