"""Jobs on scans of 4 to 5 pixels per voxel, whose footprints are staged by half
tiles: one Eq. 6 step and its loss against the oracle, for every storage type, at
view counts around the batches of eight views, ragged volumes, and volumes that
reach beyond the detector (half tiles that are off it, cross its edge, or do not
fit the buffer)."""
import numpy as np
import pytest
import torch

import oracle
from cases import motion_errors, random_case
from paper_2401_09283_gb300.job import MotionJob

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda", 0)


# Bounds: the motion gradient's of the specification (1e-3 per parameter group); the
# loss is a sum of squares of volume differences (1e-5 each in L2), so 2e-5 and its
# rounding.
@pytest.mark.parametrize("dtype", [torch.float32, torch.float16, torch.bfloat16])
@pytest.mark.parametrize("shape,views,nu,nv,pitch", [
    ((16, 16, 16), 2, 128, 96, 1 / 3),    # one tile, inside the detector
    ((33, 20, 18), 9, 160, 192, 0.34),    # tile remainders, a batch and one view
    ((24, 17, 40), 17, 96, 64, 0.33),     # far beyond the detector on every side
    ((9, 48, 31), 8, 320, 88, 0.36),      # one half tile and one slice
])
def test_job_step_of_half_tiles_matches_oracle(dtype, shape, views, nu, nv, pitch):
    cfg, P, _, proj, _, origin = random_case(views + nu, shape, views, nu, nv, pitch, 1.0)
    stored = torch.as_tensor(proj).to(dtype)
    used, vw, th = stored.double().numpy(), np.full(views, 0.02), np.zeros((views, 6))
    Ph = oracle.compose(P, th)
    vol = oracle.bp_forward(Ph, used, shape, (1.0,) * 3, origin, vw, oracle.WEIGHT_FDK, cfg.sid)
    loss, dvol = oracle.sharpness(vol)
    gP, _ = oracle.bp_vjp(Ph, used, dvol, (1.0,) * 3, origin, vw, oracle.WEIGHT_FDK,
                          oracle.DERIV_CENTRAL, cfg.sid, want_proj=False)
    g = oracle.chain_motion(P, th, gP)
    s0 = 0.1 / np.abs(g).max()
    job = MotionJob(stored.to(DEV), torch.as_tensor(P, device=DEV), vol_shape=shape,
                    spacing=(1.0,) * 3, origin=origin, sid=cfg.sid,
                    view_weight=torch.as_tensor(vw, device=DEV), optimizer="gd", lr=s0, lr_rot=s0,
                    gauge=False, max_iters=1)
    job.step(1)
    got, hist, _ = job.motion()
    job.close()
    e = motion_errors(got, -s0 * g)
    assert e[0] <= 1e-3 and e[1] <= 1e-3
    assert abs(hist[0] - loss) <= 2e-5 * abs(loss) + 1e-12
