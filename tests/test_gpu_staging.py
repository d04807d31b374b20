"""The staged kernels at the sizes where their copies, slots, records and view
chunks can go wrong, against the oracle: detector sizes around the TMA box, view
counts around the slots and the 32-view batches, volumes around the tile, every
storage type; tiles that cross the detector's edges; and the kernel variant for
footprints wider than the staging buffer against the path of unaligned rows."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from cases import motion_errors, random_case, rel_l2
from paper_2401_09283_gb300 import bp
from paper_2401_09283_gb300 import native as N

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - GPU machine only
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

DEV = torch.device("cuda:0")


def cuda(x):
    return torch.as_tensor(np.ascontiguousarray(x)).to(DEV)


# The volume bound of the specification (1e-5), the motion gradient's (1e-3 per
# parameter group) and the data gradient's (1e-5); half storage is compared with
# the oracle on the dequantised data, so the same bounds hold.
@pytest.mark.parametrize("dtype", [torch.float32, torch.float16, torch.bfloat16])
@pytest.mark.parametrize("shape,views,nu,nv,pitch,spacing", [
    ((1, 1, 1), 1, 8, 1, 9.0, 2.0),        # one voxel, one row
    ((16, 16, 16), 2, 88, 7, 1.0, 1.0),    # fewer rows than a box, wider than a buffer
    ((17, 15, 33), 3, 80, 8, 1.1, 1.0),    # tile remainders, exactly one box of rows
    ((5, 40, 18), 31, 96, 65, 0.9, 1.0),   # more rows than a buffer; one batch less one view
    ((33, 17, 16), 32, 64, 64, 1.0, 1.2),
    ((18, 33, 20), 33, 72, 40, 1.3, 1.5),  # a batch and one view
    ((40, 24, 30), 66, 48, 33, 1.2, 1.0),  # volume beyond the detector on every side
])
def test_staging_edges(dtype, shape, views, nu, nv, pitch, spacing):
    cfg, P, th, proj, delta, origin = random_case(100 + views + nu, shape, max(views, 2), nu, nv,
                                                  pitch, spacing)
    P, th, proj = P[:views], th[:views], proj[:views]  # (the generator needs two views)
    stored = torch.as_tensor(proj).to(dtype)
    used = stored.double().numpy()
    args = dict(spacing=(spacing,) * 3, origin=origin, weight="fdk", sid=cfg.sid)
    vw = np.full(views, 0.01)
    d = [cuda(x) for x in (P, th, vw)]
    vol = bp.bp_forward(stored.to(DEV), d[0], d[1], vol_shape=shape, view_weight=d[2], **args)
    gm, _, gd = bp.bp_vjp(cuda(delta), stored.to(DEV), d[0], d[1], view_weight=d[2],
                          want_proj=True, **args)
    gm1, _, _ = bp.bp_vjp(cuda(delta), stored.to(DEV), d[0], d[1], view_weight=d[2], **args)
    Ph = oracle.compose(P, th)
    ref = oracle.bp_forward(Ph, used, shape, (spacing,) * 3, origin, vw, oracle.WEIGHT_FDK, cfg.sid)
    oP, oD = oracle.bp_vjp(Ph, used, delta.astype(np.float64), (spacing,) * 3, origin, vw,
                           oracle.WEIGHT_FDK, oracle.DERIV_CENTRAL, cfg.sid)
    om = oracle.chain_motion(P, th, oP)
    assert rel_l2(vol.cpu().numpy(), ref) <= 1e-5
    e = motion_errors(gm.cpu().numpy(), om)
    assert e[0] <= 1e-3
    if om[:, 3:].any():
        assert e[1] <= 1e-3
    else:  # a single voxel at the centre of rotation: exactly 0 in the oracle
        assert np.abs(gm.cpu().numpy()[:, 3:]).max() <= 1e-3 * np.abs(om[:, :3]).max()
    assert torch.equal(gm, gm1)  # the fused kernel's motion part is the motion kernel's
    assert rel_l2(gd.cpu().numpy(), oD) <= 1e-5


def test_wide_footprints_take_the_unstaged_variant_bit_for_bit():
    # 128^3 x 128 views at 5 px per voxel (two launches, chosen per view on the
    # device) against rows with one pixel of padding, which are never staged
    n, views, nu, nv = 128, 128, 256, 192
    cfg, P, th, proj, delta, origin = random_case(7, (n, n, n), views, nu, nv, 0.32, 1.0)
    p = cuda(proj)
    odd = torch.zeros(views, nv, nu + 1, device=DEV)
    odd[..., :nu] = p
    vw, Pd, thd = cuda(np.ones(views)), cuda(P), cuda(th)
    args = dict(spacing=(1.0,) * 3, origin=origin, weight="fdk", sid=cfg.sid)
    vol = bp.bp_forward(p, Pd, thd, vol_shape=(n, n, n), view_weight=vw, **args)
    gm, _, _ = bp.bp_vjp(cuda(delta), p, Pd, thd, view_weight=vw, **args)
    pd = N.proj_desc(p, cfg.sid)
    pd.row_stride, pd.view_stride = nu + 1, nv * (nu + 1)
    vd = N.vol_desc((n, n, n), (1.0,) * 3, origin)
    ctx, s = N.context(0), torch.cuda.current_stream().cuda_stream
    v2, g2 = torch.empty_like(vol), torch.empty_like(gm)
    N.check("bp_forward", N.lib().bp_forward(ctx, N.ptr(odd), ctypes.byref(pd), N.ptr(Pd),
                                             N.ptr(thd), N.ptr(vw), 1, ctypes.byref(vd), N.ptr(v2),
                                             s), ctx)
    dv = cuda(delta)
    N.check("bp_vjp", N.lib().bp_vjp(ctx, N.ptr(dv), N.ptr(odd), ctypes.byref(pd), N.ptr(Pd),
                                     N.ptr(thd), N.ptr(vw), 1, 0, ctypes.byref(vd), N.ptr(g2), None,
                                     None, s), ctx)
    assert torch.equal(vol, v2)
    assert torch.equal(gm, g2)
    assert float(vol.abs().max()) > 0.0 and float(gm.abs().max()) > 0.0
