"""Tiles that come near the source plane in front of them: views whose source lies
just beyond a corner, an edge or a face of a tile, at distances down to a millionth
of a voxel, and a matrix with a NaN in one row.  Such tiles are neither staged nor
INTERIOR (tests/test_plan_host.py); their values still match the oracle."""
import numpy as np
import pytest
import torch

import oracle
from cases import rel_l2
from paper_2401_09283_gb300 import bp

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda", 0)
SHAPE = (32, 32, 32)


def matrices(f, nu, nv):
    """Views along z whose source plane lies d in front of the volume's first slice."""
    K = np.array([[f, 0, (nu - 1) / 2], [0, f, (nv - 1) / 2], [0, 0, 1.0]])
    return np.stack([K @ np.array([[1, 0, 0, -x], [0, 1, 0, -y], [0, 0, 1.0, d]])
                     for d in (1e-6, 1e-3, 0.1, 1.0) for x, y in ((0, 0), (15.5, 0), (31, 31), (-3, 7))])


# The specification's bounds (volume and data gradient 1e-5, motion gradient 1e-3) plus
# the FP32 resolution of a position beside the source: a tile spans 16 f pixels, four
# roundings of 2^-24 of that, times the image's slope (0.2 of its values per pixel).  A
# voxel a millionth in front of the source plane projects millions of pixels off the
# detector, or, on the principal ray, onto its centre: there 1/w is 1e6, so plain
# weights and a comparison that leaves out the first slices.
@pytest.mark.parametrize("dtype", [torch.float32, torch.float16])
@pytest.mark.parametrize("f", [3.0, 40.0, 2000.0])
@pytest.mark.parametrize("deriv", ["central", "exact"])
def test_tiles_near_the_source_plane(dtype, f, deriv):
    nu, nv = 64, 48
    P = matrices(f, nu, nv)
    V = len(P)
    # a smooth image: the exact derivative jumps on noise
    u, v = np.meshgrid(np.arange(nu), np.arange(nv))
    proj = np.stack([np.sin(0.07 * u + j) * np.cos(0.05 * v) for j in range(V)]).astype(np.float32)
    stored = torch.as_tensor(proj).to(dtype)
    used = stored.double().numpy()
    delta = np.random.default_rng(3).standard_normal(SHAPE).astype(np.float32)
    delta[:2] = 0.0
    geo = dict(spacing=(1.0,) * 3, origin=(0.0,) * 3, weight="none", sid=100.0)
    args = [stored.to(DEV), torch.as_tensor(P, device=DEV), None]
    vol = bp.bp_forward(*args, vol_shape=SHAPE, **geo)
    _, gP, gd = bp.bp_vjp(torch.as_tensor(delta, device=DEV), *args, deriv=deriv, want_motion=False,
                          want_Phat=True, want_proj=True, **geo)
    vw = np.ones(V)
    o = ((1.0,) * 3, (0.0,) * 3, vw, oracle.WEIGHT_NONE)
    ref = oracle.bp_forward(P, used, SHAPE, *o, 100.0)
    oP, oD = oracle.bp_vjp(P, used, delta.astype(np.float64), *o, oracle.DERIV_CENTRAL
                           if deriv == "central" else oracle.DERIV_BILINEAR_EXACT, 100.0)
    res = 0.2 * 16 * f * 4 * 2.0 ** -24
    assert rel_l2(vol[2:].cpu().numpy(), ref[2:]) <= 1e-5 + res
    assert np.isfinite(vol.cpu().numpy()).all()
    assert rel_l2(gd.cpu().numpy(), oD) <= 1e-5 + res
    assert rel_l2(gP.cpu().numpy(), oP) <= 1e-3 + res


def test_nan_in_a_matrix_row_leaves_the_other_views_alone():
    nu, nv = 64, 48
    P = matrices(40.0, nu, nv)[12:]
    P = np.concatenate([P, P])
    P[1, 0, 3] = np.nan
    P[3, 1, 0] = np.inf
    P[5, 2, 2] = np.nan
    proj = np.random.default_rng(1).standard_normal((len(P), nv, nu)).astype(np.float32)
    delta = torch.ones(SHAPE, device=DEV)
    geo = dict(spacing=(1.0,) * 3, origin=(0.0,) * 3, weight="none", sid=100.0)
    p, Pd = torch.as_tensor(proj, device=DEV), torch.as_tensor(P, device=DEV)
    _, gP, gd = bp.bp_vjp(delta, p, Pd, None, want_motion=False, want_Phat=True, want_proj=True, **geo)
    bp.bp_forward(p, Pd, None, vol_shape=SHAPE, **geo)
    good = [0, 2, 4, 6, 7]
    _, g2, d2 = bp.bp_vjp(delta, p[good].contiguous(), Pd[good].contiguous(), None, want_motion=False,
                          want_Phat=True, want_proj=True, **geo)
    assert torch.equal(gP[good], g2)
    assert rel_l2(gd[good].cpu().numpy(), d2.cpu().numpy()) <= 1e-6
