"""Calls with little free device memory: what a call needs comes before what it can do
without (the aligned copy of odd rows, their block image), and what earlier calls keep
makes room."""
import contextlib
import ctypes

import pytest
import torch

from cases import random_case, rel_l2
from paper_2401_09283_gb300 import bp
from paper_2401_09283_gb300 import native as N

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda", 0)
MIB = 1 << 20
VIEWS, NV, NU, N3 = 100, 400, 1003, 76  # 40.1M pixels, 43.9M voxel-views


@pytest.fixture
def fresh(monkeypatch):
    """A context without workspaces, in place of the shared one."""
    ctx = ctypes.c_void_p()
    assert N.lib().bp_ctx_create(0, ctypes.byref(ctx)) == 0
    monkeypatch.setitem(N._ctx, 0, ctx)
    yield ctx
    torch.cuda.synchronize()
    monkeypatch.undo()
    N.lib().bp_ctx_destroy(ctx)


@contextlib.contextmanager
def left(mib):
    """Device memory taken (never touched) until `mib` MiB are free."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info(0)[0] - mib * MIB, dtype=torch.uint8, device=DEV)
    try:
        yield
        torch.cuda.synchronize()
    finally:
        del hog
        torch.cuda.empty_cache()


def case(pad):
    """A random scan in half precision; `pad` more columns than it uses per row."""
    cfg, P, _, _, _, origin = random_case(1, (N3,) * 3, VIEWS, 16, 12, 0.3, 1.0)
    p = torch.randn(VIEWS, NV, NU + pad, device=DEV).half()
    dv = torch.randn(N3, N3, N3, device=DEV)
    return cfg, torch.as_tensor(P, device=DEV), p, dv, origin


def vjp(cfg, P, p, dv, origin, gm, gd):
    pd = N.ProjDesc(NU, NV, VIEWS, N.F16, p.shape[2], p.shape[1] * p.shape[2], None, cfg.sid)
    vd = N.vol_desc((N3,) * 3, (1.0,) * 3, origin)
    ctx = N.context(0)
    N.check("bp_vjp", N.lib().bp_vjp(
        ctx, N.ptr(dv), N.ptr(p), ctypes.byref(pd), N.ptr(P), None, None, 1, 0, ctypes.byref(vd),
        N.ptr(gm), None, N.ptr(gd) if gd is not None else None,
        torch.cuda.current_stream().cuda_stream), ctx)


# Needed: the gradient images, 306 MiB, and 8 MiB or so of records.  The copy is 77 MiB,
# the block image 612 MiB.  (5 pad columns make the rows whole 16-byte chunks.)
@pytest.mark.parametrize("pad,data", [(0, False), (0, True), (5, True)])
def test_vjp_takes_what_it_needs_first(fresh, pad, data):
    args = case(pad)
    gm = torch.empty(VIEWS, 6, dtype=torch.float64, device=DEV)
    gd = torch.empty(VIEWS, NV, NU, device=DEV) if data else None
    vjp(*args, gm, gd)
    torch.cuda.synchronize()
    ref, refd = gm.clone(), gd.clone() if data else None
    # the same call in another fresh context, with 360 MiB left: copy and block image fit
    # beside the images or before them, not both
    small = ctypes.c_void_p()
    assert N.lib().bp_ctx_create(0, ctypes.byref(small)) == 0
    shared, N._ctx[0] = N._ctx[0], small
    try:
        with left(360):
            vjp(*args, gm, gd)
        kept = N.lib().bp_ctx_workspace_bytes(small)
    finally:
        N._ctx[0] = shared
        N.lib().bp_ctx_destroy(small)
    assert kept < 360 * MIB
    assert rel_l2(gm.cpu().numpy(), ref.cpu().numpy()) <= 1e-5  # (the order of FP32 sums)
    if data:
        assert rel_l2(gd.cpu().numpy(), refd.cpu().numpy()) <= 1e-5


def test_workspaces_that_calls_can_do_without_make_room(fresh):
    cfg, P, p, dv, origin = case(0)
    geo = dict(spacing=(1.0,) * 3, origin=origin, sid=cfg.sid)
    vol = bp.bp_forward(p, P, None, vol_shape=(N3,) * 3, **geo)
    torch.cuda.synchronize()
    held = N.lib().bp_ctx_workspace_bytes(fresh)
    assert held >= p.numel() * 2  # the aligned copy is kept
    gm = torch.empty(VIEWS, 6, dtype=torch.float64, device=DEV)
    with left(280):  # less than the images, more with the copy's 77 MiB
        vjp(cfg, P, p, dv, origin, gm, None)
    assert bool(torch.isfinite(gm).all()) and float(gm.abs().max()) > 0.0
    assert torch.equal(vol, bp.bp_forward(p, P, None, vol_shape=(N3,) * 3, **geo))
