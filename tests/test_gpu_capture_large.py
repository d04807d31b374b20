"""A large call that is captured after a small one with as many views: it needs no
workspace that the small one did not make (a forward at the start of a graph, say, in a
program that has run a preview)."""
import ctypes

import pytest
import torch

from cases import random_case
from paper_2401_09283_gb300 import bp
from paper_2401_09283_gb300 import native as N

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda", 0)


def test_large_forward_is_captured_after_a_small_one(monkeypatch):
    views, nu, nv, big = 4096, 16, 12, (40, 41, 42)  # 2.8e8 voxel-views
    cfg, P, _, proj, _, _ = random_case(2, big, views, nu, nv, 6.0, 1.0)
    p, Pd = torch.as_tensor(proj, device=DEV), torch.as_tensor(P, device=DEV)

    def forward(shape):
        o = tuple(-(n - 1) / 2.0 for n in shape[::-1])
        return bp.bp_forward(p, Pd, None, vol_shape=shape, spacing=(1.0,) * 3, origin=o, sid=cfg.sid)

    assert views * 40 * 41 * 42 >= 1 << 28
    ref = forward(big)
    fresh = ctypes.c_void_p()  # a context that has run nothing
    assert N.lib().bp_ctx_create(0, ctypes.byref(fresh)) == 0
    monkeypatch.setitem(N._ctx, 0, fresh)
    forward((8, 8, 8))
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        vol = forward(big)
    g.replay()
    assert torch.equal(vol, ref)
    assert float(vol.abs().max()) > 0.0
    torch.cuda.synchronize()
    del g
    monkeypatch.undo()
    N.lib().bp_ctx_destroy(fresh)
