"""The classification of a box of voxels and the plan of its staged footprint
(csrc/bp_plan.h, the function that the kernels run), compiled for the host: ranges
that come near the source plane, overflow an int, or are not finite are neither
staged nor INTERIOR, bounded ones are as a plain integer reference says, and every
sample of a staged or INTERIOR box reads inside its rectangle."""
import ctypes
import math
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2401_09283_gb300", "csrc")
SKIP, INTERIOR, EDGE = 0, 1, 2

SOURCE = r"""
#include "bp_plan.h"
using namespace bpk;
extern "C" void plan(const float* r, int front, int nu, int nv, int au, int av, int CH, int cols, int rows,
                     int halo, int seq, int* out) {
  const BoxRange q = {r[0], r[1], r[2], r[3], r[4], r[5], front};
  const BoxPlan p = plan_box(q, nu, nv, au, av, CH, cols, rows, halo, seq != 0);
  const int o[7] = {p.mode, p.csafe, p.staged, p.sx0, p.sv0, p.sh, p.scpr};
  for (int k = 0; k < 7; ++k) out[k] = o[k];
}
// Corners and samples of a 16^3 tile in the kernels' FP32 order; g: U0, ru[3], V0, rv[3],
// W0, rw[3].  Returns the samples of a staged or INTERIOR box that read outside.
extern "C" int outside(const float* g, int nu, int nv, int au, int av, int CH, int cols, int rows,
                       int halo, int* out) {
  auto at = [&](const float* a, float x, float y, float z) {
    return fmaf(a[3], z, fmaf(a[2], y, fmaf(a[1], x, a[0])));
  };
  float r[6] = {INFINITY, -INFINITY, INFINITY, -INFINITY, INFINITY, 0.0f};
  int front = 0;
  for (int c = 0; c < 8; ++c) {
    const float x = c & 1 ? 7.5f : -7.5f, y = c & 2 ? 7.5f : -7.5f, z = c & 4 ? 7.5f : -7.5f;
    const float w = at(g + 8, x, y, z);
    r[4] = fminf(r[4], w);
    if (!in_front(w)) continue;
    ++front;
    const float a = at(g, x, y, z) / w, b = at(g + 4, x, y, z) / w;
    r[0] = fminf(r[0], a);
    r[1] = fmaxf(r[1], a);
    r[2] = fminf(r[2], b);
    r[3] = fmaxf(r[3], b);
  }
  r[5] = 2.0f * g[8] - r[4];
  plan(r, front, nu, nv, au, av, CH, cols, rows, halo, 0, out);
  const bool staged = out[2], interior = out[0] == MODE_INTERIOR;
  if (out[0] == MODE_SKIP || !(staged || interior)) return 0;
  int bad = 0;
  for (int e = 0; e < 4096; ++e) {
    const float x = (e & 15) - 7.5f, y = (e >> 4 & 15) - 7.5f, z = (e >> 8) - 7.5f;
    const float q = 1.0f / at(g + 8, x, y, z);
    for (int s = -1; s <= 1; ++s) {  // the approximate reciprocal is one ulp off at most
      const float i = s ? nextafterf(q, s * INFINITY) : q;
      const float fx = floorf(at(g, x, y, z) * i), fy = floorf(at(g + 4, x, y, z) * i);
      if (interior && !(fx >= -au && fx <= nu - 2 - au && fy >= -av && fy <= nv - 2 - av)) ++bad;
      const float sx = (float)(out[3] - au + halo), sy = (float)(out[4] - av + halo);
      if (staged && !(fx >= sx && fx + 1 + halo <= out[3] - au + out[6] * CH - 1 && fy >= sy &&
                      fy + 1 + halo <= out[4] - av + out[5] - 1))
        ++bad;
    }
  }
  return bad;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cc = shutil.which("g++")
    if not cc:
        pytest.skip("needs g++")
    d = tmp_path_factory.mktemp("plan")
    src, so = d / "plan.cpp", d / "plan.so"
    src.write_text(SOURCE)
    subprocess.run([cc, "-std=c++17", "-O2", "-fwrapv", "-ffp-contract=off", "-fPIC", "-shared", "-I", CSRC, str(src), "-o",
                    str(so)], check=True)
    return ctypes.CDLL(str(so))


def plan(lib, r, nu, nv, au, av, CH=4, cols=84, rows=64, halo=1, seq=0, front=8):
    out = (ctypes.c_int * 7)()
    lib.plan((ctypes.c_float * 6)(*r), front, nu, nv, au, av, CH, cols, rows, halo, seq, out)
    return list(out)


INF, NAN = math.inf, math.nan


# corners at w > 0 of which one is tiny, or an entry of the matrix is not finite
@pytest.mark.parametrize("r", [
    (-300.0, 5e9, -30.0, 20.0, 1e-7, 9.0),      # beyond an int: wrapped to a small footprint
    (-5e9, 300.0, -30.0, 20.0, 1e-7, 9.0),
    (-30.0, 20.0, -300.0, 5e9, 1e-7, 9.0),
    (-30.0, 20.0, -5e9, 5e9, 1e-7, 9.0),
    (-5e9, 5e9, -5e9, 5e9, 1e-7, 9.0),
    (-2147483000.0, 2147483000.0, -1.0, 1.0, 1.0, 9.0),
    (-INF, INF, -1.0, 1.0, 1.0, 2.0), (-1.0, INF, -1.0, 1.0, 1.0, 2.0),
    (NAN, NAN, -1.0, 1.0, 1.0, 2.0), (-1.0, 1.0, NAN, NAN, 1.0, 2.0),
    (-1.0, 1.0, -1.0, 1.0, 0.0, 2.0), (-1.0, 1.0, -1.0, 1.0, NAN, 2.0),
    (-30.0, 30.0, -20.0, 20.0, 1e-4, 2.0),      # rounding of w beyond the margin
    (0.0, 0.0, 0.0, 0.0, 1.0, INF),
])
@pytest.mark.parametrize("au,av", [(300, 100), (-1048576, 100), (300, 1048576), (0, 0)])
def test_unbounded_boxes_take_the_checked_path(lib, r, au, av):
    for nu, nv in ((616, 480), (1 << 20, 1 << 10)):
        mode, csafe, staged = plan(lib, r, nu, nv, au, av)[:3]
        assert mode != INTERIOR and not csafe and not staged
        # one corner behind the source plane, and all of them
        assert plan(lib, (-1.0, 1.0, -1.0, 1.0, -0.1, 2.0), nu, nv, 300, 100, front=7)[0:3] == [EDGE, 0, 0]
        assert plan(lib, (INF, -INF, INF, -INF, -2.0, -1.0), nu, nv, 300, 100, front=0)[0:3] == [SKIP, 0, 0]


def test_bounded_boxes_match_an_integer_reference(lib):
    rng = np.random.default_rng(4)
    seen = set()
    for _ in range(20000):
        nu, nv = int(rng.integers(1, 700)), int(rng.integers(1, 500))
        au, av = int(rng.integers(-90, nu + 90)), int(rng.integers(-90, nv + 90))
        c = rng.uniform(0, 1, 2).astype(np.float32)
        e = rng.uniform(0, [60, 50]).astype(np.float32)
        r = [float(np.float32(x)) for x in (c[0] - e[0], c[0] + e[0], c[1] - e[1], c[1] + e[1])]
        CH, cols, rows = [(4, 84, 64), (8, 80, 64), (4, 116, 56), (8, 120, 56), (4, 84, 0)][rng.integers(5)]
        halo = int(rng.integers(2))
        mode, csafe, staged, sx0, sv0, sh, scpr = plan(lib, r + [1.0, 1.1], nu, nv, au, av, CH,
                                                       cols, rows, halo)
        m = np.float32(0.01)
        f = [math.floor(np.float32(r[0]) - m), math.floor(np.float32(r[1]) + m) + 1,
             math.floor(np.float32(r[2]) - m), math.floor(np.float32(r[3]) + m) + 1]
        x0 = (f[0] + au - halo) // CH * CH
        cpr, h = (f[1] + au + halo - x0) // CH + 1, f[3] + av - (f[2] + av) + 2 * halo + 1
        skip = r[1] <= -au - 1.01 or r[0] >= nu - au + 0.01 or r[3] <= -av - 1.01 or r[2] >= nv - av + 0.01
        assert (mode == SKIP) == skip
        if not skip:
            assert staged == (cpr * CH <= cols and h <= rows)
            if staged:
                assert (sx0, sv0, sh, scpr) == (x0, f[2] + av - halo, h, cpr)
            inside = r[0] >= -au + 0.01 and r[1] <= nu - 1 - au - 0.01 and r[2] >= -av + 0.01 \
                and r[3] <= nv - 1 - av - 0.01
            assert (mode == INTERIOR) == inside
        seen.add((mode, staged, csafe))
    assert {(SKIP, 0, 0), (INTERIOR, 0, 0), (INTERIOR, 1, 1), (EDGE, 0, 0), (EDGE, 1, 0)} <= seen


def test_samples_stay_inside_the_planned_rectangle(lib):
    """Tiles at every distance from the source, down to 1e-6 voxels: the property that
    the sample loops, which check nothing, rely on."""
    rng = np.random.default_rng(5)
    kinds = np.zeros(3, int)
    out = (ctypes.c_int * 7)()
    for n in range(4000):
        nu, nv, f = 616, 480, 10.0 ** rng.uniform(0.5, 4)
        K = np.array([[f, 0, 307.5], [0, f, 239.5], [0, 0, 1.0]])
        R = np.linalg.qr(rng.standard_normal((3, 3)))[0] if n % 3 else np.eye(3)[rng.permutation(3)]
        near = rng.uniform(-1, 1, 3) * np.array([7.5, 7.5, 0.0]) if n % 2 else np.zeros(3)
        t = near + np.array([0, 0, 10.0 ** rng.uniform(-6, 3)])
        t[2] += np.abs(R[2]).sum() * 7.5  # the nearest corner's distance from the source plane
        M = (K @ np.hstack([R, t[:, None]])) * 10.0 ** rng.uniform(-3, 3)
        au, av = (int(np.clip(np.floor(M[k, 3] / M[2, 3]), -1048576, 1048576)) for k in (0, 1))
        g = np.concatenate([np.r_[M[k, 3] - a * M[2, 3], M[k, :3] - a * M[2, :3]]
                            for k, a in ((0, au), (1, av), (2, 0))]).astype(np.float32)
        CH, cols, rows = [(4, 84, 64), (8, 80, 64), (4, 116, 56), (4, 84, 0)][n % 4]
        bad = lib.outside(g.ctypes.data_as(ctypes.c_void_p), nu, nv, au, av, CH, cols, rows, n & 1,
                          out)
        assert bad == 0, (n, list(out))
        kinds += [out[0] == INTERIOR, out[2], out[0] == EDGE]
    assert (kinds > 100).all(), kinds
