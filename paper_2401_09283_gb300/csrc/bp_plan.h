// Classification of a box of voxels in one view and the plan of its staged footprint,
// from the ranges of its corners' projections.  Plain C++, so that the host tests the
// function that the kernels run.
#pragma once

#include <cmath>

#ifdef __CUDACC__
#define BP_HD __host__ __device__ __forceinline__
#else
#define BP_HD inline
#endif

namespace bpk {

enum { MODE_SKIP = 0, MODE_INTERIOR = 1, MODE_EDGE = 2 };

struct BoxRange {
  float xmin, xmax, ymin, ymax;  // u/w, v/w in the anchored frame
  float wmin, wmax;              // used where every corner is in front
  int nfront;                    // corners in front of the source plane
};

// Whether a corner is in front of the source plane: not at or behind it, not so near
// that the hardware takes the reciprocal as infinite (subnormal w), not a NaN.
BP_HD bool in_front(float w) { return w >= 1.17549435e-38f; }

struct BoxPlan {
  int mode, csafe, staged;
  int sx0, sv0, sh, scpr;        // staged: first pixel, rows, 16-byte chunks per row
};

// au, av: the anchor pixel; CH pixels per 16 bytes; halo: the stencil's reach beyond the
// bilinear taps; a footprint of up to cols x rows pixels fits (0 rows: never staged);
// seq: no box counts as central-safe.
//
// The float conditions below are what bounds the integers: a box is only INTERIOR
// (unchecked taps) or staged (unchecked shared-memory taps) where all its corners lie
// beyond the source plane, and where its extent times the spread of w says that a
// sample's rounding error, at most 6 ulp of the extent times that spread, is below the
// 0.01 px margin (16384 * 6 * 2^-24 = 0.006).  They also exclude infinities and NaNs,
// and corners so near the source plane that a range exceeds what an int holds.
BP_HD BoxPlan plan_box(const BoxRange& r, int nu, int nv, int au, int av, int CH, int cols,
                       int rows, int halo, bool seq) {
  BoxPlan p = {MODE_EDGE, 0, 0, 0, 0, 0, 0};
  const float m = 0.01f;
  // detector [0, n-1] in the anchored frame
  const float ulo = -(float)au, uhi = (float)(nu - 1) - (float)au;
  const float vlo = -(float)av, vhi = (float)(nv - 1) - (float)av;
  if (r.nfront == 0) {
    p.mode = MODE_SKIP;
    return p;
  }
  if (r.nfront != 8) return p;
  if (r.xmax <= ulo - 1.0f - m || r.xmin >= uhi + 1.0f + m || r.ymax <= vlo - 1.0f - m ||
      r.ymin >= vhi + 1.0f + m) {
    p.mode = MODE_SKIP;
    return p;
  }
  const float lim = 16384.0f * (r.wmin / r.wmax);
  if (!(r.wmax <= 1e38f && r.xmax - r.xmin <= lim && r.ymax - r.ymin <= lim &&
        fabsf(r.xmin) <= 4194304.0f && fabsf(r.ymin) <= 4194304.0f))
    return p;
  if (r.xmin >= ulo + m && r.xmax <= uhi - m && r.ymin >= vlo + m && r.ymax <= vhi - m)
    p.mode = MODE_INTERIOR;
  // central differences at the tap pixels use interior neighbours only: taps in
  // [1, n-2], i.e. floor in [1, n-3]
  p.csafe = !seq && r.xmin >= ulo + 1.0f + m && r.xmax <= uhi - 1.0f - m &&
            r.ymin >= vlo + 1.0f + m && r.ymax <= vhi - 1.0f - m;
  const int u0 = (int)floorf(r.xmin - m) + au, u1 = (int)floorf(r.xmax + m) + 1 + au;
  const int v0 = (int)floorf(r.ymin - m) + av, v1 = (int)floorf(r.ymax + m) + 1 + av;
  const int x0 = (u0 - halo) & ~(CH - 1);  // floor to a 16-byte boundary
  const int y0 = v0 - halo;
  const int cpr = (u1 + halo - x0) / CH + 1, h = v1 + halo - y0 + 1;
  if (cpr * CH <= cols && h <= rows) {
    p.staged = 1;
    p.sx0 = x0;
    p.sv0 = y0;
    p.sh = h;
    p.scpr = cpr;
  }
  return p;
}

}  // namespace bpk
