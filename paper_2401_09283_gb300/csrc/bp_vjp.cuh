// The motion VJP (Eqs. 4-5), optionally fused with the data VJP: one kernel template,
// compiled by bp_vjp_motion.cu (CENTRAL motion), bp_vjp_fused.cu (CENTRAL, both
// gradients) and bp_vjp_exact.cu (BILINEAR_EXACT).  Decomposition, records and staging
// as described in bp_project.cu.
#pragma once

#include "bp_scatter.cuh"

namespace bpk {

// ------------------------------------------------------- VJP w.r.t. Phat

// Sum of 16 per-lane values over the warp, scattered: lane l ends with the
// total of slot 8*b4 + 4*b3 + 2*b2 + b1 (b_i = bit i of l); lanes 2s and 2s+1
// hold the same slot.
__device__ __forceinline__ float warp_reduce_scatter16(float (&v)[16], int lane) {
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    const bool hi = lane & 16;
    float send = hi ? v[s] : v[s + 8];
    float keep = hi ? v[s + 8] : v[s];
    v[s] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
  }
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const bool hi = lane & 8;
    float send = hi ? v[s] : v[s + 4];
    float keep = hi ? v[s + 4] : v[s];
    v[s] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
  }
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const bool hi = lane & 4;
    float send = hi ? v[s] : v[s + 2];
    float keep = hi ? v[s + 2] : v[s];
    v[s] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
  }
  {
    const bool hi = lane & 2;
    float send = hi ? v[0] : v[1];
    float keep = hi ? v[1] : v[0];
    v[0] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
  }
  v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
  return v[0];
}

__device__ __forceinline__ int scatter_slot(int lane) {
  return ((lane >> 4) & 1) * 8 + ((lane >> 3) & 1) * 4 + ((lane >> 2) & 1) * 2 + ((lane >> 1) & 1);
}

// Per voxel-view, with s = delta * c * omega and r = 1/w, the derivative of
// the weighted sample with respect to (u_rel, v_rel, w) (Eq. 4 in the
// anchored frame): a = s*r*(g_u, g_v, -(g_u x + g_v y)) and, with FDK, the
// derivative of omega = wgt r^2 adds -2 s r val to the w component.  The
// 3x4 outer product with (dq, 1) is accumulated as S_r = sum a_r and
// Z_r = sum a_r dz along the thread's column; dx, dy are constant per thread.
//
// Sources of the samples (SRC):
//   SRC_GLOBAL  gradient images (CENTRAL) or raw taps (EXACT) from global memory;
//   SRC_SMEM    the tile footprint staged in shared memory (EXACT; staged
//               CENTRAL tiles run vjp_view_central2 below).
enum { SRC_GLOBAL = 0, SRC_SMEM = 1 };

//
// A staged footprint is zero-padded and covers every tap, so with SRC_SMEM
// the coordinates are never clamped (EDGE then only guards the scatter of
// the fused data VJP).
template <int ZB, typename T, bool FDK, bool EXACT, bool EDGE, bool PROJ, int SRC,
          int P = StageGeom<T>::P>
__device__ __forceinline__ void vjp_view(const T* img, const float2* gimg, unsigned buf,
                                         float* pout, float* qout, long long rs, int nu, int nv,
                                         const TileView& t, float dx, float dy,
                                         const float (&delta)[ZB], float (&S)[3], float (&Z)[3]) {
  constexpr bool CLAMP = EDGE && SRC == SRC_GLOBAL;
  
  float u0 = fmaf(dy, t.ru1, fmaf(dx, t.ru0, t.U0));
  float v0 = fmaf(dy, t.rv1, fmaf(dx, t.rv0, t.V0));
  float w0 = fmaf(dy, t.rw1, fmaf(dx, t.rw0, t.W0));
#pragma unroll
  for (int k = 0; k < ZB; ++k) {
    const float dz = k - 0.5f * (ZB - 1);
    Sample s = locate<CLAMP>(fmaf(dz, t.ru2, u0), fmaf(dz, t.rv2, v0), fmaf(dz, t.rw2, w0),
                             t, nu, nv);
    if (CLAMP && !s.ok) continue;
    float gu, gv, val = 0.0f;
    if (EXACT) {
      float d00, d10, d01, d11;
      if (SRC == SRC_SMEM) {
        const unsigned q = staged_tap<T, 0>(buf, t, s.bx, s.by);
        d00 = lds<0>(q);
        d10 = lds<1>(q);
        d01 = lds<P>(q);
        d11 = lds<P + 1>(q);
      } else {
        taps<EDGE>(img, rs, nu, nv, s, d00, d10, d01, d11);
      }
      const float a = d10 - d00, b = d11 - d01;
      gu = fmaf(s.tv, b - a, a);
      const float c = d01 - d00, d = d11 - d10;
      gv = fmaf(s.tu, d - c, c);
      if (FDK) val = bilerp(s.tu, s.tv, d00, d10, d01, d11);
    } else {
      float2 g00, g10, g01, g11;
      const float2 z2 = make_float2(0.0f, 0.0f);
      if (!EDGE) {
        int iu = s.iu, iv = s.iv;
        bc_interior(BC_GLOBAL_TAP, iu, iv, nu, nv);
        const float2* p = gimg + (long long)iv * nu + iu;
        g00 = __ldg(p);
        g10 = __ldg(p + 1);
        g01 = __ldg(p + nu);
        g11 = __ldg(p + nu + 1);
      } else {
        bool uu0 = (unsigned)s.iu < (unsigned)nu, uu1 = (unsigned)(s.iu + 1) < (unsigned)nu;
        bool vv0 = (unsigned)s.iv < (unsigned)nv, vv1 = (unsigned)(s.iv + 1) < (unsigned)nv;
        const float2* p = gimg + (long long)s.iv * nu + s.iu;
        g00 = (uu0 && vv0 && s.ok) ? __ldg(p) : z2;
        g10 = (uu1 && vv0 && s.ok) ? __ldg(p + 1) : z2;
        g01 = (uu0 && vv1 && s.ok) ? __ldg(p + nu) : z2;
        g11 = (uu1 && vv1 && s.ok) ? __ldg(p + nu + 1) : z2;
      }
      gu = bilerp(s.tu, s.tv, g00.x, g10.x, g01.x, g11.x);
      gv = bilerp(s.tu, s.tv, g00.y, g10.y, g01.y, g11.y);
      if (FDK) {
        float d00, d10, d01, d11;
        taps<EDGE>(img, rs, nu, nv, s, d00, d10, d01, d11);
        val = bilerp(s.tu, s.tv, d00, d10, d01, d11);
      }
    }
    float sd = delta[k] * (FDK ? s.rwi * (s.rwi * t.wgt) : t.wgt);
    const float sr = sd * s.rwi;
    const float a0 = gu * sr, a1 = gv * sr;
    float a2 = -fmaf(a0, s.x, a1 * s.y);
    if (FDK) a2 = fmaf(-2.0f * sr, val, a2);
    S[0] += a0;
    S[1] += a1;
    S[2] += a2;
    Z[0] = fmaf(a0, dz, Z[0]);
    Z[1] = fmaf(a1, dz, Z[1]);
    Z[2] = fmaf(a2, dz, Z[2]);
    if (PROJ && delta[k] != 0.0f)  // fused data VJP: same sample, dequantised weight
      scatter_sample<EDGE>(pout, qout, nu, nv, s,
                           delta[k] * (FDK ? s.rwi * (s.rwi * t.wgtd) : t.wgtd));
  }
}

// The tile's dL/dvol in shared memory, element k of thread tid's column.  The
// fused data VJP's line pass needs [z][y][x] (row pitch TX + 1); otherwise the
// columns are stored as [k / 2][thread] pairs, one conflict-free 8-byte load
// per pair of voxels.
template <bool PROJ>
__device__ __forceinline__ int delta_base(int lx, int ly) {
  return PROJ ? ly * (TX + 1) + lx : 2 * (int)threadIdx.x;
}
template <bool PROJ>
__device__ __forceinline__ int delta_off(int k) {
  return PROJ ? k * (TY * (TX + 1)) : (k >> 1) * (2 * NT) + (k & 1);
}

// The sums of one thread's column over a view (see vjp_view).
struct Sums6 {
  float S[3], Z[3];
};

// One view from global memory of a tile that crosses the detector's edge (or
// whose footprint is not staged): the arithmetic of vjp_view, in the same
// order.  A loop over pairs of voxels, not one unrolled body: such a body was
// ~30 KB of code, and the warps, which drift apart, streamed it through the
// instruction cache.  A pair that is off the detector for the whole warp is
// left out (its gradients are 0; a non-finite upstream value keeps its pair,
// 0 * inf must stay NaN).  delta(k) gives the upstream gradient of voxel k.
template <int ZS, typename T, bool FDK, bool EXACT, bool PROJ>
__device__ __forceinline__ Sums6 vjp_view_edge(const T* img, const float2* gimg, float* pout,
                                            long long rs, int nu, int nv, const TileView& t,
                                            float dx, float dy, const float* delta, float zlo,
                                            const Sums6& from) {
  float S[3] = {from.S[0], from.S[1], from.S[2]}, Z[3] = {from.Z[0], from.Z[1], from.Z[2]};
  const float u0 = fmaf(dy, t.ru1, fmaf(dx, t.ru0, t.U0));
  const float v0 = fmaf(dy, t.rv1, fmaf(dx, t.rv0, t.V0));
  const float w0 = fmaf(dy, t.rw1, fmaf(dx, t.rw0, t.W0));
#pragma unroll 1
  for (int k0 = 0; k0 < ZS; k0 += 2) {
    constexpr int G = 2;
    Sample s[G];
    float d[G], gu[G], gv[G], val[G];
    bool live = false;
#pragma unroll
    for (int q = 0; q < G; ++q) {
      const float dz = (k0 + q) + zlo;
      s[q] = locate<true>(fmaf(dz, t.ru2, u0), fmaf(dz, t.rv2, v0), fmaf(dz, t.rw2, w0), t, nu, nv);
      d[q] = delta[delta_off<PROJ>(k0 + q)];
      val[q] = 0.0f;
      live |= (s[q].ok && (unsigned)(s[q].iu + 1) <= (unsigned)nu &&
               (unsigned)(s[q].iv + 1) <= (unsigned)nv) ||
              !(fabsf(d[q]) <= 3.402823466e38f);
    }
    if (!__any_sync(0xffffffffu, live)) continue;
#pragma unroll
    for (int q = 0; q < G; ++q) {
      float d00, d10, d01, d11;
      if (EXACT || FDK) taps<true>(img, rs, nu, nv, s[q], d00, d10, d01, d11);
      if (EXACT) {
        const float a = d10 - d00, b = d11 - d01;
        gu[q] = fmaf(s[q].tv, b - a, a);
        const float c = d01 - d00, e = d11 - d10;
        gv[q] = fmaf(s[q].tu, e - c, c);
      } else {
        const float2 z2 = make_float2(0.0f, 0.0f);
        const bool uu0 = (unsigned)s[q].iu < (unsigned)nu;
        const bool uu1 = (unsigned)(s[q].iu + 1) < (unsigned)nu;
        const bool vv0 = (unsigned)s[q].iv < (unsigned)nv;
        const bool vv1 = (unsigned)(s[q].iv + 1) < (unsigned)nv;
        const float2* p = gimg + (long long)s[q].iv * nu + s[q].iu;
        const float2 g00 = (uu0 && vv0 && s[q].ok) ? __ldg(p) : z2;
        const float2 g10 = (uu1 && vv0 && s[q].ok) ? __ldg(p + 1) : z2;
        const float2 g01 = (uu0 && vv1 && s[q].ok) ? __ldg(p + nu) : z2;
        const float2 g11 = (uu1 && vv1 && s[q].ok) ? __ldg(p + nu + 1) : z2;
        gu[q] = bilerp(s[q].tu, s[q].tv, g00.x, g10.x, g01.x, g11.x);
        gv[q] = bilerp(s[q].tu, s[q].tv, g00.y, g10.y, g01.y, g11.y);
      }
      if (FDK) val[q] = bilerp(s[q].tu, s[q].tv, d00, d10, d01, d11);
    }
#pragma unroll
    for (int q = 0; q < G; ++q) {
      if (!s[q].ok) continue;
      const float dz = (k0 + q) + zlo;
      const float sd = d[q] * (FDK ? s[q].rwi * (s[q].rwi * t.wgt) : t.wgt);
      const float sr = sd * s[q].rwi;
      const float a0 = gu[q] * sr, a1 = gv[q] * sr;
      float a2 = -fmaf(a0, s[q].x, a1 * s[q].y);
      if (FDK) a2 = fmaf(-2.0f * sr, val[q], a2);
      S[0] += a0;
      S[1] += a1;
      S[2] += a2;
      Z[0] = fmaf(a0, dz, Z[0]);
      Z[1] = fmaf(a1, dz, Z[1]);
      Z[2] = fmaf(a2, dz, Z[2]);
      if (PROJ && d[q] != 0.0f)
        scatter_sample<true>(pout, nullptr, nu, nv, s[q],
                             d[q] * (FDK ? s[q].rwi * (s[q].rwi * t.wgtd) : t.wgtd));
    }
  }
  return Sums6{{S[0], S[1], S[2]}, {Z[0], Z[1], Z[2]}};
}

// Twice the difference of one tap pixel along an axis from its neighbours l, r
// (c is the pixel itself): r - l inside, twice the one-sided difference on the
// first and last pixel, 0 off the detector -- the gradient images' values, bit
// for bit (times 2).  f is the pixel's coordinate, [lo, hi] the detector's, as
// floats that hold integers.
struct EdgeRule {
  bool first, last, off;
  __device__ __forceinline__ EdgeRule(float f, float lo, float hi)
      : first(f == lo), last(f == hi), off(f < lo || f > hi) {}
  __device__ __forceinline__ float operator()(float l, float c, float r) const {
    const float d = (last ? c : r) - (first ? c : l);
    return off ? 0.0f : (first || last) ? d + d : d;
  }
};

// Range of dz with a + b dz >= 0, intersected into [lo, hi].
__device__ __forceinline__ void clip_range(float a, float b, float& lo, float& hi) {
  const float q = __fdividef(-a, b);
  if (b > 0.0f) lo = fmaxf(lo, q);
  else if (b < 0.0f) hi = fminf(hi, q);
  else if (a < 0.0f) hi = -INFINITY;
}

// Range of dz in which a column's samples lie in [x0, x1] x [y0, y1] (anchored
// pixels; w > 0): u/w >= x0 is linear in dz, u - x0 w >= 0.
__device__ __forceinline__ void column_range(const TileView& t, float u0, float v0, float w0,
                                             float x0, float x1, float y0, float y1, float& lo,
                                             float& hi) {
  lo = -INFINITY;
  hi = INFINITY;
  clip_range(fmaf(-x0, w0, u0), fmaf(-x0, t.rw2, t.ru2), lo, hi);
  clip_range(fmaf(x1, w0, -u0), fmaf(x1, t.rw2, -t.ru2), lo, hi);
  clip_range(fmaf(-y0, w0, v0), fmaf(-y0, t.rw2, t.rv2), lo, hi);
  clip_range(fmaf(y1, w0, -v0), fmaf(y1, t.rw2, -t.rv2), lo, hi);
}

// One view of a staged CENTRAL tile that crosses the detector's edge: the
// packed arithmetic of vjp_view_central2 on the zero-padded footprint, the sums
// taken sample by sample as vjp_view_edge takes them.  Per column the slices
// that touch the detector and those that are central-safe are intervals (a
// linear inequality per detector side), so a warp visits only the pairs some
// lane needs, and pairs that are safe for every lane run without any test; in
// the others each sample is classified, the edge rules of the gradient images
// are applied to the differences where needed, and only samples that touch the
// detector are added.  The intervals are taken 0.01 px wide (on) and narrow
// (safe), far beyond their rounding error.  Reading the gradient images from
// global memory here instead (eight scattered loads per sample) took 2.5 times
// as long per (tile, view) as a central-safe one.
template <int ZS, typename G, bool FDK, bool PROJ>
__device__ __forceinline__ Sums6 vjp_view_edge2(unsigned buf, float* pout, float* qout, int nu, int nv,
                                             const TileView& t, float dx, float dy,
                                             const float* delta, float zlo, bool finite,
                                             const Sums6& from) {
  float S[3] = {from.S[0], from.S[1], from.S[2]}, Z[3] = {from.Z[0], from.Z[1], from.Z[2]};
  constexpr int P = StageGeom<G>::P;
  const float u0 = fmaf(dy, t.ru1, fmaf(dx, t.ru0, t.U0));
  const float v0 = fmaf(dy, t.rv1, fmaf(dx, t.rv0, t.V0));
  const float w0 = fmaf(dy, t.rw1, fmaf(dx, t.rw0, t.W0));
  const f2 M2 = pk2(MAGIC, MAGIC), HALF = pk2(0.5f, 0.5f), IC = staged_anchor(buf, t);
  const f2 WG = pk2(t.wgt, t.wgt), WGD = pk2(t.wgtd, t.wgtd);
  // detector pixels [xl, xr] x [yl, yr] in the anchored frame
  const float xl = -(float)t.au, xr = (float)(nu - 1 - t.au);
  const float yl = -(float)t.av, yr = (float)(nv - 1 - t.av);
  constexpr float M = 0.01f;
  const float HZ = -zlo;
  float lo, hi;
  column_range(t, u0, v0, w0, xl - 1.0f - M, xr + 1.0f + M, yl - 1.0f - M, yr + 1.0f + M, lo, hi);
  int k0 = 0, k1 = ZS;  // slices that touch the detector in some lane
  if (finite) {
    const bool some = lo <= hi;
    k0 = __reduce_min_sync(0xffffffffu,
                           some ? (int)ceilf(fminf(fmaxf(lo + HZ, 0.0f), (float)ZS)) : ZS);
    k1 = __reduce_max_sync(0xffffffffu,
                           some ? (int)floorf(fminf(fmaxf(hi + HZ, -1.0f), ZS - 1.0f)) + 1 : 0);
  }
  column_range(t, u0, v0, w0, xl + 1.0f + M, xr - 1.0f - M, yl + 1.0f + M, yr - 1.0f - M, lo, hi);
  // slices [s0, s1) are central-safe in every lane
  const bool some = finite && lo <= hi;
  const int s0 = __reduce_max_sync(
      0xffffffffu, some ? (int)ceilf(fminf(fmaxf(lo + HZ, 0.0f), (float)ZS)) : ZS);
  const int s1 = __reduce_min_sync(
      0xffffffffu, some ? (int)floorf(fminf(fmaxf(hi + HZ, -1.0f), ZS - 1.0f)) + 1 : 0);
#pragma unroll 1
  for (int k = k0 & ~1; k < k1; k += 2) {
    const bool safe = k >= s0 && k + 2 <= s1;
    const float dz0 = k - HZ;
    const f2 dz = pk2(dz0, dz0 + 1.0f);
    const f2 u = fma2(dz, pk2(t.ru2, t.ru2), pk2(u0, u0));
    const f2 v = fma2(dz, pk2(t.rv2, t.rv2), pk2(v0, v0));
    const f2 w = fma2(dz, pk2(t.rw2, t.rw2), pk2(w0, w0));
    float wl, wh;
    up2(w, wl, wh);
    const f2 r = pk2(rcp_approx(wl), rcp_approx(wh));
    const f2 x = mul2(u, r), y = mul2(v, r);
    const f2 fx = sub2(add2_rd(x, M2), M2), fy = sub2(add2_rd(y, M2), M2);
    float d[2], xs[2], ys[2], fxs[2], fys[2];
    up2(x, xs[0], xs[1]);
    up2(y, ys[0], ys[1]);
    up2(fx, fxs[0], fxs[1]);
    up2(fy, fys[0], fys[1]);
    bool use[2] = {true, true};
    unsigned flags = safe ? 1u : 0u;  // 1: a sample to add, 2 / 4: one at the border along u / v
#pragma unroll
    for (int q = 0; q < 2; ++q) d[q] = delta[delta_off<PROJ>(k + q)];
    if (!safe) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      use[q] = (fxs[q] >= xl - 1.0f && fxs[q] <= xr && fys[q] >= yl - 1.0f && fys[q] <= yr) ||
               !(fabsf(d[q]) <= 3.402823466e38f);
      if (use[q])  // a central-safe sample has its floor pixel in [1, n-3]
        flags |= 1u | (fxs[q] >= xl + 1.0f && fxs[q] <= xr - 2.0f ? 0u : 2u) |
                 (fys[q] >= yl + 1.0f && fys[q] <= yr - 2.0f ? 0u : 4u);
    }
    flags = __reduce_or_sync(0xffffffffu, flags);
    if (!flags) continue;
    }
    const f2 tu = sub2(x, fx), tv = sub2(y, fy);
    unsigned ql, qh;
    staged_pair<G, 1>(buf, t, IC, fx, fy, ql, qh);
    const f2 a0 = lds2<-P>(ql, qh), a1 = lds2<-P + 1>(ql, qh);
    const f2 b0 = lds2<-1>(ql, qh), b1 = lds2<0>(ql, qh), b2 = lds2<1>(ql, qh),
             b3 = lds2<2>(ql, qh);
    const f2 c0 = lds2<P - 1>(ql, qh), c1 = lds2<P>(ql, qh), c2 = lds2<P + 1>(ql, qh),
             c3 = lds2<P + 2>(ql, qh);
    const f2 e0 = lds2<2 * P>(ql, qh), e1 = lds2<2 * P + 1>(ql, qh);
    // twice the gradient images' values at the four tap pixels
    f2 gu00, gu10, gu01, gu11, gv00, gv10, gv01, gv11;
#define BP_RULE(rule, g, l, c, r_)                                        \
  {                                                                       \
    float l0, l1, m0, m1, n0, n1;                                         \
    up2(l, l0, l1);                                                       \
    up2(c, m0, m1);                                                       \
    up2(r_, n0, n1);                                                      \
    g = pk2(rule##0(l0, m0, n0), rule##1(l1, m1, n1));                    \
  }
    if (flags & 2u) {
      const EdgeRule p0(fxs[0], xl, xr), p1(fxs[1], xl, xr);
      BP_RULE(p, gu00, b0, b1, b2)
      BP_RULE(p, gu01, c0, c1, c2)
      const EdgeRule q0(fxs[0] + 1.0f, xl, xr), q1(fxs[1] + 1.0f, xl, xr);
      BP_RULE(q, gu10, b1, b2, b3)
      BP_RULE(q, gu11, c1, c2, c3)
    } else {
      gu00 = sub2(b2, b0);
      gu10 = sub2(b3, b1);
      gu01 = sub2(c2, c0);
      gu11 = sub2(c3, c1);
    }
    if (flags & 4u) {
      const EdgeRule p0(fys[0], yl, yr), p1(fys[1], yl, yr);
      BP_RULE(p, gv00, a0, b1, c1)
      BP_RULE(p, gv10, a1, b2, c2)
      const EdgeRule q0(fys[0] + 1.0f, yl, yr), q1(fys[1] + 1.0f, yl, yr);
      BP_RULE(q, gv01, b1, c1, e0)
      BP_RULE(q, gv11, b2, c2, e1)
    } else {
      gv00 = sub2(c1, a0);
      gv10 = sub2(c2, a1);
      gv01 = sub2(e0, b1);
      gv11 = sub2(e1, b2);
    }
#undef BP_RULE
    const f2 D = pk2(d[0], d[1]);
    const f2 sr = mul2(mul2(D, FDK ? mul2(r, mul2(r, WG)) : WG), r);
    float gu[2], gv[2], val[2], srs[2], sgs[2];
    up2(bilerp2(tu, tv, gu00, gu10, gu01, gu11), gu[0], gu[1]);
    up2(bilerp2(tu, tv, gv00, gv10, gv01, gv11), gv[0], gv[1]);
    if (FDK) up2(bilerp2(tu, tv, b1, b2, c1, c2), val[0], val[1]);
    up2(sr, srs[0], srs[1]);
    up2(mul2(sr, HALF), sgs[0], sgs[1]);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      if (!use[q]) continue;
      const float a0s = gu[q] * sgs[q], a1s = gv[q] * sgs[q];
      float a2s = -fmaf(a0s, xs[q], a1s * ys[q]);
      if (FDK) a2s = fmaf(-2.0f * srs[q], val[q], a2s);
      S[0] += a0s;
      S[1] += a1s;
      S[2] += a2s;
      Z[0] = fmaf(a0s, dz0 + q, Z[0]);
      Z[1] = fmaf(a1s, dz0 + q, Z[1]);
      Z[2] = fmaf(a2s, dz0 + q, Z[2]);
    }
    if (PROJ) {
      float tus[2], tvs_[2], sp[2];
      up2(tu, tus[0], tus[1]);
      up2(tv, tvs_[0], tvs_[1]);
      up2(mul2(D, FDK ? mul2(r, mul2(r, WGD)) : WGD), sp[0], sp[1]);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        if (!use[q] || d[q] == 0.0f) continue;
        Sample s;
        s.tu = tus[q];
        s.tv = tvs_[q];
        s.iu = (int)fxs[q] + t.au;
        s.iv = (int)fys[q] + t.av;
        scatter_sample<true>(pout, qout, nu, nv, s, sp[q]);
      }
    }
  }
  return Sums6{{S[0], S[1], S[2]}, {Z[0], Z[1], Z[2]}};
}

// Whether scatters go to the block image (see vjp_view_central2).
template <int BLK>
__device__ __forceinline__ bool to_blocks(const float* qout) {
  return BP_VJP_BLOCKS && (BLK == 1 || (BLK == 2 && qout));
}

// The CENTRAL sample loop from a staged central-safe footprint with packed
// pairs of voxels (k, k+1): the steps of vjp_view in the same order on
// f32x2 pairs, with the w-component kept negated (na2 = -a2) so that no
// negation instruction is needed.  Even and odd voxels are summed in the two
// halves of the pair accumulators and added at the end.  ZS slices from dz = zlo on,
// dcol their upstream gradients.
// With SEQ the sums are taken sample by sample instead, on top of S and Z.
// BLK: whether the fused data VJP goes to the block image qout: 0 or 1, or 2, a test per
// sample.  That takes three instructions of about 80, but one copy of the body: with four
// slots, where there is one CTA per SM or two, two copies spilled (32^3 x 60 views, both
// gradients, 38.0 against 36.3 us).
template <int ZS, typename G, bool FDK, bool PROJ, bool LINES, bool SEQ, int BLK>
__device__ __forceinline__ void vjp_view_central2(unsigned buf, float* pout, float* qout, int nu,
                                                  int nv, const TileView& t, float dx, float dy,
                                                  const float* dcol, float zlo,
                                                  float (&S)[3], float (&Z)[3]) {
  constexpr int P = StageGeom<G>::P;
  const f2 IC = staged_anchor(buf, t);
  const float u0 = fmaf(dy, t.ru1, fmaf(dx, t.ru0, t.U0));
  const float v0 = fmaf(dy, t.rv1, fmaf(dx, t.rv0, t.V0));
  const float w0 = fmaf(dy, t.rw1, fmaf(dx, t.rw0, t.W0));
  const f2 U0 = pk2(u0, u0), V0 = pk2(v0, v0), W0 = pk2(w0, w0);
  const f2 RU = pk2(t.ru2, t.ru2), RV = pk2(t.rv2, t.rv2), RW = pk2(t.rw2, t.rw2);
  const f2 M2 = pk2(MAGIC, MAGIC), TWO = pk2(2.0f, 2.0f), FOUR = pk2(4.0f, 4.0f);
  const f2 WG = pk2(0.5f * t.wgt, 0.5f * t.wgt);  // half: the differences are twice the gradients
  const f2 WGD = pk2(t.wgtd, t.wgtd);
  // pixel index offset of the floor bits: (av - MAGIC_BITS) nu + au - MAGIC_BITS
  const unsigned pofs = (unsigned)(t.av - MAGIC_BITS) * (unsigned)nu + (unsigned)(t.au - MAGIC_BITS);
  const f2 zero = pk2(0.0f, 0.0f);
  f2 dz = pk2(zlo, zlo + 1.0f);
  f2 S0 = zero, S1 = zero, S2 = zero, Z0 = zero, Z1 = zero, Z2 = zero;
#pragma unroll
  for (int p = 0; p < ZS / 2; ++p) {
    if (p) dz = add2(dz, TWO);
    const f2 u = fma2(dz, RU, U0), v = fma2(dz, RV, V0), w = fma2(dz, RW, W0);
    float wl, wh;
    up2(w, wl, wh);
    const f2 r = pk2(rcp_approx(wl), rcp_approx(wh));
    const f2 x = mul2(u, r), y = mul2(v, r);
    const f2 rx = add2_rd(x, M2), ry = add2_rd(y, M2);
    const f2 fx = sub2(rx, M2), fy = sub2(ry, M2);
    const f2 tu = sub2(x, fx), tv = sub2(y, fy);
    unsigned ql, qh;
    staged_pair<G, 1>(buf, t, IC, fx, fy, ql, qh);
    const f2 a0 = lds2<-P>(ql, qh), a1 = lds2<-P + 1>(ql, qh);
    const f2 b0 = lds2<-1>(ql, qh), b1 = lds2<0>(ql, qh), b2 = lds2<1>(ql, qh),
             b3 = lds2<2>(ql, qh);
    const f2 c0 = lds2<P - 1>(ql, qh), c1 = lds2<P>(ql, qh), c2 = lds2<P + 1>(ql, qh),
             c3 = lds2<P + 2>(ql, qh);
    const f2 e0 = lds2<2 * P>(ql, qh), e1 = lds2<2 * P + 1>(ql, qh);
    // twice the central-difference gradient images at the four tap pixels
    const f2 gu = bilerp2(tu, tv, sub2(b2, b0), sub2(b3, b1), sub2(c2, c0), sub2(c3, c1));
    const f2 gv = bilerp2(tu, tv, sub2(c1, a0), sub2(c2, a1), sub2(e0, b1), sub2(e1, b2));
    // (from shared memory: the column's 16 registers would spill others; fused VJP
    // of c2 15.85 -> 15.32 ms, motion VJP 10.5 -> 10.0 ms when it was measured)
    const f2 D = LINES ? pk2(dcol[delta_off<true>(2 * p)], dcol[delta_off<true>(2 * p + 1)])
                       : *reinterpret_cast<const f2*>(dcol + delta_off<false>(2 * p));
    const f2 sd = mul2(D, FDK ? mul2(r, mul2(r, WG)) : WG);
    const f2 sg = mul2(sd, r);
    const f2 A0 = mul2(gu, sg), A1 = mul2(gv, sg);
    f2 NA2 = fma2(A0, x, mul2(A1, y));
    if (FDK) NA2 = fma2(mul2(sg, FOUR), bilerp2(tu, tv, b1, b2, c1, c2), NA2);
    if constexpr (SEQ) {
      float a0[2], a1[2], n2[2], z[2];
      up2(A0, a0[0], a0[1]);
      up2(A1, a1[0], a1[1]);
      up2(NA2, n2[0], n2[1]);
      up2(dz, z[0], z[1]);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        S[0] += a0[q];
        S[1] += a1[q];
        S[2] -= n2[q];
        Z[0] = fmaf(a0[q], z[q], Z[0]);
        Z[1] = fmaf(a1[q], z[q], Z[1]);
        Z[2] = fmaf(-n2[q], z[q], Z[2]);
      }
      continue;
    }
    S0 = add2(S0, A0);
    S1 = add2(S1, A1);
    S2 = sub2(S2, NA2);
    Z0 = fma2(A0, dz, Z0);
    Z1 = fma2(A1, dz, Z1);
    Z2 = fma2(NA2, dz, Z2);  // minus the sum
    if (PROJ) {
      // fused data VJP, per voxel: the same sample's bilinear weights (the
      // scalar scatter's formulas, packed), dequantised view weight, four
      // FP32 atomic adds per voxel; interior tiles only (no bounds checks)
      const f2 SD = mul2(D, FDK ? mul2(r, mul2(r, WGD)) : WGD);
      const f2 Q1 = mul2(SD, tv), Q0 = sub2(SD, Q1);
      const f2 W11 = mul2(Q1, tu), W01 = sub2(Q1, W11), W10 = mul2(Q0, tu), W00 = sub2(Q0, W10);
      float bxl, bxh, byl, byh;
      up2(rx, bxl, bxh);
      up2(ry, byl, byh);
      float w[4][2];
      up2(W00, w[0][0], w[0][1]);
      up2(W10, w[1][0], w[1][1]);
      up2(W01, w[2][0], w[2][1]);
      up2(W11, w[3][0], w[3][1]);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        int bxi = __float_as_int(h ? bxh : bxl), byi = __float_as_int(h ? byh : byl);
#ifdef BP_BOUNDS_CHECK
        int iu = bxi - MAGIC_BITS + t.au, iv = byi - MAGIC_BITS + t.av;
        bc_interior(BC_SCATTER, iu, iv, nu, nv);
        bxi = iu + MAGIC_BITS - t.au;
        byi = iv + MAGIC_BITS - t.av;
#endif
        // (iv * nu + iu) from the floor bits, in 32-bit wraparound arithmetic
        const unsigned px = (unsigned)byi * (unsigned)nu + (unsigned)bxi + pofs;
        if (to_blocks<BLK>(qout)) {  // one vector reduction into the block image
          red_v4(block_at(qout, px), w[0][h], w[1][h], w[2][h], w[3][h]);
          continue;
        }
        float* q = pout + px;
        atomicAdd(q, w[0][h]);
        atomicAdd(q + 1, w[1][h]);
        atomicAdd(q + nu, w[2][h]);
        atomicAdd(q + nu + 1, w[3][h]);
      }
    }
  }
  if (SEQ) return;
  float lo, hi;
  up2(S0, lo, hi); S[0] += lo + hi;
  up2(S1, lo, hi); S[1] += lo + hi;
  up2(S2, lo, hi); S[2] += lo + hi;
  up2(Z0, lo, hi); Z[0] += lo + hi;
  up2(Z1, lo, hi); Z[1] += lo + hi;
  up2(Z2, lo, hi); Z[2] -= lo + hi;
}

// Fused data VJP by lines (below) or per sample (the scalar loop).
#ifndef BP_VJP_LINES
#define BP_VJP_LINES 1
#endif
#ifndef BP_VJP_LINE_DU
#define BP_VJP_LINE_DU 0.5f
#endif

// Data VJP of one staged central-safe (hence interior) tile-view, by lines:
// thread (a, b) walks the 16 voxels of the tile's line along the axis, x or
// y, whose voxels project closest together on the detector (there the sample
// moves by less than the per-view threshold along u per voxel and barely
// along v), in the direction of increasing u.  The bilinear weights of
// consecutive samples that fall in the same detector cell (same floor pixel)
// are summed in registers, and a cell's four pixels are added to dL/dproj
// (FP32 L2 atomics) only when the line leaves it: about 4 (du + 1/16) atomic
// adds per sample instead of 4.  The arithmetic runs on packed pairs of
// consecutive voxels (f32x2), as in the motion loop.  Exact to rounding: the
// same weights, summed in another order.  dsm holds the tile's dL/dvol as
// [z][y][x] with a row pitch of TX + 1.
template <int ZB, bool FDK, int BLK>
__device__ __forceinline__ void proj_lines(float* __restrict__ pout, float* __restrict__ qout,
                                           int nu, int nv, const TileView& t,
                                           const float* __restrict__ dsm) {
  static_assert(ZB == TX && TY == TX, "lines run along a 16-voxel tile edge");
  const int a = threadIdx.x & (TX - 1), b = threadIdx.x / TX;
  const bool alongx = fabsf(t.ru0) <= fabsf(t.ru1);
  const float fa = a - 0.5f * (TX - 1), fb = b - 0.5f * (ZB - 1);
  // x-lines: voxels (k, a, b); y-lines: (a, k, b)
  const float ou = alongx ? t.ru1 : t.ru0, ov = alongx ? t.rv1 : t.rv0;
  const float ow = alongx ? t.rw1 : t.rw0;
  float su = alongx ? t.ru0 : t.ru1, sv = alongx ? t.rv0 : t.rv1;
  float sw = alongx ? t.rw0 : t.rw1;
  const float u0 = fmaf(fb, t.ru2, fmaf(fa, ou, t.U0));
  const float v0 = fmaf(fb, t.rv2, fmaf(fa, ov, t.V0));
  const float w0 = fmaf(fb, t.rw2, fmaf(fa, ow, t.W0));
  // walk in the direction of increasing u: step kk visits voxel k = 15 - kk
  // when the axis runs against u (the negated steps give the same positions)
  const bool rev = su < 0.0f;
  if (rev) {
    su = -su;
    sv = -sv;
    sw = -sw;
  }
  const float* dl = alongx ? dsm + (b * TY + a) * (TX + 1) : dsm + b * TY * (TX + 1) + a;
  const int dstep = alongx ? 1 : TX + 1;
  const f2 U0 = pk2(u0, u0), V0 = pk2(v0, v0), W0 = pk2(w0, w0);
  const f2 SU = pk2(su, su), SV = pk2(sv, sv), SW = pk2(sw, sw);
  const f2 M2 = pk2(MAGIC, MAGIC), TWO = pk2(2.0f, 2.0f), WGD = pk2(t.wgtd, t.wgtd);
  const unsigned pofs = (unsigned)(t.av - MAGIC_BITS) * (unsigned)nu + (unsigned)(t.au - MAGIC_BITS);
  // index of the pixel with floor bits (bx, by), in 32-bit wraparound arithmetic
  auto pixel = [&](int bx, int by) {
#ifdef BP_BOUNDS_CHECK
    int fc = bx - MAGIC_BITS + t.au, fr = by - MAGIC_BITS + t.av;
    bc_interior(BC_SCATTER, fc, fr, nu, nv);
    bx = fc + MAGIC_BITS - t.au;
    by = fr + MAGIC_BITS - t.av;
#endif
    return (unsigned)by * (unsigned)nu + (unsigned)bx + pofs;
  };
  int cb = 0, rb = 0;  // the open cell, as floor bits
  bool have = false;
  float a0 = 0.0f, a1 = 0.0f, b0 = 0.0f, b1 = 0.0f;
  f2 dk = pk2(-0.5f * (TX - 1), 1.0f - 0.5f * (TX - 1));
#pragma unroll 2
  for (int p = 0; p < TX / 2; ++p) {
    if (p) dk = add2(dk, TWO);
    const f2 u = fma2(dk, SU, U0), v = fma2(dk, SV, V0), w = fma2(dk, SW, W0);
    float wl, wh;
    up2(w, wl, wh);
    const f2 r = pk2(rcp_approx(wl), rcp_approx(wh));
    const f2 x = mul2(u, r), y = mul2(v, r);
    const f2 rx = add2_rd(x, M2), ry = add2_rd(y, M2);
    const f2 tu = sub2(x, sub2(rx, M2)), tv = sub2(y, sub2(ry, M2));
    const int k0 = rev ? TX - 1 - 2 * p : 2 * p, k1 = rev ? k0 - 1 : k0 + 1;
    const f2 D = pk2(dl[k0 * dstep], dl[k1 * dstep]);
    const f2 SD = mul2(D, FDK ? mul2(r, mul2(r, WGD)) : WGD);
    const f2 Q1 = mul2(SD, tv), Q0 = sub2(SD, Q1);
    const f2 W11 = mul2(Q1, tu), W01 = sub2(Q1, W11), W10 = mul2(Q0, tu), W00 = sub2(Q0, W10);
    float bxf[2], byf[2], ww[4][2];
    up2(rx, bxf[0], bxf[1]);
    up2(ry, byf[0], byf[1]);
    up2(W00, ww[0][0], ww[0][1]);
    up2(W10, ww[1][0], ww[1][1]);
    up2(W01, ww[2][0], ww[2][1]);
    up2(W11, ww[3][0], ww[3][1]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int bx = __float_as_int(bxf[h]), by = __float_as_int(byf[h]);
      const bool keep = have && bx == cb && by == rb;
      if (have && !keep) {  // the line leaves the open cell: add its four pixels
        const unsigned px = pixel(cb, rb);
        if (to_blocks<BLK>(qout)) {
          red_v4(block_at(qout, px), a0, a1, b0, b1);
        } else {
          float* q = pout + px;
          atomicAdd(q, a0);
          atomicAdd(q + 1, a1);
          atomicAdd(q + nu, b0);
          atomicAdd(q + nu + 1, b1);
        }
      }
      a0 = (keep ? a0 : 0.0f) + ww[0][h];
      a1 = (keep ? a1 : 0.0f) + ww[1][h];
      b0 = (keep ? b0 : 0.0f) + ww[2][h];
      b1 = (keep ? b1 : 0.0f) + ww[3][h];
      cb = bx;
      rb = by;
      have = true;
    }
  }
  const unsigned px = pixel(cb, rb);
  if (to_blocks<BLK>(qout)) {
    red_v4(block_at(qout, px), a0, a1, b0, b1);
    return;
  }
  float* q = pout + px;
  atomicAdd(q, a0);
  atomicAdd(q + 1, a1);
  atomicAdd(q + nu, b0);
  atomicAdd(q + nu + 1, b1);
}

// One view of one tile, or of one half of it: the sample loop (from the staged
// footprint when it was staged), added to the thread's sums.  Staged CENTRAL
// (central-safe) tiles run the packed motion loop and, when the data VJP is fused,
// the line pass above; the other tiles scatter the data VJP per sample.  ZS slices
// from dz = zlo on, dcol their upstream gradients.
template <int ZB, int ZS, int NS, typename T, bool FDK, bool EXACT, bool PROJ, int STAGE>
__device__ __forceinline__ void vjp_tile_view(const T* img, const float2* gimg, unsigned buf,
                                              bool staged, float* pout, float* qout,
                                              const ProjInfo& pi, const TileView& t,
                                              const TileIdx& ti, float zlo,
                                              const float (&delta)[ZB], const float* dcol,
                                              bool finite, const float* dsm, float (&S)[3],
                                              float (&Z)[3]) {
  using G = Geo<T, STAGE>;
  static_assert(ZS == ZB || (!EXACT && !PROJ), "half tiles: CENTRAL motion VJP only");
  // the lower half's sums go on in the upper half, in the order of the slices
  const Sums6 from = ZS == ZB ? Sums6{{0.0f, 0.0f, 0.0f}, {0.0f, 0.0f, 0.0f}}
                              : Sums6{{S[0], S[1], S[2]}, {Z[0], Z[1], Z[2]}};
  auto take = [&](const Sums6& q) {
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      S[r] = q.S[r];
      Z[r] = q.Z[r];
    }
  };
  if (!EXACT && staged && t.csafe) {
    // With the fused data VJP: the line pass where samples along
    // the ray-parallel axis move by at most BP_VJP_LINE_DU px per voxel
    // (there it merges most: about 4 (du + 1/16) atomics per sample), else
    // four atomics per sample from the packed loop, with fewer instructions
    if constexpr (PROJ) {
      if (BP_VJP_LINES && fminf(fabsf(t.ru0), fabsf(t.ru1)) <= BP_VJP_LINE_DU * t.W0) {
        vjp_view_central2<ZB, G, FDK, false, PROJ, false, 0>(
            buf, pout, qout, pi.nu, pi.nv, t, ti.dx, ti.dy, dcol, zlo, S, Z);
        if (NS > VJP_NS) proj_lines<ZB, FDK, 2>(pout, qout, pi.nu, pi.nv, t, dsm);
        else if (BP_VJP_BLOCKS && qout) proj_lines<ZB, FDK, 1>(pout, qout, pi.nu, pi.nv, t, dsm);
        else proj_lines<ZB, FDK, 0>(pout, qout, pi.nu, pi.nv, t, dsm);
        return;
      }
    }
    if constexpr (PROJ && NS > VJP_NS)
      vjp_view_central2<ZS, G, FDK, PROJ, PROJ, ZS != ZB, 2>(
          buf, pout, qout, pi.nu, pi.nv, t, ti.dx, ti.dy, dcol, zlo, S, Z);
    else if (PROJ && BP_VJP_BLOCKS && qout)
      vjp_view_central2<ZS, G, FDK, PROJ, PROJ, ZS != ZB, PROJ ? 1 : 0>(
          buf, pout, qout, pi.nu, pi.nv, t, ti.dx, ti.dy, dcol, zlo, S, Z);
    else
      vjp_view_central2<ZS, G, FDK, PROJ, PROJ, ZS != ZB, 0>(
          buf, pout, qout, pi.nu, pi.nv, t, ti.dx, ti.dy, dcol, zlo, S, Z);
  } else if (!EXACT && staged) {
    take(vjp_view_edge2<ZS, G, FDK, PROJ>(buf, pout, qout, pi.nu, pi.nv, t, ti.dx, ti.dy, dcol, zlo,
                                          finite, from));
  } else if (EXACT && staged) {
    // (the per-sample paths keep scalar scatters in the fused kernel: block
    // reductions of their in-range samples measured 1 % slower there,
    // 15.12 against 14.94 ms on c2, while the data VJP alone gains 10 %)
    if constexpr (EXACT) {
      if (t.mode == MODE_INTERIOR || !PROJ)
        vjp_view<ZB, T, FDK, EXACT, false, PROJ, SRC_SMEM>(img, gimg, buf, pout, nullptr, pi.rs,
                                                           pi.nu, pi.nv, t, ti.dx, ti.dy, delta, S,
                                                           Z);
      else
        vjp_view<ZB, T, FDK, EXACT, true, PROJ, SRC_SMEM>(img, gimg, buf, pout, nullptr, pi.rs,
                                                          pi.nu, pi.nv, t, ti.dx, ti.dy, delta, S,
                                                          Z);
    }
  } else {
    // CENTRAL with staging: interior tiles come here where their footprint does not fit
    // or is beside the detector's edge, and take the checked path, one code path less.
    // The exact derivative keeps one unrolled body per path, with the column in
    // registers: the looped edge path made its sample loop spill (256^3 x 248, both
    // gradients, 20.8 against 18.9 ms; motion 7.14 against 6.88).
    if constexpr (EXACT || STAGE == STAGE_NONE) {
      if (t.mode == MODE_INTERIOR) {
        vjp_view<ZB, T, FDK, EXACT, false, PROJ, SRC_GLOBAL>(img, gimg, buf, pout, nullptr, pi.rs,
                                                             pi.nu, pi.nv, t, ti.dx, ti.dy, delta,
                                                             S, Z);
        return;
      }
    }
    if constexpr (EXACT && STAGE != STAGE_NONE)
      vjp_view<ZB, T, FDK, EXACT, true, PROJ, SRC_GLOBAL>(img, gimg, buf, pout, nullptr, pi.rs,
                                                          pi.nu, pi.nv, t, ti.dx, ti.dy, delta, S,
                                                          Z);
    else
      take(vjp_view_edge<ZS, T, FDK, EXACT, PROJ>(img, gimg, pout, pi.rs, pi.nu, pi.nv, t, ti.dx,
                                                  ti.dy, dcol, zlo, from));
  }
}

// The warp's reduce-scatter of the 12 sums of one (tile, view) into redv.
__device__ __forceinline__ void vjp_reduce(const TileIdx& ti, const float (&S)[3],
                                           const float (&Z)[3], float (&redv)[12]) {
  const int lane = threadIdx.x & 31;
  float v[16];
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    v[4 * r + 0] = ti.dx * S[r];
    v[4 * r + 1] = ti.dy * S[r];
    v[4 * r + 2] = Z[r];
    v[4 * r + 3] = S[r];
  }
  v[12] = v[13] = v[14] = v[15] = 0.0f;
  const float tot = warp_reduce_scatter16(v, lane);
  const int slot = scatter_slot(lane);
  if (!(lane & 1) && slot < 12) redv[slot] = tot;
}

// Write the record of one (tile, view): fixed-order sum of the 8 warps'
// values (0 when the tile is off the detector: not live), plus the anchors (16
// consecutive threads, slot = 0 .. PSLOTS-1).
__device__ __forceinline__ void vjp_write_record(const TileView& t, bool live,
                                                 const float (*redv)[12], bool bad, int slot, int j,
                                                 int tile, int ntiles,
                                                 float* __restrict__ partials) {
  if (slot >= PSLOTS) return;
  float val = 0.0f;
  if (slot < 12) {
    if (live)
      for (int w = 0; w < NT / 32; ++w) val += redv[w][slot];
    if (bad) val = __int_as_float(0x7fc00000);
  } else if (slot == 12) {
    val = (float)t.au;
  } else if (slot == 13) {
    val = (float)t.av;
  }
  partials[((long long)j * ntiles + tile) * PSLOTS + slot] = val;
}

// Motion VJP (optionally fused with the data VJP).  Grid: (view chunk, tile),
// tiles fastest, so the CTAs resident at any time share a few views whose
// data and dL/dproj rows stay in L2.  Per tile the views of the chunk are
// processed in order through the staging pipe (STAGE), like the forward.  The
// warp that finishes a view last also sums the 8 warps' values and writes the
// view's record, before it refills the slot (so the next writers of the
// slot's red[] come after it).
//
// With the fused data VJP the tile's dL/dvol is also kept in shared memory
// ([z][y][x], row pitch TX + 1) for the line pass.
constexpr int DSM_BYTES = ZB_VJP * TY * (TX + 1) * 4;
constexpr int COL_BYTES = ZB_VJP * NT * 4;  // without the line pass
// (The staged exact derivative reads its column from registers only.)
template <bool EXACT, bool PROJ>
__host__ __device__ constexpr int column_bytes() {
  return EXACT ? 0 : PROJ ? DSM_BYTES : COL_BYTES;
}
template <typename G, int NS, bool EXACT, bool PROJ>
__host__ __device__ constexpr int vjp_smem_bytes() {
  return stage_smem_bytes<G, NS>() + column_bytes<EXACT, PROJ>();
}

// One work item of the VJP: views [item / ntiles * vchunk, + vchunk) of tile
// item % ntiles.  All threads of the CTA call it with the CTA's shared memory.
template <int ZB, int NS, typename T, bool FDK, bool EXACT, bool PROJ, int STAGE>
__device__ __forceinline__ void vjp_item(const float* __restrict__ dvol, const T* __restrict__ proj,
                                         const CUtensorMap* map, const ProjInfo& pi,
                                         const float2* __restrict__ grad,
                                         const ViewGeom* __restrict__ geom, const VolInfo& vi,
                                         float* __restrict__ partials, float* __restrict__ dproj,
                                         float* __restrict__ dblk, int vchunk, int item,
                                         TileView (*tvs)[batch_records<STAGE>()],
                                         float (*red)[NT / 32][12],
                                         StagePipe<NS>& pipe,
                                         unsigned char* dyn_smem) {
  using G = Geo<T, STAGE>;
  constexpr bool CONV = STAGE && StageGeom<G>::CONV;
  constexpr int SLOT = StageGeom<G>::BYTES, NB = batch_records<STAGE>();
  // steps per view; step idx is half idx % HALVES of view vbeg + idx / HALVES
  constexpr int HALVES = STAGE == STAGE_HALF ? 2 : 1, ZS = ZB / HALVES;
  static_assert(NB % HALVES == 0 && ZS % 2 == 0, "whole views per batch, whole pairs per half");
  unsigned char* slots = dyn_smem + StageGeom<G>::F_BYTES;
  float* dsm =
      reinterpret_cast<float*>(dyn_smem + (STAGE ? stage_smem_bytes<G, NS>() : 0));
  constexpr int HALO = EXACT ? 0 : 1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int ntiles = vi.tiles_x * vi.tiles_y * vi.tiles_z;
  const int tile = item % ntiles;
  const int vbeg = (item / ntiles) * vchunk, vend = min(pi.nviews, vbeg + vchunk);
  const TileIdx ti = tile_index<ZB>(vi, tile);
  const int i = ti.tx * TX + ti.lx, j = ti.ty * TY + ti.ly;
  float delta[ZB];
  bool nz = false, finite = true;
#pragma unroll
  for (int k = 0; k < ZB; ++k) {
    const int z = ti.tz * ZB + k;
    delta[k] = (i < vi.nx && j < vi.ny && z < vi.nz)
                   ? __ldg(dvol + ((long long)z * vi.ny + j) * vi.nx + i)
                   : 0.0f;
    nz |= delta[k] != 0.0f;
    finite = finite && fabsf(delta[k]) <= 3.402823466e38f;
  }
  finite = __all_sync(0xffffffffu, finite);
  float* dcol = dsm + delta_base<PROJ>(ti.lx, ti.ly);  // this thread's column
  if (!EXACT || STAGE == STAGE_NONE) {
#pragma unroll
    for (int k = 0; k < ZB; ++k) dcol[delta_off<PROJ>(k)] = delta[k];
  }
  const int nvw = vend - vbeg, nst = nvw * HALVES, nbatch = (nst + NB - 1) / NB;
  if (!__syncthreads_or(nz)) {  // no upstream gradient in this tile: zero records
    for (int e = threadIdx.x; e < nvw * PSLOTS; e += NT)
      partials[((long long)(vbeg + e / PSLOTS) * ntiles + tile) * PSLOTS + e % PSLOTS] = 0.0f;
    return;
  }
  // Where the records are made decides how many registers spill: at one place inside the
  // loop with two slots (at three places 9.62 against 9.34 ms for the 256^3 x 248 motion
  // VJP), before it and inside without staging (2.28 against 2.17 ms for 128^3 x 200 at
  // 4.8 px per voxel) and with four slots, which have registers to spare (32^3 x 60 motion
  // 47.2 against 45.4 us).
  constexpr bool BEFORE = STAGE == STAGE_NONE || NS > VJP_NS;
  auto setup = [&](int k) {  // the records of batch k
    auto records = [&](const TileIdx& box) {
      setup_batch<G, STAGE != STAGE_NONE, HALVES, EXACT>(
          tvs[k & 1], geom, vbeg + k * (NB / HALVES), min(NB, nst - k * NB), box, pi.nu, pi.nv,
          HALO, pi.seq != 0);
    };
    // (the box again, not kept over the sample loop: no spills in the motion kernel,
    // 9.34 against 9.19 ms; the fused one has them elsewhere, and more with it)
    if constexpr (PROJ || EXACT || BEFORE) records(ti);
    else records(tile_index<ZB>(vi, tile));
  };
  // the record of step x's view (x is the view's last step)
  auto record = [&](int x, bool bad) {
    const TileView* q = tvs[(x / NB) & 1] + x % NB;
    bool live = q->mode != MODE_SKIP;
    if (HALVES == 2) live = live || q[-1].mode != MODE_SKIP;
    vjp_write_record(*q, live, red[x % NS], bad, lane, vbeg + x / HALVES, tile, ntiles, partials);
  };
  if constexpr (BEFORE) {
#pragma unroll 1
    for (int k = 0; k < min(2, nbatch); ++k) setup(k);
    __syncthreads();
    if (STAGE && warp < NS && warp < nst)
      stage_issue<G>(slots + warp * SLOT, map, tvs[0][warp], vbeg + warp / HALVES,
                     &pipe.full[warp]);
  }
  bool bad = false;
  PipePos<NS> pos;
  float S[3], Z[3];
  for (int idx = 0; idx < nst; ++idx) {
    const int v = vbeg + idx / HALVES, half = idx % HALVES, k = idx / NB, b = idx - k * NB;
    if (b == 0 && (!BEFORE || k >= 1)) {
      if (k >= 1) {
        __syncthreads();  // every warp is done with batch k-1, its records are written
        if (CONV && warp == 0) record(idx - 1, bad);  // (the barrier path writes them one late)
        if (CONV) __syncthreads();
      }
#pragma unroll 1
      for (int q = k ? k + 1 : 0; q <= k + 1 && q < nbatch; ++q) setup(q);
      __syncthreads();
      if (STAGE && !BEFORE && k == 0 && warp < NS && warp < nst)
        stage_issue<G>(slots + warp * SLOT, map, tvs[0][warp], vbeg + warp / HALVES,
                       &pipe.full[warp]);
    }
    const TileView& t = tvs[k & 1][b];
    const unsigned slot = pos.slot;
    unsigned char* buf = slots + slot * SLOT;
    if (STAGE && !bad) {  // (the lanes poll on their own; with CONV the CTA votes below)
      const bool ok = mbar_wait(&pipe.full[slot], pos.parity);
      bad = CONV ? !ok : !__all_sync(0xffffffffu, ok);
    }
    pos.next();
    const int in = idx + NS;
    const TileView& tn = tvs[(in / NB) & 1][in % NB];
    if constexpr (CONV) {
      // every warp has seen this phase and is done with F and step idx-1
      bad = __syncthreads_or(bad);
      if (b > 0 && half == 0 && warp == ((idx + 4) & 7)) record(idx - 1, bad);
      if (t.staged) {
        convert_stage<T, G>(reinterpret_cast<float*>(dyn_smem), reinterpret_cast<const T*>(buf), t);
        __syncthreads();  // F holds this step's footprint; the raw slot is free
      }
      if (warp == (idx & 7) && in < nst && !bad)
        stage_issue<G>(buf, map, tn, vbeg + in / HALVES, &pipe.full[slot]);
    }
    if (half == 0) {
#pragma unroll
      for (int r = 0; r < 3; ++r) S[r] = Z[r] = 0.0f;
    }
    if (t.mode != MODE_SKIP) {
      const T* img = proj + (long long)v * pi.vs;
      const float2* gimg = EXACT ? nullptr : grad + (long long)v * pi.nv * pi.nu;
      float* pout = PROJ ? dproj + (long long)v * pi.nv * pi.nu : nullptr;
      float* qout =
          PROJ && dblk ? dblk + (long long)v * 4 * pi.nv * pi.nu : nullptr;
      vjp_tile_view<ZB, ZS, NS, T, FDK, EXACT, PROJ, STAGE>(
          img, gimg, smem_addr(CONV ? dyn_smem : buf), STAGE && t.staged, pout, qout, pi, t, ti,
          half * ZS - 0.5f * (ZB - 1), delta, dcol + delta_off<PROJ>(half * ZS), finite, dsm, S, Z);
      if (HALVES == 1) vjp_reduce(ti, S, Z, red[slot][warp]);
    }
    if (HALVES == 2 && half == 1) vjp_reduce(ti, S, Z, red[slot][warp]);
    if constexpr (!CONV) {
      if (!STAGE) __syncthreads();  // no pipe to keep the warps within two views
      if (STAGE && bad) {
        if (half == HALVES - 1) record(idx, true);
      } else if (last_warp(&pipe.done[slot])) {
        if (half == HALVES - 1) record(idx, false);
        __syncwarp();
        if (STAGE && in < nst)
          stage_issue<G>(buf, map, tn, vbeg + in / HALVES, &pipe.full[slot]);
      }
    }
  }
  if (CONV) {
    __syncthreads();
    if (warp == 0) record(nst - 1, bad);
  }
  if (STAGE && bad) pipe_drain(pipe);
}

template <int ZB, int NS, typename T, bool FDK, bool EXACT, bool PROJ, int STAGE>
__global__ void __launch_bounds__(NT, NS > VJP_NS ? 2 : VJP_MINB)
    vjp_motion_kernel(const float* __restrict__ dvol, const T* __restrict__ proj,
                      const __grid_constant__ CUtensorMap map, ProjInfo pi,
                      const float2* __restrict__ grad, const ViewGeom* __restrict__ geom,
                      VolInfo vi, float* __restrict__ partials, float* __restrict__ dproj,
                      float* __restrict__ dblk, int vchunk, const int* __restrict__ wide) {
  if (wide) {  // are all views of the chunk (at most 32) wide?
    const int j = blockIdx.x / (vi.tiles_x * vi.tiles_y * vi.tiles_z) * vchunk + (threadIdx.x & 31);
    const bool w = (int)(threadIdx.x & 31) >= vchunk || j >= pi.nviews || wide[j] != 0;
    if (__all_sync(0xffffffffu, w) == (STAGE != STAGE_NONE)) return;  // the other's launch
  }
  __shared__ TileView tvs[2][batch_records<STAGE>()];
  __shared__ float red[NS][NT / 32][12];
  __shared__ StagePipe<NS> pipe;
  extern __shared__ __align__(128) unsigned char dyn_smem[];
  pipe_init(pipe);
  vjp_item<ZB, NS, T, FDK, EXACT, PROJ, STAGE>(dvol, proj, &map, pi, grad, geom, vi, partials, dproj,
                                           dblk, vchunk, blockIdx.x, tvs, red, pipe, dyn_smem);
}

// Items up to which the VJP runs two CTAs per SM with four staging slots.
constexpr int VJP_FEW = 304, VJP_NS_FEW = 4;

template <int NS, typename T, bool FDK, bool EXACT, bool PROJ, int STAGE>
static cudaError_t vjp_launch(const float* dvol, const void* proj, const CUtensorMap& map,
                              const ProjInfo& pi,
                              const float2* grad, const ViewGeom* geom, const VolInfo& vi,
                              float* partials, float* dproj, float* blk, int vc,
                              unsigned nblocks, const int* wide, cudaStream_t s) {
  const int smem =
      STAGE ? vjp_smem_bytes<Geo<T, STAGE>, NS, EXACT, PROJ>() : column_bytes<false, PROJ>();
  if (STAGE) {
    const cudaError_t e =
        smem_attr_once<vjp_motion_kernel<ZB_VJP, NS, T, FDK, EXACT, PROJ, STAGE>>(smem);
    if (e != cudaSuccess) return e;
  }
  vjp_motion_kernel<ZB_VJP, NS, T, FDK, EXACT, PROJ, STAGE><<<nblocks, NT, smem, s>>>(
      dvol, (const T*)proj, map, pi, grad, geom, vi, partials, dproj, blk, vc, wide);
  return cudaGetLastError();
}

template <typename T, bool FDK, bool EXACT, bool PROJ>
cudaError_t vjp_variants(const float* dvol, const void* proj, const ProjInfo& pi,
                                const float2* grad, const ViewGeom* geom, const VolInfo& vi,
                                float* partials, float* dproj, float* blk, int vc,
                                unsigned nblocks, const int* wide, cudaStream_t s,
                                const RawStack* raw) {
  CUtensorMap map{};
  if constexpr (!EXACT && !PROJ) {
    if (wide == WIDE_HALF && stageable<T>(proj, pi) &&
        make_stage_map(proj, dtype_id<T>(), pi, &map, true) == cudaSuccess)
      return vjp_launch<VJP_NS, T, FDK, EXACT, PROJ, STAGE_HALF>(
          dvol, proj, map, pi, grad, geom, vi, partials, dproj, blk, vc, nblocks, nullptr, s);
  }
  const bool stage = stageable<T>(proj, pi) && wide != WIDE_ALL && wide != WIDE_HALF &&
                     make_stage_map(proj, dtype_id<T>(), pi, &map, false) == cudaSuccess;
  const int* sel = stage ? wide : nullptr;
  if (stage) {
    const cudaError_t e =
        nblocks <= (unsigned)VJP_FEW
            ? vjp_launch<VJP_NS_FEW, T, FDK, EXACT, PROJ, STAGE_TILE>(
                  dvol, proj, map, pi, grad, geom, vi, partials, dproj, blk, vc, nblocks, sel, s)
            : vjp_launch<VJP_NS, T, FDK, EXACT, PROJ, STAGE_TILE>(
                  dvol, proj, map, pi, grad, geom, vi, partials, dproj, blk, vc, nblocks, sel, s);
    if (e != cudaSuccess || !sel) return e;
  }
  return vjp_launch<VJP_NS, T, FDK, EXACT, PROJ, STAGE_NONE>(
      dvol, raw ? raw->proj : proj, map, raw ? raw->pi : pi, grad, geom, vi, partials, dproj, nullptr,
      vc, nblocks, sel, s);
}

template <typename T, bool FDK, bool EXACT>
cudaError_t prepare_vjp_t() {
  cudaError_t e = smem_attr_once<vjp_motion_kernel<ZB_VJP, VJP_NS, T, FDK, EXACT, false,
                                                   STAGE_TILE>>(vjp_smem_bytes<T, VJP_NS, EXACT, false>());
  if constexpr (!EXACT) {
    if (e == cudaSuccess)
      e = smem_attr_once<vjp_motion_kernel<ZB_VJP, VJP_NS, T, FDK, EXACT, false, STAGE_HALF>>(
          vjp_smem_bytes<Half<T>, VJP_NS, EXACT, false>());
  }
  if (e == cudaSuccess)
    e = smem_attr_once<vjp_motion_kernel<ZB_VJP, VJP_NS_FEW, T, FDK, EXACT, false, STAGE_TILE>>(
        vjp_smem_bytes<T, VJP_NS_FEW, EXACT, false>());
  return e;
}

#define BP_VJP_VARIANT(T, FDK, EXACT, PROJ)                                                       \
  template cudaError_t vjp_variants<T, FDK, EXACT, PROJ>(                                         \
      const float*, const void*, const ProjInfo&, const float2*, const ViewGeom*, const VolInfo&, \
      float*, float*, float*, int, unsigned, const int*, cudaStream_t, const RawStack*);
#define BP_VJP_VARIANTS(EXACT, PROJ)            \
  BP_VJP_VARIANT(float, false, EXACT, PROJ)     \
  BP_VJP_VARIANT(float, true, EXACT, PROJ)      \
  BP_VJP_VARIANT(__half, false, EXACT, PROJ)    \
  BP_VJP_VARIANT(__half, true, EXACT, PROJ)     \
  BP_VJP_VARIANT(__nv_bfloat16, false, EXACT, PROJ) \
  BP_VJP_VARIANT(__nv_bfloat16, true, EXACT, PROJ)
#define BP_VJP_PREPARE(EXACT)                                      \
  template cudaError_t prepare_vjp_t<float, false, EXACT>();       \
  template cudaError_t prepare_vjp_t<float, true, EXACT>();        \
  template cudaError_t prepare_vjp_t<__half, false, EXACT>();      \
  template cudaError_t prepare_vjp_t<__half, true, EXACT>();       \
  template cudaError_t prepare_vjp_t<__nv_bfloat16, false, EXACT>(); \
  template cudaError_t prepare_vjp_t<__nv_bfloat16, true, EXACT>();

}  // namespace bpk
