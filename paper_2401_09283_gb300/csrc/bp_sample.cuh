// What the forward (bp_forward.cu), the motion VJP (bp_vjp.cuh) and the data VJP
// (bp_project.cu) share: packed arithmetic, the tile records, the staging of footprints
// and the taps.
#pragma once

#include "bp_internal.cuh"
#include "bp_plan.h"
#include "bp_tma.cuh"

namespace bpk {

// CTAs per SM the register budget is sized for (256 threads each).
constexpr int FWD_MINB = 4;
constexpr int VJP_MINB = 3;
// Staging slots (three at three CTAs per SM in the forward, three or four at
// two in the VJP: slower, 3.69 against 3.58 and 10.9 against 9.9 ms on c2; three at
// the same occupancy, in buffers of 76 x 56 pixels and batches of 16 views: 3.49
// against 3.45 and 9.62 against 9.46).
constexpr int FWD_NS = 2;
constexpr int VJP_NS = 2;

constexpr float MAGIC = 12582912.0f;   // 1.5 * 2^23
constexpr int MAGIC_BITS = 0x4B400000;
// Staged byte addresses are computed as subnormal floats: a float whose value is
// n 2^-149 (0 <= n < 2^23) has the bit pattern n, and sums and products of such
// values are exact.  One pixel is four bytes, 2^-147.
#define BP_PIXEL 5.60519385729926828e-45f

// Footprint staging buffers: 64 rows at a fixed row pitch P (elements), so tap
// offsets are immediates, filled by TMA in boxes of P x 8 pixels.  FP32
// footprints are sampled in place (pitch 84; 80 measured the same).  FP16 and
// BF16 footprints arrive raw (pitch 80; 88 bank-conflicts more, 30.8 against
// 30.5 ms for a 384^3 x 248 VJP) and are converted once per (tile, view) into an
// FP32 buffer of the same pitch, which the sample loops read like FP32 data.
constexpr int BOX_ROWS = 8;
template <typename G>
struct StageGeom {
  static constexpr bool CONV = sizeof(G) != 4;                 // converted to FP32
  static constexpr int CH = 16 / (int)sizeof(G);               // elements per 16 bytes
  static constexpr int P = CONV ? 80 : 84;                     // row pitch in elements
  static constexpr int ROWS = 64;
  static constexpr int BOX_BYTES = P * BOX_ROWS * (int)sizeof(G);
  static constexpr int BYTES = P * ROWS * (int)sizeof(G);      // one footprint buffer
  static constexpr int F_BYTES = CONV ? P * ROWS * 4 : 0;      // converted footprint
};
// Buffers of half tiles (16 x 16 x 8 voxels), for scans of 4 to 5 pixels per voxel,
// whose whole tiles project wider and higher than the buffers above.  116 floats:
// 93 % of the half tiles of a 128^3 volume at 4.8 px per voxel fit (108 wide 80 %,
// 48 rows 77 %), four CTAs per SM, and as few bank conflicts as 84 (124 has more).
template <typename T>
struct Half {};
template <typename T>
struct StageGeom<Half<T>> {
  static constexpr bool CONV = sizeof(T) != 4;
  static constexpr int CH = 16 / (int)sizeof(T);
  static constexpr int P = CONV ? 120 : 116;
  static constexpr int ROWS = 56;
  static constexpr int BOX_BYTES = P * BOX_ROWS * (int)sizeof(T);
  static constexpr int BYTES = P * ROWS * (int)sizeof(T);
  static constexpr int F_BYTES = CONV ? P * ROWS * 4 : 0;
};
template <typename G>
constexpr bool aligned_boxes() {  // TMA boxes land on 128-byte boundaries
  return StageGeom<G>::BOX_BYTES % 128 == 0 && StageGeom<G>::F_BYTES % 128 == 0;
}
static_assert(aligned_boxes<float>() && aligned_boxes<__half>() && aligned_boxes<Half<float>>() &&
                  aligned_boxes<Half<__half>>(),
              "TMA boxes land on 128-byte boundaries");

// How a kernel variant gets its footprints: from global memory, staged whole tiles,
// staged half tiles.
enum { STAGE_NONE = 0, STAGE_TILE = 1, STAGE_HALF = 2 };
template <typename T, int STAGE>
using Geo = std::conditional_t<STAGE == STAGE_HALF, Half<T>, T>;
// Records per batch of views (half tiles: two records per view in the VJP).
template <int STAGE>
__host__ __device__ constexpr int batch_records() {
  return STAGE == STAGE_HALF ? VB / 2 : VB;
}

template <typename T>
__device__ __forceinline__ float ldv(const T* p);
template <>
__device__ __forceinline__ float ldv<float>(const float* p) {
  return __ldg(p);
}
template <>
__device__ __forceinline__ float ldv<__half>(const __half* p) {
  return __half2float(__ldg(p));
}
template <>
__device__ __forceinline__ float ldv<__nv_bfloat16>(const __nv_bfloat16* p) {
  return __bfloat162float(__ldg(p));
}

__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Packed FP32 pairs (Blackwell f32x2 instructions): two voxels' values in
// one 64-bit register, one instruction per pair.  Each element is rounded
// exactly like the scalar instruction, so packed and scalar code give
// identical results; the packing halves the issue slots of the FP32 work.
typedef unsigned long long f2;

__device__ __forceinline__ f2 pk2(float lo, float hi) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void up2(f2 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 add2_rd(f2 a, f2 b) {  // rounded toward -inf
  f2 r;
  asm("add.rm.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// ------------------------------------------------------------ bounds check
// Debug builds (-DBP_BOUNDS_CHECK) check every staged, gathered and
// scattered index against the range it must lie in.  A failed check sets a
// bit in a device flag word (one per source file), records the first failure, and redirects the
// access to a safe in-range position (the result is then wrong but nothing
// outside the buffers is touched); the host reads the word through
// bp_bounds_check.  Release builds compile the checks out.
enum { BC_STAGED_TAP = 0, BC_GLOBAL_TAP = 1, BC_SCATTER = 2, BC_STAGE_DST = 3, BC_SELFTEST = 7 };
#ifdef BP_BOUNDS_CHECK
static __device__ unsigned int g_bc_flags;
static __device__ unsigned long long g_bc_first;
static __device__ int g_bc_lost_view = -1;  // the view whose footprints never arrive
static __device__ __noinline__ void bc_fail(unsigned code, int a, int b) {
  atomicOr(&g_bc_flags, 1u << code);
  const unsigned long long rec = (1ull << 63) | ((unsigned long long)code << 56) |
                                 ((unsigned long long)(a & 0x0fffffff) << 28) |
                                 (unsigned long long)(b & 0x0fffffff);
  atomicCAS(&g_bc_first, 0ull, rec);
}
static __global__ void bc_selftest_kernel() { bc_fail(BC_SELFTEST, 7, 9); }
#endif

static inline cudaError_t file_bounds_status(unsigned* flags, long long* first, int op, cudaStream_t s) {
#ifdef BP_BOUNDS_CHECK
  if (op == 2) {
    bc_selftest_kernel<<<1, 1, 0, s>>>();
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  if (op == 3) {
    const int v = (int)*first;
    return cudaMemcpyToSymbol(g_bc_lost_view, &v, sizeof(v));
  }
  cudaError_t e = cudaStreamSynchronize(s);
  unsigned long long f = 0;
  if (e == cudaSuccess) e = cudaMemcpyFromSymbol(flags, g_bc_flags, sizeof(unsigned));
  if (e == cudaSuccess) e = cudaMemcpyFromSymbol(&f, g_bc_first, sizeof(f));
  *first = (long long)(f & ~(1ull << 63)) | (f ? 0 : -1LL);
  if (e == cudaSuccess && op == 1) {
    const unsigned z = 0;
    const unsigned long long z64 = 0;
    e = cudaMemcpyToSymbol(g_bc_flags, &z, sizeof(z));
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_bc_first, &z64, sizeof(z64));
  }
  return e;
#else
  (void)flags;
  (void)first;
  (void)op;
  (void)s;
  return cudaErrorNotSupported;
#endif
}

// Unchecked global gathers and scatters (INTERIOR tiles) need both tap
// columns and rows on the detector.
__device__ __forceinline__ void bc_interior(int code, int& iu, int& iv, int nu, int nv) {
#ifdef BP_BOUNDS_CHECK
  if (!((unsigned)iu < (unsigned)(nu - 1) && (unsigned)iv < (unsigned)(nv - 1))) {
    bc_fail(code, iu, iv);
    iu = 0;
    iv = 0;
  }
#else
  (void)code;
  (void)iu;
  (void)iv;
  (void)nu;
  (void)nv;
#endif
}

// ------------------------------------------------------------ tile set-up

struct TileIdx {
  int tx, ty, tz, lx, ly;
  float dx, dy;
  double qc[3];
  float hx, hy, zlo, zhi;  // extent of the CTA's box about the tile centre
};

// zs: the CTA's slices of the tile, [zs * ZS, zs * ZS + ZS).
template <int ZB, int ZS = ZB>
__device__ __forceinline__ TileIdx tile_index(const VolInfo& vi, int tile, int zs = 0) {
  TileIdx ti;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  ti.lx = (warp & 1) * 8 + (lane & 7);
  ti.ly = (warp >> 1) * 4 + (lane >> 3);
  ti.tx = tile % vi.tiles_x;
  ti.ty = (tile / vi.tiles_x) % vi.tiles_y;
  ti.tz = tile / (vi.tiles_x * vi.tiles_y);
  ti.dx = ti.lx - 0.5f * (TX - 1);
  ti.dy = ti.ly - 0.5f * (TY - 1);
  ti.qc[0] = ti.tx * TX + 0.5 * (TX - 1) - vi.cx;
  ti.qc[1] = ti.ty * TY + 0.5 * (TY - 1) - vi.cy;
  ti.qc[2] = ti.tz * ZB + 0.5 * (ZB - 1) - vi.cz;
  ti.hx = 0.5f * (TX - 1);
  ti.hy = 0.5f * (TY - 1);
  ti.zlo = zs * ZS - 0.5f * (ZB - 1);
  ti.zhi = ti.zlo + (ZS - 1);
  return ti;
}

// Cooperative set-up of the records of views j0 .. j0+nb-1 (nb <= 32) for
// this CTA's box; whole warps call it.  Eight lanes serve one view; lane c
// evaluates box corner c, lanes 0-2 also one row each in FP64 (eight FP64
// instructions per warp, of 16 cycles each on an SM's FP64 pipe; all rows in every
// lane, with the conversions, were 32: 256^3 x 248 forward 3.59 -> 3.53 ms).  FP64
// is used only where the precision
// matters -- the projection (uc, vc, wc) of the tile centre and
// the anchored values U0 = uc - au wc, V0 = vc - av wc; the anchor pixel
// itself only has to be near the projection and comes from FP32.  The
// corners are evaluated in FP32 in the anchored frame (errors ~1e-5 px,
// far below the 0.01 px classification margin): u/w and v/w are
// linear-fractional in the voxel position, so over a box with w > 0 their
// extremes are at the corners, and the box is
//   SKIP      every sample is 0 (projection at or beyond -1 / n),
//   INTERIOR  every tap (floor and floor+1) lies on the detector,
//   EDGE      otherwise (clamped coordinates, checked taps)
// (plan_box, which also guards against boxes that come near the source plane).
// With STAGE, bounded boxes also get a staging plan: the rectangle of
// detector pixels that any tap (plus `halo` pixels each side) can read,
// NOT clipped to the detector (off-detector pixels are staged as zeros, so
// the sample loop needs neither checks nor clamps), if it fits the buffer.
// seq: no tile counts as central-safe (its sums are then taken sample by sample).
// With HALVES = 2 record b is the lower (even b) or upper half, in z, of the box in
// view j0 + b / 2 (whole views: j0 is of a lower half).
// EARLY: what the corners give goes to the record before the plan, which then needs
// fewer registers (the forward's call; inlined in the VJP it spilled more).
template <typename G, bool STAGE, int HALVES = 1, bool EARLY = false>
__device__ __forceinline__ void setup_batch(TileView* tvs, const ViewGeom* __restrict__ geom, int j0, int nb,
                            const TileIdx& ti, int nu, int nv, int halo = 0, bool seq = false) {
  const int b = threadIdx.x >> 3, c = threadIdx.x & 7;
  if ((int)(threadIdx.x >> 5) * 4 >= nb) return;  // a warp without a view
  const ViewGeom& g = geom[j0 + min(b, nb - 1) / HALVES];
  const float zmid = 0.5f * (ti.zlo + ti.zhi);
  const float zlo = HALVES == 2 && (b & 1) ? zmid + 0.5f : ti.zlo;
  const float zhi = HALVES == 2 && !(b & 1) ? zmid - 0.5f : ti.zhi;
  // lanes 0, 1, 2 of a view hold the rows u, v, w of the tile centre's projection
  const int row = min(c, 2);
  const double* M = g.P + 4 * row;
  const double pc = fma(M[0], ti.qc[0], fma(M[1], ti.qc[1], fma(M[2], ti.qc[2], M[3])));
  const float pf = (float)pc;
  const double wc = __shfl_sync(0xffffffffu, pc, 2, 8);
  const float wf = __shfl_sync(0xffffffffu, pf, 2, 8);
  int ar = 0;  // the row's anchor
  if (wc > 0.0 && c < 2)
    ar = (int)fminf(fmaxf(floorf(pf / wf), -1048576.0f), 1048576.0f);
  const int au = __shfl_sync(0xffffffffu, ar, 0, 8), av = __shfl_sync(0xffffffffu, ar, 1, 8);
  const float p0 = c < 2 ? (float)fma(-(double)ar, wc, pc) : pf;
  TileView t;
  t.U0 = __shfl_sync(0xffffffffu, p0, 0, 8);
  t.V0 = __shfl_sync(0xffffffffu, p0, 1, 8);
  t.W0 = wf;
  const float fau = (float)au, fav = (float)av;
  const float4 R0 = g.R[0], R1 = g.R[1], R2 = g.R[2];
  t.rw0 = R2.x;
  t.rw1 = R2.y;
  t.rw2 = R2.z;
  t.ru0 = fmaf(-fau, t.rw0, R0.x);
  t.ru1 = fmaf(-fau, t.rw1, R0.y);
  t.ru2 = fmaf(-fau, t.rw2, R0.z);
  t.rv0 = fmaf(-fav, t.rw0, R1.x);
  t.rv1 = fmaf(-fav, t.rw1, R1.y);
  t.rv2 = fmaf(-fav, t.rw2, R1.z);
  // this lane's corner
  const float d0 = (c & 1) ? ti.hx : -ti.hx;
  const float d1 = (c & 2) ? ti.hy : -ti.hy;
  const float d2 = (c & 4) ? zhi : zlo;
  const float w = fmaf(t.rw2, d2, fmaf(t.rw1, d1, fmaf(t.rw0, d0, t.W0)));
  const float u = fmaf(t.ru2, d2, fmaf(t.ru1, d1, fmaf(t.ru0, d0, t.U0)));
  const float v = fmaf(t.rv2, d2, fmaf(t.rv1, d1, fmaf(t.rv0, d0, t.V0)));
  t.au = au;
  t.av = av;
  t.wgt = R0.w;
  t.wgtd = R1.w;
  t.ic = 0.0f;
  t.mode = t.csafe = t.staged = t.sx0 = t.sv0 = t.sh = t.scpr = t.srpp = t.smag = t.soff = 0;
  const bool mine = c == 0 && b < nb;
  if (EARLY && mine) tvs[b] = t;
  const bool pos = in_front(w);
  int npos = pos ? 1 : 0;
  float xmin = INFINITY, xmax = -INFINITY, ymin = INFINITY, ymax = -INFINITY, wmin = w;
  if (pos) {
    xmin = xmax = u / w;
    ymin = ymax = v / w;
  }
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) {
    npos += __shfl_xor_sync(0xffffffffu, npos, o);
    wmin = fminf(wmin, __shfl_xor_sync(0xffffffffu, wmin, o));
    xmin = fminf(xmin, __shfl_xor_sync(0xffffffffu, xmin, o));
    xmax = fmaxf(xmax, __shfl_xor_sync(0xffffffffu, xmax, o));
    ymin = fminf(ymin, __shfl_xor_sync(0xffffffffu, ymin, o));
    ymax = fmaxf(ymax, __shfl_xor_sync(0xffffffffu, ymax, o));
  }
  if (!mine) return;
  constexpr int CH = StageGeom<G>::CH, P = StageGeom<G>::P;
  // w is linear: its extremes lie symmetrically about the box's centre
  const float wmax = 2.0f * fmaf(t.rw2, 0.5f * (zlo + zhi), t.W0) - wmin;
  const BoxRange q = {xmin, xmax, ymin, ymax, wmin, wmax, npos};
  const BoxPlan plan = plan_box(q, nu, nv, au, av, CH, P, STAGE ? StageGeom<G>::ROWS : 0, halo, seq);
  const int du = au - plan.sx0, dv = av - plan.sv0;
  TileView& o = EARLY ? tvs[b] : t;
  o.mode = plan.mode;
  o.csafe = plan.csafe;
  o.staged = plan.staged;
  if (STAGE && plan.staged) {
    o.sx0 = plan.sx0;
    o.sv0 = plan.sv0;
    o.sh = plan.sh;
    o.scpr = plan.scpr;
    o.srpp = 32 / plan.scpr;
    o.smag = (65536 + plan.scpr - 1) / plan.scpr;
    o.soff = (int)((unsigned)dv * (unsigned)P - (unsigned)MAGIC_BITS * (unsigned)P + (unsigned)du -
                   (unsigned)MAGIC_BITS);
    o.ic = (float)(dv * P + du);
  }
  if (!EARLY) tvs[b] = t;
}

// The same as a call, for the forward: inlined, at three places or at one, it took
// registers from the sample loop (3.26 against 3.41 to 3.55 ms on 256^3 x 248).  The VJP
// inlines it at one place (bp_vjp.cuh).
template <typename G, bool STAGE>
__device__ __noinline__ void setup_batch_call(TileView* tvs, const ViewGeom* __restrict__ geom,
                                              int j0, int nb, const TileIdx& ti, int nu, int nv) {
  setup_batch<G, STAGE, 1, STAGE>(tvs, geom, j0, nb, ti, nu, nv);
}

// Detector position of one voxel in the anchored frame.
struct Sample {
  float rwi;     // 1/w
  float x, y;    // u/w - au, v/w - av (clamped in EDGE mode)
  float tu, tv;  // fractional parts
  int iu, iv;    // absolute floor pixel
  int bx, by;    // bit patterns of x + MAGIC, y + MAGIC (rounded down)
  bool ok;       // w > 0
};

template <bool EDGE>
__device__ __forceinline__ Sample locate(float u, float v, float w, const TileView& t, int nu,
                                         int nv) {
  Sample s;
  s.ok = true;
  if (EDGE) s.ok = w > 1e-20f;  // a voxel at (or behind) the source plane contributes nothing
  s.rwi = rcp_approx(w);
  float x = u * s.rwi, y = v * s.rwi;
  if (EDGE) {
    // Clamp far-off coordinates into (-2, -1) or (n, n+1): all four taps are
    // then outside the detector, so value and derivatives are 0 there (a
    // clamp to exactly -1 would sit on the kink of the zero-padded
    // interpolant, where the exact derivative is d[0], not 0).
    x = fminf(fmaxf(x, -1.5f - (float)t.au), (float)nu + 0.5f - (float)t.au);
    y = fminf(fmaxf(y, -1.5f - (float)t.av), (float)nv + 0.5f - (float)t.av);
  }
  float rx = __fadd_rd(x, MAGIC), ry = __fadd_rd(y, MAGIC);
  s.tu = x - (rx - MAGIC);
  s.tv = y - (ry - MAGIC);
  s.bx = __float_as_int(rx);
  s.by = __float_as_int(ry);
  s.iu = s.bx - MAGIC_BITS + t.au;
  s.iv = s.by - MAGIC_BITS + t.av;
  s.x = x;
  s.y = y;
  return s;
}

// Four taps of a [nv][rs] image at (iu..iu+1, iv..iv+1), zero outside.
template <bool EDGE, typename T>
__device__ __forceinline__ void taps(const T* img, long long rs, int nu, int nv, const Sample& s,
                                     float& d00, float& d10, float& d01, float& d11) {
  if (!EDGE) {
    int iu = s.iu, iv = s.iv;
    bc_interior(BC_GLOBAL_TAP, iu, iv, nu, nv);
    const T* p = img + (long long)iv * rs + iu;
    d00 = ldv(p);
    d10 = ldv(p + 1);
    d01 = ldv(p + rs);
    d11 = ldv(p + rs + 1);
  } else {
    bool u0 = (unsigned)s.iu < (unsigned)nu, u1 = (unsigned)(s.iu + 1) < (unsigned)nu;
    bool v0 = (unsigned)s.iv < (unsigned)nv, v1 = (unsigned)(s.iv + 1) < (unsigned)nv;
    const T* p = img + (long long)s.iv * rs + s.iu;
    d00 = (u0 && v0 && s.ok) ? ldv(p) : 0.0f;
    d10 = (u1 && v0 && s.ok) ? ldv(p + 1) : 0.0f;
    d01 = (u0 && v1 && s.ok) ? ldv(p + rs) : 0.0f;
    d11 = (u1 && v1 && s.ok) ? ldv(p + rs + 1) : 0.0f;
  }
}

__device__ __forceinline__ float bilerp(float tu, float tv, float d00, float d10, float d01,
                                        float d11) {
  float top = fmaf(tu, d10 - d00, d00);
  float bot = fmaf(tu, d11 - d01, d01);
  return fmaf(tv, bot - top, top);
}

__device__ __forceinline__ f2 bilerp2(f2 tu, f2 tv, f2 d00, f2 d10, f2 d01, f2 d11) {
  const f2 top = fma2(tu, sub2(d10, d00), d00);
  const f2 bot = fma2(tu, sub2(d11, d01), d01);
  return fma2(tv, sub2(bot, top), top);
}

// ------------------------------------------------------ footprint staging

// Each (tile, view) reads a small rectangle of one detector image (the tile
// footprint from the set-up).  Voxels project ~2.6 px apart on the larger
// detectors, so a warp's 32 taps of one load are scattered over 4-6 L1
// lines; from shared memory the same taps are a single wavefront (bar bank
// conflicts).  The footprint is therefore copied to shared memory by TMA, in
// boxes of P x 8 pixels (pixels off the detector arrive as zeros), two views
// ahead: one warp issues at most eight copies per view, where a cp.async copy
// by all threads cost ~50 of the ~540 instructions of a (thread, view) and two
// CTA barriers.  Footprints that do not fit the buffer, or are unbounded,
// read global memory instead.

// NS staging slots, used by consecutive views in turn.  full[s] completes once
// per view (when its footprint has arrived, at once if it has none); done[s]
// counts the warps that have finished the view, and the warp that finishes
// last refills the slot, so no warp waits for another one to free a slot.
// Every warp waits on full[s] for every view, staged or not: it may then be at
// most one phase behind, which the parity tells apart.
//
// A warp whose wait runs out (a copy that never arrives; in any lane) is bad: it no longer counts
// itself as finished, so that no slot is refilled from that step on and the other warps
// run out of time too, where they need more; what it computes from there on shows as
// NaN; and it stays for the copies that may still be in flight (pipe_drain).
template <int NS>
struct StagePipe {
  unsigned long long full[NS];
  unsigned done[NS];
};

template <int NS>
__device__ __forceinline__ void pipe_init(StagePipe<NS>& p) {  // ends with a CTA barrier
  if (threadIdx.x < NS) {
    mbar_init(&p.full[threadIdx.x], 1);
    p.done[threadIdx.x] = 0u;
    mbar_init_fence();
  }
  __syncthreads();
}

// A warp's place in the pipe: the slot of its current view and the parity of
// that slot's phase.
template <int NS>
struct PipePos {
  unsigned slot = 0, parity = 0;
  __device__ __forceinline__ void next() {
    if (++slot == NS) {
      slot = 0;
      parity ^= 1u;
    }
  }
};

// A bad warp, before it ends: give the copies in flight the same time again, so that none
// lands in shared memory that another CTA has been given.  (Of a slot's two parities one
// is that of a finished phase, whose wait returns at once.)
template <int NS>
__device__ __forceinline__ void pipe_drain(StagePipe<NS>& p) {
#pragma unroll 1
  for (int k = 0; k < 2 * NS; ++k) mbar_wait(&p.full[k / 2], k & 1);
}

// One whole warp: request the footprint of record t (view v) into buf.
template <typename G>
__device__ __forceinline__ void stage_issue(unsigned char* buf, const CUtensorMap* map,
                                            const TileView& t, int v, unsigned long long* bar) {
  constexpr int BOX = StageGeom<G>::BOX_BYTES;
  const int lane = threadIdx.x & 31;
  int nb = t.staged ? (t.sh + BOX_ROWS - 1) / BOX_ROWS : 0;
#ifdef BP_BOUNDS_CHECK
  if ((unsigned)nb > StageGeom<G>::ROWS / BOX_ROWS || (t.sx0 & (StageGeom<G>::CH - 1))) {
    if (lane == 0) bc_fail(BC_STAGE_DST, t.sh, t.sx0);
    nb = 0;
  }
  if (nb && v == g_bc_lost_view) {  // announced, never copied
    if (lane == 0) mbar_arrive_expect(bar, (unsigned)(nb * BOX));
    return;
  }
#endif
  if (lane == 0) {
    if (nb) mbar_arrive_expect(bar, (unsigned)(nb * BOX));
    else mbar_arrive(bar);
  }
  __syncwarp();
  if (lane < nb) tma_load_3d(buf + lane * BOX, map, t.sx0, t.sv0 + lane * BOX_ROWS, v, bar);
}

// Whether the calling warp is the last of the CTA's warps to finish with a
// slot.  Acquire-release: the last warp sees what every other warp wrote
// before, and its refill comes after all their reads (lane 0 acquires, the second
// __syncwarp hands that on: a shuffle orders no memory).
__device__ __forceinline__ bool last_warp(unsigned* done) {
  __syncwarp();
  unsigned old = 0;
  if ((threadIdx.x & 31) == 0)
    asm volatile("atom.acq_rel.cta.shared::cta.inc.u32 %0, [%1], %2;"
                 : "=r"(old)
                 : "r"(smem_addr(done)), "r"(NT / 32 - 1)
                 : "memory");
  const bool last = __shfl_sync(0xffffffffu, old, 0) == NT / 32 - 1;
  __syncwarp();
  return last;
}

// All threads: convert the raw FP16/BF16 rectangle of record t (staged by
// stage_issue<T>) into FP32 at the same pitch, in 16-byte chunks, rows per warp
// pass (no divisions).
template <typename T, typename G>
__device__ __forceinline__ void convert_stage(float* F, const T* R, const TileView& t) {
  constexpr int CONV_P = StageGeom<G>::P;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int lr = (lane * t.smag) >> 16, lc = lane - lr * t.scpr;
  if (lr >= t.srpp) return;
  for (int r = warp * t.srpp + lr; r < t.sh; r += (NT / 32) * t.srpp) {
    const uint4 w = *reinterpret_cast<const uint4*>(R + r * CONV_P + lc * 8);
    const unsigned ws[4] = {w.x, w.y, w.z, w.w};
    float f[8];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if constexpr (std::is_same<T, __half>::value) {
        const float2 v = __half22float2(*reinterpret_cast<const __half2*>(&ws[q]));
        f[2 * q] = v.x;
        f[2 * q + 1] = v.y;
      } else {
        f[2 * q] = __uint_as_float(ws[q] << 16);
        f[2 * q + 1] = __uint_as_float(ws[q] & 0xffff0000u);
      }
    }
    float4* d = reinterpret_cast<float4*>(F + r * CONV_P + lc * 8);
    d[0] = make_float4(f[0], f[1], f[2], f[3]);
    d[1] = make_float4(f[4], f[5], f[6], f[7]);
  }
}

// Sampling of the staged FP32 footprint.  buf is its shared-memory address, P
// the row pitch, H the stencil's reach beyond the bilinear taps (1 for the
// CENTRAL 4x4-minus-corners stencil, 0 otherwise; the staging plan covers it).

template <int OFF>  // OFF in floats
__device__ __forceinline__ float lds(unsigned a) {
  float r;
  asm volatile("ld.shared.f32 %0, [%1+%2];" : "=f"(r) : "r"(a), "n"(OFF * 4));
  return r;
}
template <int OFF>
__device__ __forceinline__ f2 lds2(unsigned a, unsigned b) {
  const float lo = lds<OFF>(a), hi = lds<OFF>(b);
  return pk2(lo, hi);
}

#ifdef BP_BOUNDS_CHECK
// Column and row of the floor pixel in the staged rectangle; true if bad.
template <typename G, int H>
__device__ __forceinline__ bool bc_staged(const TileView& t, int fx, int fy) {
  const int ru = fx + t.au - t.sx0, rv = fy + t.av - t.sv0;
  if (t.staged && ru - H >= 0 && ru + 1 + H < t.scpr * StageGeom<G>::CH && rv - H >= 0 &&
      rv + 1 + H < t.sh)
    return false;
  bc_fail(BC_STAGED_TAP, ru, rv);
  return true;
}
#endif

// Address of one sample's floor pixel: (bx, by) are the bit patterns of
// x + MAGIC and y + MAGIC rounded down, i.e. MAGIC_BITS + floor.
template <typename G, int H>
__device__ __forceinline__ unsigned staged_tap(unsigned buf, const TileView& t, int bx, int by) {
  constexpr int P = StageGeom<G>::P;
#ifdef BP_BOUNDS_CHECK
  if (bc_staged<G, H>(t, bx - MAGIC_BITS, by - MAGIC_BITS)) {
    bx = MAGIC_BITS + t.sx0 + H - t.au;
    by = MAGIC_BITS + t.sv0 + H - t.av;
  }
#endif
  const unsigned o = (unsigned)by * (unsigned)P + (unsigned)bx + (unsigned)t.soff;
  return buf + 4u * o;
}

// Address of the anchor pixel in the footprint at buf (it may lie outside it, even
// before it), as the subnormal float of staged_pair.
__device__ __forceinline__ f2 staged_anchor(unsigned buf, const TileView& t) {
  const float a = fmaf(t.ic, BP_PIXEL, __uint_as_float(buf));
  return pk2(a, a);
}

// Addresses of a pair of samples' floor pixels from their floors (fx, fy) as floats
// and the anchor's: two packed FMAs whose results' bit patterns are the addresses.
// (Index arithmetic on the floor bits took four to six integer instructions, a sum
// around 1.5 * 2^21 still one per sample to take the magic number out and the buffer
// in: 256^3 x 248 forward 3.52 -> 3.43 ms, motion VJP 9.60 -> 9.39, a BF16 384^3 x 248
// VJP 30.2 -> 29.3, with the two packed operations less in the VJP's loop.)
template <typename G, int H>
__device__ __forceinline__ void staged_pair(unsigned buf, const TileView& t, f2 ic, f2 fx, f2 fy,
                                            unsigned& al, unsigned& ah) {
  constexpr float P = (float)StageGeom<G>::P;
  const f2 o = fma2(fy, pk2(P * BP_PIXEL, P * BP_PIXEL), fma2(fx, pk2(BP_PIXEL, BP_PIXEL), ic));
  float lo, hi;
  up2(o, lo, hi);
  al = __float_as_uint(lo);
  ah = __float_as_uint(hi);
#ifdef BP_BOUNDS_CHECK
  float xl, xh, yl, yh;
  up2(fx, xl, xh);
  up2(fy, yl, yh);
  const unsigned safe = buf + 4u * (unsigned)(H * StageGeom<G>::P + H);
  if (bc_staged<G, H>(t, (int)xl, (int)yl)) al = safe;
  if (bc_staged<G, H>(t, (int)xh, (int)yh)) ah = safe;
  // the address must also be the one that integer arithmetic gives
  const unsigned rl = buf + 4u * (unsigned)(((int)yl + t.av - t.sv0) * StageGeom<G>::P + (int)xl +
                                            t.au - t.sx0);
  const unsigned rh = buf + 4u * (unsigned)(((int)yh + t.av - t.sv0) * StageGeom<G>::P + (int)xh +
                                            t.au - t.sx0);
  if (al != safe && al != rl) { bc_fail(BC_STAGED_TAP, (int)al, (int)rl); al = safe; }
  if (ah != safe && ah != rh) { bc_fail(BC_STAGED_TAP, (int)ah, (int)rh); ah = safe; }
#else
  (void)buf;
  (void)t;
#endif
}

template <typename G, int NS>
__host__ __device__ constexpr int stage_smem_bytes() {
  return StageGeom<G>::F_BYTES + NS * StageGeom<G>::BYTES;
}

template <typename T>
static bool stageable(const void* proj, const ProjInfo& pi) {
  return stage_aligned(proj, sizeof(T) == 4 ? 0 : 1, pi);
}

// Opt a kernel into more than 48 KiB of dynamic shared memory, once per
// device (so that later launches -- including ones being captured into a
// CUDA graph -- make no attribute call).
template <auto Kernel>
static cudaError_t smem_attr_once(int bytes) {
  static int done[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return cudaGetLastError();
  if (dev >= 0 && dev < 64 && done[dev]) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev] = 1;
  return e;
}

template <typename T>
constexpr int dtype_id() {
  return std::is_same<T, float>::value ? 0 : std::is_same<T, __half>::value ? 1 : 2;
}

}  // namespace bpk
