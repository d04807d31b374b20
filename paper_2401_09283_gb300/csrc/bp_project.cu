// Voxel-driven kernels of the backprojection (Eq. 3) and its vector-Jacobian
// products (Eqs. 4-5) for sm_103a.
//
// Work decomposition: a CTA of 256 threads owns a 16 x 16 x ZB box of voxels
// (one z-column of ZB voxels per thread, warps of 8 x 4 columns) and loops
// over views.  For each batch of 32 views eight threads per view compute, in
// FP64 where it matters, the anchored per-tile view record (TileView): the
// integer pixel nearest the projection of the tile centre, the anchored rows and
// the classification of the whole box as entirely off the detector (SKIP),
// entirely inside it (INTERIOR) or crossing an edge (EDGE).  Each view's detector
// footprint comes to shared memory by TMA, views ahead, through a pipe of slots
// that the warps pass at their own pace.  The inner loops are plain FP32: three
// FMAs for (u, v, w), one MUFU reciprocal, floor via a round-down add of
// 1.5*2^23, bilinear interpolation with FP32 lerps (hardware texture filtering is
// not used: its weights are 8-bit fixed point).
//
// The forward is in bp_forward.cu, the motion VJP in bp_vjp.cuh; here are the gradient
// images, the choice of the VJP's variant and the stand-alone data VJP.
//
// What bounds them (ncu, 256^3 x 128 views): no unit alone.  The L1 data pipe is at
// 72 % (forward) and 73 % (motion VJP: 12 taps per voxel-view at 1.4 wavefronts),
// issue at 66 and 61 % (21 and 51 instructions per voxel-view), the FMA pipe at 59 and
// 51 %, with the 32 and 24 warps per SM that their registers allow.
#include "bp_scatter.cuh"

namespace bpk {

cudaError_t bounds_status(unsigned* flags, long long* first, int op, cudaStream_t s) {
  cudaError_t e = file_bounds_status(flags, first, op, s);
  for (auto of : {bounds_status_forward, bounds_status_vjp_motion, bounds_status_vjp_fused,
                  bounds_status_vjp_exact}) {
    unsigned f = 0;
    long long first_of = op == 3 ? *first : -1;
    if (e == cudaSuccess) e = of(&f, &first_of, op == 2 ? 0 : op, s);
    if (e != cudaSuccess) return e;
    if (op == 3) continue;
    *flags |= f;
    if (*first < 0) *first = first_of;
  }
  return e;
}

// ------------------------------------------------------- gradient images

// g_u, g_v of one view in value per pixel: (d[+1] - d[-1]) / 2 inside,
// one-sided first differences on the two edge pixels (Sec. II-B.2), in
// stored units (the per-view dequantisation scale is applied with the view
// weight); output contiguous [V][nv][nu] float2.
template <typename T>
__global__ void __launch_bounds__(256) grad_images_kernel(const T* __restrict__ proj, ProjInfo pi,
                                                         float2* __restrict__ grad) {
  // one CTA per detector row (view j, row b); consecutive threads take
  // consecutive columns (measured on c2: 0.29 ms against 0.37 ms for a flat
  // grid-stride loop with 64-bit index divisions, 0.30 ms for CTAs looping
  // over rows)
  const long long rowi = blockIdx.x;
  const int j = (int)(rowi / pi.nv), b = (int)(rowi - (long long)j * pi.nv);
  const T* row = proj + (long long)j * pi.vs + (long long)b * pi.rs;
  float2* out = grad + rowi * pi.nu;
  for (int a = threadIdx.x; a < pi.nu; a += blockDim.x) {
    float gu = 0.0f, gv = 0.0f;
    if (pi.nu >= 2) {
      if (a == 0) gu = ldv(row + 1) - ldv(row);
      else if (a == pi.nu - 1) gu = ldv(row + a) - ldv(row + a - 1);
      else gu = 0.5f * (ldv(row + a + 1) - ldv(row + a - 1));
    }
    if (pi.nv >= 2) {
      if (b == 0) gv = ldv(row + pi.rs + a) - ldv(row + a);
      else if (b == pi.nv - 1) gv = ldv(row + a) - ldv(row - pi.rs + a);
      else gv = 0.5f * (ldv(row + pi.rs + a) - ldv(row - pi.rs + a));
    }
    out[a] = make_float2(gu, gv);
  }
}

cudaError_t launch_grad_images(const void* proj, int dtype, const ProjInfo& pi, float2* grad,
                               cudaStream_t s) {
  const long long nb = (long long)pi.nviews * pi.nv;  // detector rows
  if (nb == 0 || pi.nu == 0) return cudaSuccess;
  if (nb > 0x7fffffffLL) return cudaErrorInvalidValue;
  if (dtype == 0)
    grad_images_kernel<float><<<(int)nb, 256, 0, s>>>((const float*)proj, pi, grad);
  else if (dtype == 1)
    grad_images_kernel<__half><<<(int)nb, 256, 0, s>>>((const __half*)proj, pi, grad);
  else
    grad_images_kernel<__nv_bfloat16>
        <<<(int)nb, 256, 0, s>>>((const __nv_bfloat16*)proj, pi, grad);
  return cudaGetLastError();
}

// ----------------------------------------------- block image (fused data VJP)

// dproj[v][r][c] += the four block entries covering pixel (r, c): element 0
// of (r, c), 1 of (r, c-1), 2 of (r-1, c), 3 of (r-1, c-1).  One CTA per
// detector row.
__global__ void __launch_bounds__(256) block_combine_kernel(const float* __restrict__ blk,
                                                           float* __restrict__ dproj, int nv,
                                                           int nu) {
  const long long row = blockIdx.x;  // v * nv + r
  const bool up = row % nv != 0;
  const float* q0 = blk + row * nu * 4;
  const float* q1 = q0 - (long long)nu * 4;
  float* out = dproj + row * nu;
  for (int c = threadIdx.x; c < nu; c += blockDim.x) {
    float acc = __ldg(q0 + 4 * c);
    if (c > 0) acc += __ldg(q0 + 4 * (c - 1) + 1);
    if (up) {
      acc += __ldg(q1 + 4 * c + 2);
      if (c > 0) acc += __ldg(q1 + 4 * (c - 1) + 3);
    }
    out[c] += acc;
  }
}

long long block_image_floats(const ProjInfo& pi) {
  if (!BP_VJP_BLOCKS) return 0;
  return (long long)pi.nviews * pi.nv * pi.nu * 4;
}

cudaError_t launch_block_combine(const float* blk, const ProjInfo& pi, float* dproj,
                                cudaStream_t s) {
  const long long rows = (long long)pi.nviews * pi.nv;
  if (rows <= 0 || pi.nu <= 0) return cudaSuccess;
  if (rows > 0x7fffffffLL) return cudaErrorInvalidValue;
  block_combine_kernel<<<(unsigned)rows, 256, 0, s>>>(blk, dproj, pi.nv, pi.nu);
  return cudaGetLastError();
}
// ------------------------------------------------------- VJP w.r.t. Phat

// Defined in bp_vjp.cuh, instantiated by the bp_vjp_*.cu files.
template <typename T, bool FDK, bool EXACT, bool PROJ>
cudaError_t vjp_variants(const float* dvol, const void* proj, const ProjInfo& pi,
                         const float2* grad, const ViewGeom* geom, const VolInfo& vi,
                         float* partials, float* dproj, float* blk, int vc, unsigned nblocks,
                         const int* wide, cudaStream_t s, const RawStack* raw);
template <typename T, bool FDK, bool EXACT>
cudaError_t prepare_vjp_t();

#ifndef BP_VJP_CHUNK_MIB
#define BP_VJP_CHUNK_MIB 128
#endif
// Views per chunk of the view-chunked VJP grids.  Large problems: the bytes that
// one chunk's views touch (projections, gradient images, dL/dproj rows) are kept
// near BP_VJP_CHUNK_MIB, at most 32 views (c2, fused VJP before the block image:
// 16 MiB 23.1 ms, 32 MiB 20.3 ms, 64 MiB 18.1 ms, 128 MiB 17.4 ms).  Small ones:
// one wave of CTAs (a CTA's views are a serial chain) up to ten views each, then
// at least eight views (from 1.25 waves on) until there are three waves, so that the
// last one is not a large part (motion VJP with 32 / 16 / 8 / 4 views per chunk, in a
// step of 60 views: 96^3 voxels 467 / 438 / 430 / 440 us, 32^3 268 / 231 / 212 / 204 us).
// The stand-alone data VJP takes the same rule (now / before it, us: 32^3 x 60 39 / 113,
// 64^3 x 248 251 / 290, 96^3 x 120 341 / 364, 128^3 x 248 and larger the same).
constexpr int VJP_WAVE = 152 * VJP_MINB;
static int view_chunk(const ProjInfo& pi, long long bytes_per_px, int ntiles) {
  const long long per_view = (long long)pi.nu * pi.nv * bytes_per_px;
  long long c = ((long long)BP_VJP_CHUNK_MIB << 20) / (per_view > 0 ? per_view : 1);
  if (c > VB) c = VB;
  const long long n = (long long)ntiles * pi.nviews;
  const long long f = n <= 10LL * VJP_WAVE ? (n + VJP_WAVE - 1) / VJP_WAVE
                                           : (n / (3 * VJP_WAVE) > 8 ? n / (3 * VJP_WAVE) : 8);
  if (c > f) c = f;
  return c < 1 ? 1 : (int)c;
}


template <typename T, bool FDK, bool EXACT>
static cudaError_t vjp_dispatch(const float* dvol, const void* proj, const ProjInfo& pi,
                                const float2* grad, const ViewGeom* geom, const VolInfo& vi,
                                float* partials, float* dproj, float* blk, const int* wide,
                                cudaStream_t s, const RawStack* raw) {
  const int ntiles = vi.tiles_x * vi.tiles_y * vi.tiles_z;
  // block images only where the staged CENTRAL paths scatter
  const bool useb = dproj && blk && stageable<T>(proj, pi) && !EXACT && BP_VJP_BLOCKS;
  // the block image is left out of the chunk's byte count: measured on c2,
  // counting its 16 bytes per pixel (smaller chunks) made the fused VJP 2.8 %
  // slower (15.37 against 14.94 ms), counting 8 bytes 1.7 %
  const long long bpp = (long long)sizeof(T) + (EXACT ? 0 : 8) + (dproj ? 4 : 0);
  const int vc = view_chunk(pi, bpp, ntiles);
  const unsigned nblocks = (unsigned)((long long)ntiles * ((pi.nviews + vc - 1) / vc));
  if (!dproj)
    return vjp_variants<T, FDK, EXACT, false>(dvol, proj, pi, grad, geom, vi, partials, nullptr,
                                              nullptr, vc, nblocks, wide, s, raw);
  cudaError_t e = cudaSuccess;
  if (useb) e = cudaMemsetAsync(blk, 0, sizeof(float) * (size_t)block_image_floats(pi), s);
  if (e == cudaSuccess)
    e = vjp_variants<T, FDK, EXACT, true>(dvol, proj, pi, grad, geom, vi, partials, dproj,
                                          useb ? blk : nullptr, vc, nblocks, wide, s, raw);
  if (e == cudaSuccess && useb) e = launch_block_combine(blk, pi, dproj, s);
  return e;
}

bool vjp_uses_blocks(const void* proj, int dtype, const ProjInfo& pi, int exact) {
  if (exact || !BP_VJP_BLOCKS) return false;
  if (dtype == 0) return stageable<float>(proj, pi);
  if (dtype == 1) return stageable<__half>(proj, pi);
  return stageable<__nv_bfloat16>(proj, pi);
}

// Set the VJP kernels' shared-memory attributes on the current device
// (call before capturing a graph).
// Set the VJP kernels' shared-memory attributes on the current device
// (call before capturing a graph).
template <typename T>
static cudaError_t prepare_vjp_d(int fdk, int exact) {
  if (fdk) return exact ? prepare_vjp_t<T, true, true>() : prepare_vjp_t<T, true, false>();
  return exact ? prepare_vjp_t<T, false, true>() : prepare_vjp_t<T, false, false>();
}

cudaError_t prepare_vjp(int dtype, int fdk, int exact) {
  if (dtype == 0) return prepare_vjp_d<float>(fdk, exact);
  if (dtype == 1) return prepare_vjp_d<__half>(fdk, exact);
  return prepare_vjp_d<__nv_bfloat16>(fdk, exact);
}

template <typename T>
static cudaError_t vjp_dispatch_t(int fdk, int exact, const float* dvol, const void* proj,
                                  const ProjInfo& pi, const float2* grad, const ViewGeom* geom,
                                  const VolInfo& vi, float* partials, float* dproj,
                                  float* blk, const int* wide, cudaStream_t s, const RawStack* raw) {
  if (fdk)
    return exact ? vjp_dispatch<T, true, true>(dvol, proj, pi, grad, geom, vi, partials, dproj,
                                               blk, wide, s, raw)
                 : vjp_dispatch<T, true, false>(dvol, proj, pi, grad, geom, vi, partials, dproj,
                                                blk, wide, s, raw);
  return exact ? vjp_dispatch<T, false, true>(dvol, proj, pi, grad, geom, vi, partials, dproj,
                                              blk, wide, s, raw)
               : vjp_dispatch<T, false, false>(dvol, proj, pi, grad, geom, vi, partials, dproj,
                                               blk, wide, s, raw);
}

cudaError_t launch_vjp_motion(const float* dvol, const void* proj, int dtype, const ProjInfo& pi,
                              const float2* grad, const ViewGeom* geom, const VolInfo& vi,
                              int fdk, int exact, float* partials, float* dproj, float* blk,
                              const int* wide, cudaStream_t s, const RawStack* raw) {
  if (vi.zb != ZB_VJP) return cudaErrorInvalidValue;
  if (dtype == 0)
    return vjp_dispatch_t<float>(fdk, exact, dvol, proj, pi, grad, geom, vi, partials, dproj, blk,
                                 wide, s, raw);
  if (dtype == 1)
    return vjp_dispatch_t<__half>(fdk, exact, dvol, proj, pi, grad, geom, vi, partials, dproj,
                                  blk, wide, s, raw);
  return vjp_dispatch_t<__nv_bfloat16>(fdk, exact, dvol, proj, pi, grad, geom, vi, partials,
                                       dproj, blk, wide, s, raw);
}

// ------------------------------------------------- VJP w.r.t. the data

// Adjoint of Eq. 3 in d_j: every voxel-view adds s = delta * c * omega times
// its four bilinear weights to four detector pixels of a contiguous
// [V][nv][nu] FP32 image (zeroed by the caller), with global FP32 atomics
// reduced in L2: one vector reduction into the block image bout (when given)
// for a sample whose four taps lie on the detector, else up to four scalar
// ones.  (Measured on GB300: shared-memory
// FP32 atomics are emulated, and vector atomics with zero lanes cost as much
// as full ones, so neither privatisation nor padded vectors are used.)
template <int ZB, bool FDK, bool EDGE>
__device__ __forceinline__ void proj_view(float* out, float* bout, int nu, int nv,
                                          const TileView& t, float dx, float dy,
                                          const float (&delta)[ZB]) {
  const float u0 = fmaf(dy, t.ru1, fmaf(dx, t.ru0, t.U0));
  const float v0 = fmaf(dy, t.rv1, fmaf(dx, t.rv0, t.V0));
  const float w0 = fmaf(dy, t.rw1, fmaf(dx, t.rw0, t.W0));
#pragma unroll
  for (int k = 0; k < ZB; ++k) {
    if (delta[k] == 0.0f) continue;
    const float dz = k - 0.5f * (ZB - 1);
    Sample s = locate<EDGE>(fmaf(dz, t.ru2, u0), fmaf(dz, t.rv2, v0), fmaf(dz, t.rw2, w0),
                            t, nu, nv);
    if (EDGE && !s.ok) continue;
    const float sd = delta[k] * (FDK ? s.rwi * (s.rwi * t.wgtd) : t.wgtd);
    scatter_sample<EDGE>(out, bout, nu, nv, s, sd);
  }
}

template <int ZB, bool FDK>
__global__ void __launch_bounds__(NT, 2)
    vjp_proj_kernel(const float* __restrict__ dvol, ProjInfo pi, const ViewGeom* __restrict__ geom,
                    VolInfo vi, float* __restrict__ dproj, float* __restrict__ blk, int vchunk) {
  __shared__ TileView tvs[VB];
  const int ntiles = vi.tiles_x * vi.tiles_y * vi.tiles_z;
  const int tile = blockIdx.x % ntiles;
  const int vbeg = (blockIdx.x / ntiles) * vchunk, vend = min(pi.nviews, vbeg + vchunk);
  const TileIdx ti = tile_index<ZB>(vi, tile);
  const int i = ti.tx * TX + ti.lx, j = ti.ty * TY + ti.ly;
  float delta[ZB];
  bool nz = false;
#pragma unroll
  for (int k = 0; k < ZB; ++k) {
    const int z = ti.tz * ZB + k;
    delta[k] = (i < vi.nx && j < vi.ny && z < vi.nz)
                   ? __ldg(dvol + ((long long)z * vi.ny + j) * vi.nx + i)
                   : 0.0f;
    nz |= delta[k] != 0.0f;
  }
  if (!__syncthreads_or(nz)) return;
  for (int j0 = vbeg; j0 < vend; j0 += VB) {
    const int nb = min(VB, vend - j0);
    __syncthreads();
    setup_batch<float, false>(tvs, geom, j0, nb, ti, pi.nu, pi.nv);
    __syncthreads();
    for (int b = 0; b < nb; ++b) {
      const TileView t = tvs[b];
      if (t.mode == MODE_SKIP) continue;
      float* out = dproj + (long long)(j0 + b) * pi.nv * pi.nu;
      float* bout = blk ? blk + (long long)(j0 + b) * pi.nv * pi.nu * 4 : nullptr;
      if (t.mode == MODE_INTERIOR)
        proj_view<ZB, FDK, false>(out, bout, pi.nu, pi.nv, t, ti.dx, ti.dy, delta);
      else
        proj_view<ZB, FDK, true>(out, bout, pi.nu, pi.nv, t, ti.dx, ti.dy, delta);
    }
  }
}

cudaError_t launch_vjp_proj(const float* dvol, const ProjInfo& pi, const ViewGeom* geom,
                            const VolInfo& vi, int fdk, float* dproj, float* blk, cudaStream_t s) {
  if (vi.zb != ZB_VJP) return cudaErrorInvalidValue;
  if (!BP_VJP_BLOCKS) blk = nullptr;
  const int ntiles = vi.tiles_x * vi.tiles_y * vi.tiles_z;
  const int vc = view_chunk(pi, blk ? 20 : 4, ntiles);
  const unsigned nblocks = (unsigned)((long long)ntiles * ((pi.nviews + vc - 1) / vc));
  if (blk) {
    cudaError_t e = cudaMemsetAsync(blk, 0, sizeof(float) * (size_t)block_image_floats(pi), s);
    if (e != cudaSuccess) return e;
  }
  if (fdk)
    vjp_proj_kernel<ZB_VJP, true><<<nblocks, NT, 0, s>>>(dvol, pi, geom, vi, dproj, blk, vc);
  else
    vjp_proj_kernel<ZB_VJP, false><<<nblocks, NT, 0, s>>>(dvol, pi, geom, vi, dproj, blk, vc);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess && blk) e = launch_block_combine(blk, pi, dproj, s);
  return e;
}

}  // namespace bpk

