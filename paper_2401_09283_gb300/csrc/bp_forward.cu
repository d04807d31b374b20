// The forward backprojection (Eq. 3) for sm_103a: one kernel per call, and one over
// the tiles of every member of a batch.  Decomposition, records and staging as
// described in bp_project.cu.
#include "bp_sample.cuh"

namespace bpk {

// ------------------------------------------------------------------ forward

// One view from global memory (footprint not staged).
template <int ZB, typename T, bool FDK, bool EDGE>
__device__ __forceinline__ void forward_view(const T* img, long long rs, int nu, int nv,
                                             const TileView& t, float dx, float dy, float zlo,
                                             float (&acc)[ZB]) {
  float u0 = fmaf(dy, t.ru1, fmaf(dx, t.ru0, t.U0));
  float v0 = fmaf(dy, t.rv1, fmaf(dx, t.rv0, t.V0));
  float w0 = fmaf(dy, t.rw1, fmaf(dx, t.rw0, t.W0));
#pragma unroll
  for (int k = 0; k < ZB; ++k) {
    const float dz = zlo + k;
    Sample s = locate<EDGE>(fmaf(dz, t.ru2, u0), fmaf(dz, t.rv2, v0), fmaf(dz, t.rw2, w0),
                            t, nu, nv);
    if (EDGE && !s.ok) continue;
    float d00, d10, d01, d11;
    taps<EDGE>(img, rs, nu, nv, s, d00, d10, d01, d11);
    float val = bilerp(s.tu, s.tv, d00, d10, d01, d11);
    float wv = FDK ? s.rwi * (s.rwi * t.wgt) : t.wgt;
    acc[k] = fmaf(val, wv, acc[k]);
  }
}

// One view from its staged, zero-padded footprint (no checks, no clamps, tap
// offsets are compile-time constants), with packed pairs of voxels (k, k+1):
// every step of the scalar loop above, in the same order, on f32x2 pairs.
// buf is the FP32 footprint's shared-memory address, G the buffers' geometry.
template <int ZS, typename G, bool FDK>
__device__ __forceinline__ void forward_view_staged2(unsigned buf, const TileView& t, float dx,
                                                     float dy, float zlo, f2 (&acc)[ZS / 2]) {
  constexpr int P = StageGeom<G>::P;
  const float u0 = fmaf(dy, t.ru1, fmaf(dx, t.ru0, t.U0));
  const float v0 = fmaf(dy, t.rv1, fmaf(dx, t.rv0, t.V0));
  const float w0 = fmaf(dy, t.rw1, fmaf(dx, t.rw0, t.W0));
  const f2 U0 = pk2(u0, u0), V0 = pk2(v0, v0), W0 = pk2(w0, w0);
  const f2 RU = pk2(t.ru2, t.ru2), RV = pk2(t.rv2, t.rv2), RW = pk2(t.rw2, t.rw2);
  const f2 M2 = pk2(MAGIC, MAGIC), TWO = pk2(2.0f, 2.0f), WG = pk2(t.wgt, t.wgt);
  const f2 IC = staged_anchor(buf, t);
  f2 dz = pk2(zlo, zlo + 1.0f);  // exact: halves of small integers
#pragma unroll
  for (int p = 0; p < ZS / 2; ++p) {
    if (p) dz = add2(dz, TWO);
    const f2 u = fma2(dz, RU, U0), v = fma2(dz, RV, V0), w = fma2(dz, RW, W0);
    float wl, wh;
    up2(w, wl, wh);
    const f2 r = pk2(rcp_approx(wl), rcp_approx(wh));
    const f2 x = mul2(u, r), y = mul2(v, r);
    const f2 fx = sub2(add2_rd(x, M2), M2), fy = sub2(add2_rd(y, M2), M2);
    const f2 tu = sub2(x, fx), tv = sub2(y, fy);
    unsigned ql, qh;
    staged_pair<G, 0>(buf, t, IC, fx, fy, ql, qh);
    const f2 d00 = lds2<0>(ql, qh), d10 = lds2<1>(ql, qh);
    const f2 d01 = lds2<P>(ql, qh), d11 = lds2<P + 1>(ql, qh);
    const f2 val = bilerp2(tu, tv, d00, d10, d01, d11);
    acc[p] = fma2(val, FDK ? mul2(r, mul2(r, WG)) : WG, acc[p]);
  }
}

// FP16/BF16 data (CONV) is converted once per (tile, view) from the raw slot
// into one FP32 buffer that all warps share, so that path has CTA barriers:
// wait for view v, barrier (every warp is done with the FP32 buffer), convert,
// barrier, refill the raw slot, compute.
// One tile of the forward (its slices [zs ZS, zs ZS + ZS)): every view, in
// order, accumulated per voxel.  All threads of the CTA call it; tvs, pipe and
// dyn_smem are the CTA's shared memory.  The records of batch k+1 are built at the
// start of batch k (two record slots), so the footprints of the next views are known.
// bad: a copy has never arrived (the bounded wait gave up; the same in all warps when a
// tile begins); the tile's voxels are then NaN.
template <int ZB, int ZS, int NS, typename T, bool FDK, int STAGE>
__device__ __forceinline__ void forward_tile(const T* __restrict__ proj, const CUtensorMap* map,
                                             const ProjInfo& pi, const ViewGeom* __restrict__ geom,
                                             const VolInfo& vi, float* __restrict__ vol, int tile,
                                             int zs, TileView (*tvs)[batch_records<STAGE>()],
                                             StagePipe<NS>& pipe, unsigned char* dyn_smem,
                                             PipePos<NS>& pos, bool& bad) {
  using G = Geo<T, STAGE>;
  constexpr bool CONV = STAGE && StageGeom<G>::CONV;
  constexpr int SLOT = StageGeom<G>::BYTES, NB = batch_records<STAGE>();
  unsigned char* slots = dyn_smem + StageGeom<G>::F_BYTES;
  static_assert(ZS % 2 == 0 && ZB % ZS == 0, "voxel pairs");
  const TileIdx ti = tile_index<ZB, ZS>(vi, tile, zs);
  const int warp = threadIdx.x >> 5;
  f2 acc[ZS / 2];
#pragma unroll
  for (int k = 0; k < ZS / 2; ++k) acc[k] = pk2(0.0f, 0.0f);
  const int V = pi.nviews;
  const int nbatch = (V + NB - 1) / NB;
  setup_batch_call<G, STAGE != STAGE_NONE>(tvs[0], geom, 0, min(NB, V), ti, pi.nu, pi.nv);
  if (nbatch > 1)
    setup_batch_call<G, STAGE != STAGE_NONE>(tvs[1], geom, NB, min(NB, V - NB), ti, pi.nu, pi.nv);
  __syncthreads();
  if (STAGE && !bad && warp < NS && warp < V) {
    const unsigned s = (pos.slot + warp) % NS;
    stage_issue<G>(slots + s * SLOT, map, tvs[0][warp], warp, &pipe.full[s]);
  }
  for (int v = 0; v < V; ++v) {
    const int k = v / NB, b = v - k * NB;
    if (b == 0 && k >= 1 && k + 1 < nbatch) {
      __syncthreads();  // every warp is done with batch k-1
      setup_batch_call<G, STAGE != STAGE_NONE>(tvs[(k + 1) & 1], geom, (k + 1) * NB, min(NB, V - (k + 1) * NB), ti,
                            pi.nu, pi.nv);
      __syncthreads();
    }
    // without the pipe, a barrier per view keeps the warps' footprints together
    // in the L1 cache
    if (!STAGE) __syncthreads();
    const TileView& t = tvs[k & 1][b];
    const unsigned slot = pos.slot;
    unsigned char* buf = slots + slot * SLOT;
    if (STAGE && !bad) {  // (the lanes poll on their own; with CONV the CTA votes below)
      const bool ok = mbar_wait(&pipe.full[slot], pos.parity);
      bad = CONV ? !ok : !__all_sync(0xffffffffu, ok);
    }
    pos.next();
    const int vn = v + NS;
    const TileView& tn = tvs[(vn / NB) & 1][vn % NB];
    if constexpr (CONV) {
      bad = __syncthreads_or(bad);  // every warp has seen this phase and is done with F
      if (t.staged) {
        convert_stage<T, G>(reinterpret_cast<float*>(dyn_smem), reinterpret_cast<const T*>(buf), t);
        __syncthreads();  // F holds view v; the raw slot is free
      }
      if (warp == (v & 7) && vn < V && !bad) stage_issue<G>(buf, map, tn, vn, &pipe.full[slot]);
    }
    if (t.mode != MODE_SKIP) {
      if (STAGE && t.staged) {
        forward_view_staged2<ZS, G, FDK>(smem_addr(CONV ? dyn_smem : buf), t, ti.dx, ti.dy, ti.zlo,
                                         acc);
      } else {
        const T* img = proj + (long long)v * pi.vs;
        float a[ZS];
#pragma unroll
        for (int k2 = 0; k2 < ZS / 2; ++k2) up2(acc[k2], a[2 * k2], a[2 * k2 + 1]);
        if (t.mode == MODE_INTERIOR)
          forward_view<ZS, T, FDK, false>(img, pi.rs, pi.nu, pi.nv, t, ti.dx, ti.dy, ti.zlo, a);
        else
          forward_view<ZS, T, FDK, true>(img, pi.rs, pi.nu, pi.nv, t, ti.dx, ti.dy, ti.zlo, a);
#pragma unroll
        for (int k2 = 0; k2 < ZS / 2; ++k2) acc[k2] = pk2(a[2 * k2], a[2 * k2 + 1]);
      }
    }
    if constexpr (STAGE && !CONV) {
      if (!bad && last_warp(&pipe.done[slot]) && vn < V)
        stage_issue<G>(buf, map, tn, vn, &pipe.full[slot]);
    }
  }
  const int i = ti.tx * TX + ti.lx, j = ti.ty * TY + ti.ly;
  if (i < vi.nx && j < vi.ny) {
#pragma unroll
    for (int k = 0; k < ZS / 2; ++k) {
      float lo, hi;
      up2(acc[k], lo, hi);
      if (STAGE && bad) lo = hi = __int_as_float(0x7fc00000);
      const int z = ti.tz * ZB + zs * ZS + 2 * k;
      if (z < vi.nz) vol[((long long)z * vi.ny + j) * vi.nx + i] = lo;
      if (z + 1 < vi.nz) vol[((long long)(z + 1) * vi.ny + j) * vi.nx + i] = hi;
    }
  }
}

// Whether all n views are wide (all threads of the CTA).
__device__ __forceinline__ bool all_wide(const int* __restrict__ wide, int n) {
  bool w = true;
  for (int j = threadIdx.x; j < n; j += blockDim.x) w = w && wide[j] != 0;
  return __syncthreads_and(w);
}

template <int ZB, int ZS, int NS, typename T, bool FDK, int STAGE>
__global__ void __launch_bounds__(NT, NS > FWD_NS ? 2 : FWD_MINB)
    forward_kernel(const T* __restrict__ proj, const __grid_constant__ CUtensorMap map, ProjInfo pi,
                   const ViewGeom* __restrict__ geom, VolInfo vi, float* __restrict__ vol,
                   const int* __restrict__ wide) {
  if (wide && all_wide(wide, pi.nviews) == (STAGE != STAGE_NONE)) return;  // the other's launch
  __shared__ TileView tvs[2][batch_records<STAGE>()];
  __shared__ StagePipe<NS> pipe;
  extern __shared__ __align__(128) unsigned char dyn_smem[];
  if (STAGE) pipe_init(pipe);
  PipePos<NS> pos;
  bool bad = false;
  forward_tile<ZB, ZS, NS, T, FDK, STAGE>(proj, &map, pi, geom, vi, vol, blockIdx.x / (ZB / ZS),
                                      blockIdx.x % (ZB / ZS), tvs, pipe, dyn_smem, pos, bad);
  if (STAGE && bad) pipe_drain(pipe);
}

// z-extent of the forward's tiles
constexpr int ZB_FWD = 16;

// Staging needs 16-byte aligned rows; their length does not matter (TMA fills
// with zeros beyond it).  A tensor map's strides are below 2^40 bytes.
bool stage_aligned(const void* proj, int dtype, const ProjInfo& pi) {
  const long long es = dtype == 0 ? 4 : 2;
  return ((reinterpret_cast<uintptr_t>(proj) & 15) == 0) && (pi.rs * es) % 16 == 0 &&
         (pi.vs * es) % 16 == 0 && pi.vs * es < (1LL << 40);
}
// One CTA per detector row, or, where each reads the view flags first (CHOOSE), CTAs that
// loop over rows.
template <typename U, bool CHOOSE>
__global__ void __launch_bounds__(256)
    align_rows_kernel(const U* __restrict__ src, ProjInfo pi, U* __restrict__ dst, long long rs,
                      const int* __restrict__ wide) {
  auto copy = [&](long long row) {
    const long long j = row / pi.nv, b = row - j * pi.nv;
    const U* p = src + j * pi.vs + b * pi.rs;
    U* q = dst + row * rs;
    for (int a = threadIdx.x; a < pi.nu; a += blockDim.x) q[a] = p[a];
  };
  if constexpr (CHOOSE) {
    if (all_wide(wide, pi.nviews)) return;
    const long long rows = (long long)pi.nviews * pi.nv;
    for (long long row = blockIdx.x; row < rows; row += gridDim.x) copy(row);
  } else {
    copy(blockIdx.x);
  }
}

cudaError_t launch_align_rows(const void* proj, int dtype, const ProjInfo& pi, void* dst,
                              long long rs, const int* wide, cudaStream_t s) {
  const long long rows = (long long)pi.nviews * pi.nv;
  if (rows <= 0 || pi.nu <= 0) return cudaSuccess;
  if (rows > 0x7fffffffLL) return cudaErrorInvalidValue;
  const unsigned ctas = (unsigned)(wide && rows > 152 * 16 ? 152 * 16 : rows);
  auto run = [&](auto* kernel, auto* src, auto* to) {
    kernel<<<ctas, 256, 0, s>>>(src, pi, to, rs, wide);
    return cudaGetLastError();
  };
  if (dtype == 0)
    return run(wide ? align_rows_kernel<unsigned, true> : align_rows_kernel<unsigned, false>,
               (const unsigned*)proj, (unsigned*)dst);
  return run(wide ? align_rows_kernel<unsigned short, true> : align_rows_kernel<unsigned short, false>,
             (const unsigned short*)proj, (unsigned short*)dst);
}

void stage_extent(int dtype, bool half, int* cols, int* rows) {
  if (half) {
    *cols = dtype == 0 ? StageGeom<Half<float>>::P : StageGeom<Half<__half>>::P;
    *rows = StageGeom<Half<float>>::ROWS;
  } else {
    *cols = dtype == 0 ? StageGeom<float>::P : StageGeom<__half>::P;
    *rows = StageGeom<float>::ROWS;
  }
}

// The tensor map that the staging copies read: dimensions (nu, nv, views), box
// P x BOX_ROWS x 1.  (cuTensorMapEncodeTiled is a driver call without a stream;
// it only fills in the descriptor.)
cudaError_t make_stage_map(const void* proj, int dtype, const ProjInfo& pi, CUtensorMap* map,
                           bool half) {
  using Fn = decltype(&cuTensorMapEncodeTiled);
  static const Fn encode = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult r;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault,
                                         &r) != cudaSuccess ||
        r != cudaDriverEntryPointSuccess)
      f = nullptr;
    return reinterpret_cast<Fn>(f);
  }();
  if (!encode) return cudaErrorNotSupported;
  const cuuint64_t es = dtype == 0 ? 4 : 2;
  const cuuint64_t dims[3] = {(cuuint64_t)pi.nu, (cuuint64_t)pi.nv, (cuuint64_t)pi.nviews};
  const cuuint64_t strides[2] = {(cuuint64_t)pi.rs * es, (cuuint64_t)pi.vs * es};
  int cols, rows;
  stage_extent(dtype, half, &cols, &rows);
  const cuuint32_t box[3] = {(cuuint32_t)cols, BOX_ROWS, 1};
  const cuuint32_t ones[3] = {1, 1, 1};
  const CUtensorMapDataType dt = dtype == 0   ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                 : dtype == 1 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16
                                              : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  const CUresult rc =
      encode(map, dt, 3, const_cast<void*>(proj), dims, strides, box, ones,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
             CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return rc == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}


template <int ZS, int NS, typename T, bool FDK>
static cudaError_t forward_launch(const void* proj, const ProjInfo& pi, const ViewGeom* geom,
                                  const VolInfo& vi, float* vol, const int* wide, cudaStream_t s,
                                  const RawStack* raw) {
  const int nblocks = vi.tiles_x * vi.tiles_y * vi.tiles_z * (ZB_FWD / ZS);
  CUtensorMap map{};
  if (wide == WIDE_HALF && stageable<T>(proj, pi) &&
      make_stage_map(proj, dtype_id<T>(), pi, &map, true) == cudaSuccess) {
    const int smem = stage_smem_bytes<Half<T>, FWD_NS>();
    cudaError_t e = smem_attr_once<forward_kernel<ZB_FWD, 8, FWD_NS, T, FDK, STAGE_HALF>>(smem);
    if (e != cudaSuccess) return e;
    forward_kernel<ZB_FWD, 8, FWD_NS, T, FDK, STAGE_HALF>
        <<<vi.tiles_x * vi.tiles_y * vi.tiles_z * (ZB_FWD / 8), NT, smem, s>>>(
            (const T*)proj, map, pi, geom, vi, vol, nullptr);
    return cudaGetLastError();
  }
  const bool stage = stageable<T>(proj, pi) && wide != WIDE_ALL && wide != WIDE_HALF &&
                     make_stage_map(proj, dtype_id<T>(), pi, &map, false) == cudaSuccess;
  const int* sel = stage ? wide : nullptr;
  if (stage) {
    const int smem = stage_smem_bytes<T, NS>();
    cudaError_t e = smem_attr_once<forward_kernel<ZB_FWD, ZS, NS, T, FDK, STAGE_TILE>>(smem);
    if (e != cudaSuccess) return e;
    forward_kernel<ZB_FWD, ZS, NS, T, FDK, STAGE_TILE>
        <<<nblocks, NT, smem, s>>>((const T*)proj, map, pi, geom, vi, vol, sel);
    e = cudaGetLastError();
    if (e != cudaSuccess || !sel) return e;
  }
  // From global memory half tiles throughout: a warp's taps of one view are then closer
  // together in the L1 cache (128^3 x 200 at 4.8 px per voxel 1.061 -> 0.957 ms, 256^3 x
  // 120 at 1.5 px, three iterations with the VJP, 29.3 -> 28.7).
  forward_kernel<ZB_FWD, 8, FWD_NS, T, FDK, STAGE_NONE>
      <<<vi.tiles_x * vi.tiles_y * vi.tiles_z * (ZB_FWD / 8), NT, 0, s>>>(
          (const T*)(raw ? raw->proj : proj), map, raw ? raw->pi : pi, geom, vi, vol, sel);
  return cudaGetLastError();
}

// Slices of a tile per CTA and staging slots, by the number of 16^3 tiles: with
// too few tiles to fill the SMs, half tiles, and with few enough for one CTA per
// SM, four slots (a view's arithmetic there is shorter than a copy's latency).
// Measured, ms, 16 slices and 2 slots / 8 and 2 / 8 and 4: 64 tiles x 60 views
// 0.095 / 0.071 / 0.067, 216 x 248 0.452 / 0.383 / 0.510, 512 x 248 0.748 /
// 0.794 / 1.044; quarter tiles were slower throughout.
constexpr int FWD_FEW_TILES = 76, FWD_SOME_TILES = 304;
constexpr int FWD_NS_FEW = 4;

template <typename T, bool FDK>
static cudaError_t forward_dispatch(const void* proj, const ProjInfo& pi, const ViewGeom* geom,
                                    const VolInfo& vi, float* vol, const int* wide, cudaStream_t s,
                                    const RawStack* raw) {
  const int n = vi.tiles_x * vi.tiles_y * vi.tiles_z;
  if (n <= FWD_FEW_TILES)
    return forward_launch<8, FWD_NS_FEW, T, FDK>(proj, pi, geom, vi, vol, wide, s, raw);
  if (n <= FWD_SOME_TILES)
    return forward_launch<8, FWD_NS, T, FDK>(proj, pi, geom, vi, vol, wide, s, raw);
  return forward_launch<16, FWD_NS, T, FDK>(proj, pi, geom, vi, vol, wide, s, raw);
}

template <typename T, bool FDK>
static cudaError_t prepare_forward_t() {
  constexpr int smem = stage_smem_bytes<T, FWD_NS>();
  cudaError_t e = smem_attr_once<forward_kernel<ZB_FWD, 16, FWD_NS, T, FDK, STAGE_TILE>>(smem);
  if (e == cudaSuccess) e = smem_attr_once<forward_kernel<ZB_FWD, 8, FWD_NS, T, FDK, STAGE_TILE>>(smem);
  if (e == cudaSuccess)
    e = smem_attr_once<forward_kernel<ZB_FWD, 8, FWD_NS_FEW, T, FDK, STAGE_TILE>>(
        stage_smem_bytes<T, FWD_NS_FEW>());
  if (e == cudaSuccess)
    e = smem_attr_once<forward_kernel<ZB_FWD, 8, FWD_NS, T, FDK, STAGE_HALF>>(
        stage_smem_bytes<Half<T>, FWD_NS>());
  return e;
}

cudaError_t prepare_forward(int dtype, int fdk) {
  if (dtype == 0) return fdk ? prepare_forward_t<float, true>() : prepare_forward_t<float, false>();
  if (dtype == 1)
    return fdk ? prepare_forward_t<__half, true>() : prepare_forward_t<__half, false>();
  return fdk ? prepare_forward_t<__nv_bfloat16, true>()
             : prepare_forward_t<__nv_bfloat16, false>();
}

cudaError_t launch_forward(const void* proj, int dtype, const ProjInfo& pi, const ViewGeom* geom,
                           const VolInfo& vi_in, int fdk, float* vol, const int* wide,
                           cudaStream_t s, const RawStack* raw) {
  VolInfo vi = vi_in;  // the forward tiles z by ZB_FWD
  vi.zb = ZB_FWD;
  vi.tiles_z = (vi.nz + ZB_FWD - 1) / ZB_FWD;
  if (dtype == 0)
    return fdk ? forward_dispatch<float, true>(proj, pi, geom, vi, vol, wide, s, raw)
               : forward_dispatch<float, false>(proj, pi, geom, vi, vol, wide, s, raw);
  if (dtype == 1)
    return fdk ? forward_dispatch<__half, true>(proj, pi, geom, vi, vol, wide, s, raw)
               : forward_dispatch<__half, false>(proj, pi, geom, vi, vol, wide, s, raw);
  return fdk ? forward_dispatch<__nv_bfloat16, true>(proj, pi, geom, vi, vol, wide, s, raw)
             : forward_dispatch<__nv_bfloat16, false>(proj, pi, geom, vi, vol, wide, s, raw);
}

cudaError_t bounds_status_forward(unsigned* flags, long long* first, int op, cudaStream_t s) {
  return file_bounds_status(flags, first, op, s);
}

// ------------------------------------------------------------------ batches
// The forward over the tiles of every member of a batch.  The member table is
// a __grid_constant__ parameter, so the tile code reads each job's sizes and
// pointers from read-only parameter space, as the per-job kernels read their
// arguments.  Each tile runs the per-job block code, so the results are bit
// for bit those of the per-job launches.  Members are staged (checked by the
// host) in the batch's dtype.
//
// The forward is persistent: SMs x (resident CTAs per SM) blocks take tiles
// from an atomic counter, so tiles run in order (CTAs resident at the same
// time work on neighbouring tiles) and CTAs that drew cheap tiles (off the
// detector) take more; no CTA waits on another.  (The batch's VJP stage
// launches each member's own VJP kernel: a grouped launch over all members'
// (tile, view chunk) items read the job fields through run-time-indexed
// parameter loads and ran 8.7 % slower than the per-job kernel.)

template <int ZB, typename T, bool FDK>
__global__ void __launch_bounds__(NT, FWD_MINB)
    batch_forward_kernel(const __grid_constant__ BatchTable t, unsigned* __restrict__ counter) {
  __shared__ TileView tvs[2][VB];
  __shared__ StagePipe<FWD_NS> pipe;
  __shared__ int item;
  extern __shared__ __align__(128) unsigned char dyn_smem[];
  pipe_init(pipe);
  PipePos<FWD_NS> pos;
  bool bad = false;
  const int n = t.njobs, total = t.off_fwd[n];
  for (;;) {
    bad = __syncthreads_or(bad);  // every thread is done with the previous tile
    if (threadIdx.x == 0) item = (int)atomicAdd(counter, 1u);
    __syncthreads();
    const int w = item;
    if (w >= total) break;
    const int j = batch_find(t.off_fwd, n, w);
    const BatchJob& J = t.job[j];
    forward_tile<ZB, ZB, FWD_NS, T, FDK, STAGE_TILE>((const T*)J.proj, &J.map, J.pi, J.geom, J.vif, J.vol,
                                       w - t.off_fwd[j], 0, tvs, pipe, dyn_smem, pos, bad);
  }
  if (bad) pipe_drain(pipe);
}

int forward_zb() { return ZB_FWD; }

template <typename T, bool FDK>
static cudaError_t batch_forward_t(const BatchTable& tab, unsigned* counter, int sms,
                                   cudaStream_t s) {
  const int smem = stage_smem_bytes<T, FWD_NS>();
  cudaError_t e = smem_attr_once<batch_forward_kernel<ZB_FWD, T, FDK>>(smem);
  if (e != cudaSuccess) return e;
  batch_forward_kernel<ZB_FWD, T, FDK><<<sms * FWD_MINB, NT, smem, s>>>(tab, counter);
  return cudaGetLastError();
}

cudaError_t launch_batch_forward(const BatchTable& tab, unsigned* counter, int dtype, int fdk,
                                 int sms, cudaStream_t s) {
  if (dtype == 0) return fdk ? batch_forward_t<float, true>(tab, counter, sms, s)
                             : batch_forward_t<float, false>(tab, counter, sms, s);
  if (dtype == 1) return fdk ? batch_forward_t<__half, true>(tab, counter, sms, s)
                             : batch_forward_t<__half, false>(tab, counter, sms, s);
  return fdk ? batch_forward_t<__nv_bfloat16, true>(tab, counter, sms, s)
             : batch_forward_t<__nv_bfloat16, false>(tab, counter, sms, s);
}

// Shared-memory attributes of the batch kernels on the current device (call
// before capturing a graph; the members' VJP kernels are prepared by
// prepare_vjp).
cudaError_t prepare_batch(int dtype, int fdk, int exact) {
  (void)exact;
  if (dtype == 0)
    return fdk ? smem_attr_once<batch_forward_kernel<ZB_FWD, float, true>>(stage_smem_bytes<float, FWD_NS>())
               : smem_attr_once<batch_forward_kernel<ZB_FWD, float, false>>(stage_smem_bytes<float, FWD_NS>());
  if (dtype == 1)
    return fdk ? smem_attr_once<batch_forward_kernel<ZB_FWD, __half, true>>(stage_smem_bytes<__half, FWD_NS>())
               : smem_attr_once<batch_forward_kernel<ZB_FWD, __half, false>>(stage_smem_bytes<__half, FWD_NS>());
  return fdk ? smem_attr_once<batch_forward_kernel<ZB_FWD, __nv_bfloat16, true>>(
                   stage_smem_bytes<__nv_bfloat16, FWD_NS>())
             : smem_attr_once<batch_forward_kernel<ZB_FWD, __nv_bfloat16, false>>(
                   stage_smem_bytes<__nv_bfloat16, FWD_NS>());
}

}  // namespace bpk
