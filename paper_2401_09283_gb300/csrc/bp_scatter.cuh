// Scatter of one sample's bilinear weights into dL/dproj, for the fused and the
// stand-alone data VJP.
#pragma once

#include "bp_sample.cuh"

namespace bpk {

// ----------------------------------------------- block image (fused data VJP)

// The fused data VJP of interior tiles adds a sample's four bilinear weights
// with ONE 16-byte vector reduction instead of four scalar ones, into a block
// image: entry (r, c) holds the 2x2 pixel block with top-left pixel (r, c) as
// 4 consecutive floats, (r,c), (r,c+1), (r+1,c), (r+1,c+1), so a sample whose
// floor pixel is (iu, iv) adds to entry iv*nu + iu, a 16-byte aligned
// address with the same index arithmetic as the pixel itself.
// block_combine_kernel adds the blocks into dL/dproj afterwards (pixel (r, c)
// is element (dr, dc) of the entries (r-dr, c-dc)).
#ifndef BP_VJP_BLOCKS
#define BP_VJP_BLOCKS 1
#endif

__device__ __forceinline__ void red_v4(float* p, float a, float b, float c, float d) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c),
               "f"(d)
               : "memory");
}



// Entry px of a block image: one widening multiply-add.
__device__ __forceinline__ float* block_at(float* blk, unsigned px) {
  return reinterpret_cast<float*>(reinterpret_cast<char*>(blk) + (unsigned long long)px * 16u);
}

// Four bilinear-weighted scatter-adds of one sample into a [nv][nu] image
// (global FP32 atomics; taps off the detector are dropped in EDGE mode).
// With a block image bout (see below), a sample whose four taps lie on the
// detector adds them with one vector reduction there instead.
template <bool EDGE>
__device__ __forceinline__ void scatter_sample(float* out, float* bout, int nu, int nv,
                                               const Sample& s, float sd) {
  const float b1 = sd * s.tv, b0 = sd - b1;
  const float w11 = b1 * s.tu, w01 = b1 - w11, w10 = b0 * s.tu, w00 = b0 - w10;
  if (!EDGE) {
    int iu = s.iu, iv = s.iv;
    bc_interior(BC_SCATTER, iu, iv, nu, nv);
    if (BP_VJP_BLOCKS && bout) {
      red_v4(bout + 4 * ((long long)iv * nu + iu), w00, w10, w01, w11);
      return;
    }
    float* p = out + (long long)iv * nu + iu;
    atomicAdd(p, w00);
    atomicAdd(p + 1, w10);
    atomicAdd(p + nu, w01);
    atomicAdd(p + nu + 1, w11);
  } else {
    float* p = out + (long long)s.iv * nu + s.iu;
    const bool uu0 = (unsigned)s.iu < (unsigned)nu, uu1 = (unsigned)(s.iu + 1) < (unsigned)nu;
    const bool vv0 = (unsigned)s.iv < (unsigned)nv, vv1 = (unsigned)(s.iv + 1) < (unsigned)nv;
    if (BP_VJP_BLOCKS && bout && uu0 && uu1 && vv0 && vv1) {
      red_v4(bout + 4 * ((long long)s.iv * nu + s.iu), w00, w10, w01, w11);
      return;
    }
    if (uu0 && vv0) atomicAdd(p, w00);
    if (uu1 && vv0) atomicAdd(p + 1, w10);
    if (uu0 && vv1) atomicAdd(p + nu, w01);
    if (uu1 && vv1) atomicAdd(p + nu + 1, w11);
  }
}

}  // namespace bpk
