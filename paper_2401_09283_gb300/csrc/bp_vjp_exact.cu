// The BILINEAR_EXACT motion VJP, alone and fused with the data VJP.
#include "bp_vjp.cuh"

namespace bpk {

BP_VJP_VARIANTS(true, false)
BP_VJP_VARIANTS(true, true)
BP_VJP_PREPARE(true)

cudaError_t bounds_status_vjp_exact(unsigned* flags, long long* first, int op, cudaStream_t s) {
  return file_bounds_status(flags, first, op, s);
}

}  // namespace bpk
