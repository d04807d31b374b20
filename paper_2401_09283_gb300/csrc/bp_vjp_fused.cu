// The CENTRAL motion VJP fused with the data VJP.
#include "bp_vjp.cuh"

namespace bpk {

BP_VJP_VARIANTS(false, true)

cudaError_t bounds_status_vjp_fused(unsigned* flags, long long* first, int op, cudaStream_t s) {
  return file_bounds_status(flags, first, op, s);
}

}  // namespace bpk
