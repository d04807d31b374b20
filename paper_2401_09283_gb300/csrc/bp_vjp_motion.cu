// The CENTRAL motion VJP.
#include "bp_vjp.cuh"

namespace bpk {

BP_VJP_VARIANTS(false, false)
BP_VJP_PREPARE(false)

cudaError_t bounds_status_vjp_motion(unsigned* flags, long long* first, int op, cudaStream_t s) {
  return file_bounds_status(flags, first, op, s);
}

}  // namespace bpk
