// GEMM instances of the training step's weight gradients (both operands MN-major; the kernel is in
// fd_gemm_kernel.cuh).
#include "fd_gemm_kernel.cuh"

namespace fd {

cudaError_t launch_gemm_wgrad(const CUtensorMap& tmA, const CUtensorMap& tmB,
                              const CUtensorMap& tmO, const GemmParams& p, int bn, bool pair,
                              int num_sms, cudaStream_t s) {
  if (pair && bn == 256)
    return launch_bn<256, true, 0, false, true>(tmA, tmB, tmO, tmO, tmO, p, num_sms, s);
  if (pair) return cudaErrorInvalidValue;
  switch (bn) {
    case 64: return launch_bn<64, false, 0, false, true>(tmA, tmB, tmO, tmO, tmO, p, num_sms, s);
    case 128: return launch_bn<128, false, 0, false, true>(tmA, tmB, tmO, tmO, tmO, p, num_sms, s);
    case 192: return launch_bn<192, false, 0, false, true>(tmA, tmB, tmO, tmO, tmO, p, num_sms, s);
    case 256: return launch_bn<256, false, 0, false, true>(tmA, tmB, tmO, tmO, tmO, p, num_sms, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace fd
