// Instances of the persistent lateral kernel for non-square frames, nx = 640, 768, 1024
// (any window, paper order).
#include "lateral_kernel.cuh"

namespace ssoct {

cudaError_t launch_lateral_pairs_1024(const Plan& p, const LateralParams& lp, const void* tmap, int num_sms,
                                     cudaStream_t s) {
#define X(a, b) if (p.nx == a && p.ny == b) return launch_fw<a, b, false, false>(p, lp, tmap, num_sms, s);
  X(640, 64) X(640, 128) X(640, 256) X(640, 384) X(640, 512) X(640, 768) X(640, 1024)
  X(768, 64) X(768, 128) X(768, 256) X(768, 384) X(768, 512) X(768, 640) X(768, 1024)
  X(1024, 64) X(1024, 128) X(1024, 256) X(1024, 384) X(1024, 512) X(1024, 640) X(1024, 768)
#undef X
  return cudaErrorInvalidValue;
}

}  // namespace ssoct
