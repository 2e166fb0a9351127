// Instances of the persistent lateral kernel for non-square frames, nx = 64, 128, 256
// (any window, paper order).
#include "lateral_kernel.cuh"

namespace ssoct {

cudaError_t launch_lateral_pairs_256(const Plan& p, const LateralParams& lp, const void* tmap, int num_sms,
                                     cudaStream_t s) {
#define X(a, b) if (p.nx == a && p.ny == b) return launch_fw<a, b, false, false>(p, lp, tmap, num_sms, s);
  X(64, 256) X(64, 384) X(64, 512) X(64, 640) X(64, 768) X(64, 1024)
  X(128, 256) X(128, 384) X(128, 512) X(128, 640) X(128, 768) X(128, 1024)
  X(256, 64) X(256, 128) X(256, 384) X(256, 512) X(256, 640) X(256, 768) X(256, 1024)
#undef X
  return cudaErrorInvalidValue;
}

}  // namespace ssoct
