// Instances of the persistent lateral kernel for non-square frames, nx = 384, 512
// (any window, paper order).
#include "lateral_kernel.cuh"

namespace ssoct {

cudaError_t launch_lateral_pairs_512(const Plan& p, const LateralParams& lp, const void* tmap, int num_sms,
                                     cudaStream_t s) {
#define X(a, b) if (p.nx == a && p.ny == b) return launch_fw<a, b, false, false>(p, lp, tmap, num_sms, s);
  X(384, 64) X(384, 128) X(384, 256) X(384, 512) X(384, 640) X(384, 768) X(384, 1024)
  X(512, 64) X(512, 128) X(512, 256) X(512, 384) X(512, 640) X(512, 768) X(512, 1024)
#undef X
  return cudaErrorInvalidValue;
}

}  // namespace ssoct
