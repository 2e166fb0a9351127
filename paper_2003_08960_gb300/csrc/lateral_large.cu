// Instances of the persistent lateral kernel for the square frames of 640, 768
// and 1024 pixels (a unit of its own, so that the units compile side by side).
#include "lateral_kernel.cuh"

namespace ssoct {

cudaError_t launch_lateral_large(const Plan& p, const LateralParams& lp, const void* tmap, int num_sms,
                                 cudaStream_t s) {
#define X(n) if (p.nx == n && p.ny == n) return launch_square<n, n>(p, lp, tmap, num_sms, s);
  X(640) X(768) X(1024)
#undef X
  return cudaErrorInvalidValue;
}

}  // namespace ssoct
