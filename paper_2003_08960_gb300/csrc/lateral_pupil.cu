// Instances of the persistent lateral kernel for the aberration path on square
// frames: the chirp is a table of one value per sensor pixel (any window).
#include "lateral_kernel.cuh"

namespace ssoct {

bool lateral_pupil_supported(int nx, int ny) { return nx == ny && nx >= 256 && lateral_supported(nx, ny); }

cudaError_t launch_lateral_pupil(const Plan& p, const LateralParams& lp, int num_sms, cudaStream_t s) {
#define X(n) if (p.nx == n && p.ny == n) return launch_fw<n, n, false, false, true>(p, lp, p.tmap, num_sms, s);
  X(256) X(384) X(512) X(640) X(768) X(1024)
#undef X
  return cudaErrorInvalidValue;
}

}  // namespace ssoct
