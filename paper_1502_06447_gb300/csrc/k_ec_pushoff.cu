// Instances of the event-chain kernel (ec_kernel.cuh): slow push-off, hard tethers.
#include "ec_kernel.cuh"

namespace ecmc {

cudaError_t launch_ec_pushoff_tether(const ECParams &P, int lanes, cudaStream_t s) {
  if (lanes == 8) return launch_ec_t<8, false, false, true, false, true>(P, s);
  if (lanes == 16) return launch_ec_t<16, false, false, true, false, true>(P, s);
  if (lanes == 32) return launch_ec_t<32, false, false, true, false, true>(P, s);
  if (lanes == 4) return launch_ec_t<4, false, false, true, false, true>(P, s);
  return cudaErrorInvalidValue;
}

}  // namespace ecmc
