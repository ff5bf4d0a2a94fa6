// Instances of the event-chain kernel (ec_kernel.cuh): bead springs, screened domain form.
#include "ec_kernel.cuh"

namespace ecmc {

cudaError_t launch_ec_spring_screened(const ECParams &P, int lanes, cudaStream_t s) {
  if (lanes == 8) return launch_ec_t<8, true, false, true, true, false>(P, s);
  if (lanes == 16) return launch_ec_t<16, true, false, true, true, false>(P, s);
  if (lanes == 32) return launch_ec_t<32, true, false, true, true, false>(P, s);
  if (lanes == 4) return launch_ec_t<4, true, false, true, true, false>(P, s);
  return cudaErrorInvalidValue;
}

}  // namespace ecmc
