// Instances of the event-chain kernel (ec_kernel.cuh): plain FP64 domain form, hard tethers.
#include "ec_kernel.cuh"

namespace ecmc {

cudaError_t launch_ec_fp64(const ECParams &P, int lanes, cudaStream_t s) {
  if (lanes == 8) return launch_ec_t<8, false, false, true, false, false>(P, s);
  if (lanes == 16) return launch_ec_t<16, false, false, true, false, false>(P, s);
  if (lanes == 32) return launch_ec_t<32, false, false, true, false, false>(P, s);
  if (lanes == 4) return launch_ec_t<4, false, false, true, false, false>(P, s);
  return cudaErrorInvalidValue;
}

}  // namespace ecmc
