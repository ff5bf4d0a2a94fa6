// Launch of the event-chain kernel (ec_kernel.cuh): the serial instances and
// the choice of instance and lanes.
#include "ec_kernel.cuh"

namespace ecmc {

int tile_lanes(int64_t n_units, int lanes, int block_tiles) {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return lanes;
  return spread_lanes(n_units, lanes, block_tiles, sms);
}

cudaError_t launch_ec(const ECParams &P, int lanes, int fp32f, int pushoff, cudaStream_t s) {
  const bool spring = P.k_spring > 0.0;
  if (!P.domain) {
    // one unit: a whole warp, whatever the lanes asked for
    if (spring) return fp32f ? launch_ec_t<32, true, false, false, true, false>(P, s)
                             : launch_ec_t<32, false, false, false, true, false>(P, s);
    return fp32f ? launch_ec_t<32, true, false, false, false, false>(P, s)
                 : launch_ec_t<32, false, false, false, false, false>(P, s);
  }
  cudaError_t e = cudaErrorInvalidValue;
  // (a tile whose staging does not fit a block 32 / lanes times runs with
  // more lanes)
  for (int g = tile_lanes(P.n_units, lanes, P.block_tiles); g <= 32 && e == cudaErrorInvalidValue; g *= 2) {
    if (P.reps) e = fp32f ? launch_ec_batch_screened(P, g, s) : launch_ec_batch_fp64(P, g, s);
    else if (pushoff) e = spring ? launch_ec_pushoff_spring(P, g, s) : launch_ec_pushoff_tether(P, g, s);
    else if (spring) e = fp32f ? launch_ec_spring_screened(P, g, s) : launch_ec_spring_fp64(P, g, s);
    else e = fp32f ? launch_ec_screened(P, g, s) : launch_ec_fp64(P, g, s);
  }
  return e;
}

}  // namespace ecmc
