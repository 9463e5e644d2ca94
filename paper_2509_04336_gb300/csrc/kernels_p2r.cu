// kernels_p2r.cu -- precision 2 (mixed, float-float phase): the walks of the relative-binning likelihood.
#include "kernels_impl.cuh"

namespace gwns {

GWNS_FF_WALK(launch_walk_ff_relbin, 1, 0)

cudaError_t launch_walk_ff_relbin_chain(GWNS_WALK_ARGS) {
  if (waveform != 0) return cudaErrorInvalidValue;
  GWNS_DISPATCH_N(GWNS_FF_WALK_ONE_11, 2, 0)
  return cudaGetLastError();
}

}  // namespace gwns
