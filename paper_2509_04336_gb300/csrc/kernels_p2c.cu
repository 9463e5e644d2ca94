// kernels_p2c.cu -- precision 2 (mixed, float-float phase): the walk that can look ahead over acceptances.
#include "kernels_impl.cuh"

namespace gwns {

GWNS_FF_WALK(launch_walk_ff_chain, 0, 1)

}  // namespace gwns
