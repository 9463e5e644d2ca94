// kernels_p2w.cu -- precision 2 (mixed, float-float phase): the walk without flow, relative binning or look-ahead over acceptances.
#include "kernels_impl.cuh"

namespace gwns {

GWNS_FF_WALK(launch_walk_ff_plain, 0, 0)

}  // namespace gwns
