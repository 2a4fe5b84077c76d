// lane_class2.cu -- the lane-group kernel compiled for gap class 2 (swgb_internal.h).
#include "lane_kernel.cuh"

namespace swgb {

typedef void (*LaneKernel)(DbView, const SearchParams*, SearchState*, Scratch);

LaneKernel lane_kernel_class2() { return lane_kernel<2>; }

}  // namespace swgb
