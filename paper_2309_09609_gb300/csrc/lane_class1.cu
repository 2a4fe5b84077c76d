// lane_class1.cu -- the lane-group kernel compiled for gap class 1 (swgb_internal.h).
#include "lane_kernel.cuh"

namespace swgb {

typedef void (*LaneKernel)(DbView, const SearchParams*, SearchState*, Scratch);

LaneKernel lane_kernel_class1() { return lane_kernel<1>; }

}  // namespace swgb
