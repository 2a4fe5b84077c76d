// lane_kernel.cu -- launching the lane-group kernel (lane_kernel.cuh), and its
// instance with the gap penalties read at run time.
#include "lane_kernel.cuh"

namespace swgb {

typedef void (*LaneKernel)(DbView, const SearchParams*, SearchState*, Scratch);

// One translation unit per gap class (lane_class*.cu).
LaneKernel lane_kernel_class0();
LaneKernel lane_kernel_class1();
LaneKernel lane_kernel_class2();
LaneKernel lane_kernel_class0() { return lane_kernel<0>; }

static LaneKernel pick_lane(int gclass) {
  return gclass == 1 ? lane_kernel_class1() : gclass == 2 ? lane_kernel_class2() : lane_kernel_class0();
}

int lane_blocks_per_sm(bool wide) {
  const int smem = wide ? LANE_SMEM_WIDE : LANE_SMEM;
  for (int g = 0; g < GAP_CLASSES; g++) {  // every variant the plan may launch
    if (cudaFuncSetAttribute(pick_lane(g), cudaFuncAttributeMaxDynamicSharedMemorySize,
                             LANE_SMEM_WIDE) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
  }
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, pick_lane(0), LANE_WARPS * 32,
                                                    (size_t)smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return nb;
}

cudaError_t launch_lanes(int gclass, bool wide, int blocks, const DbView& db,
                         const SearchParams* params, SearchState* state, const Scratch& scr,
                         cudaStream_t stream) {
  cudaGetLastError();  // a stale error must not be read as this launch's
  pick_lane(gclass)<<<blocks, LANE_WARPS * 32, wide ? LANE_SMEM_WIDE : LANE_SMEM, stream>>>(
      db, params, state, scr);
  return cudaGetLastError();
}

}  // namespace swgb
