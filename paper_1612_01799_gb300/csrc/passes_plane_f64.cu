// The x and y passes of small planes, one kernel per direction, FP64.
#include "passes_any_launch.cuh"
#include "passes_plane.cuh"

namespace gsp {
template cudaError_t plane_xy<double>(const DevicePlan &, const PtrArray &, const PtrArray &, int, cudaStream_t, bool);
}  // namespace gsp
