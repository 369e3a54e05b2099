// The x and y passes of small planes, one kernel per direction, FP32.
#include "passes_any_launch.cuh"
#include "passes_plane.cuh"

namespace gsp {
template cudaError_t plane_xy<float>(const DevicePlan &, const PtrArray &, const PtrArray &, int, cudaStream_t, bool);
}  // namespace gsp
