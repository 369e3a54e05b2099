// Runtime-length forms, y passes, FP32.
#include "passes_any_launch.cuh"

namespace gsp {
GSP_INSTANTIATE_ANY_Y(float)
}  // namespace gsp
