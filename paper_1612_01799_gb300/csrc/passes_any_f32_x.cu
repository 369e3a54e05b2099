// Runtime-length forms, x passes, FP32.
#include "passes_any_launch.cuh"

namespace gsp {
GSP_INSTANTIATE_ANY_X(float)
}  // namespace gsp
