// Runtime-length forms, y passes, FP64.
#include "passes_any_launch.cuh"

namespace gsp {
GSP_INSTANTIATE_ANY_Y(double)
}  // namespace gsp
