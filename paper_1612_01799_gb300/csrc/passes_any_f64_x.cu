// Runtime-length forms, x passes, FP64.
#include "passes_any_launch.cuh"

namespace gsp {
GSP_INSTANTIATE_ANY_X(double)
}  // namespace gsp
