// Runtime-length forms, y passes, double-float.
#include "passes_any_launch.cuh"

namespace gsp {
GSP_INSTANTIATE_ANY_Y(DF)
}  // namespace gsp
