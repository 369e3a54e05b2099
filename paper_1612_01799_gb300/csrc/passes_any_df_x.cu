// Runtime-length forms, x passes, double-float.
#include "passes_any_launch.cuh"

namespace gsp {
GSP_INSTANTIATE_ANY_X(DF)
}  // namespace gsp
