// Runtime-length forms, z pass, FP64.
#include "passes_any_launch.cuh"

namespace gsp {
GSP_INSTANTIATE_ANY_Z(double)
}  // namespace gsp
