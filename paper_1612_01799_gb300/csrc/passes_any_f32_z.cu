// Runtime-length forms, z pass, FP32.
#include "passes_any_launch.cuh"

namespace gsp {
GSP_INSTANTIATE_ANY_Z(float)
}  // namespace gsp
